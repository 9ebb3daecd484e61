"""The chained FP32 spawning steps and the family observation at their edges:
walker counts around the 256-walker groups, steps whose children do not fit,
families from one walker to hundreds.  The three-launch route (modes in memory)
gives the same walkers, live counts and flags bit for bit; the own-pair sums and
their squares follow from the walkers of the state."""
import copy

import numpy as np
import pytest

from paper_2608_14544_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def q():
    import torch

    from paper_2608_14544_gb300 import build, qcl

    build.build()
    torch.cuda.set_device(0)
    return qcl


def _run(q, cfg, n0, cap, splits, mem):
    q.set_option(q.OPT_MODES_IN_MEMORY, mem)
    try:
        r = q.SpawnRun(q.Model(cfg["model"]), n0, cap, 11, sum(splits) // 5 + 1,
                       precision=q.PREC_FP32_BULK)
        r.sample(cfg["init"])
        for n in splits:
            r.propagate(n, cfg["dt"], 5)
    finally:
        q.set_option(q.OPT_MODES_IN_MEMORY, 0)
    return r


@pytest.mark.parametrize("cfg_id,rep", [(1, "adiabatic"), (3, "adiabatic"), (2, "diabatic")])
@pytest.mark.parametrize("n0,cap,kappa", [(1, 2000, 40.0), (255, 90_000, 20.0), (257, 700, 1.0),
                                          (256, 300, 20.0), (3, 4000, 60.0), (600, 601, 20.0)])
def test_chained_steps_and_families(q, cfg_id, rep, n0, cap, kappa):
    cfg = copy.deepcopy(wl.config(cfg_id))
    cfg["model"]["repr"] = rep
    cfg["model"]["hop_scale"] = kappa
    a = _run(q, cfg, n0, cap, (7, 18), 0)
    b = _run(q, cfg, n0, cap, (7, 18), 1)
    assert a.n_live() == b.n_live()
    assert a.status() == b.status()
    sa, sb = a.state(), b.state()
    for key in sa:
        assert np.array_equal(sa[key], sb[key]), key
    assert np.array_equal(a.sums(), b.sums())
    # the last output's own-pair block: sums over families of X and X^2
    m = (sa["m"].astype(np.float64) + sa["m_lo"]) * 2.0 ** sa["m_exp"]
    z = m * np.exp(-1j * (sa["phi"].astype(np.float64) + sa["phi_lo"])) * 1j ** sa["q"]
    row = a.sums()[-1]
    own = 0 if rep == "diabatic" else 8
    for k in range(4):
        hit = (2 * sa["alpha"] + sa["beta"]) == k
        for c, x in ((0, z.real), (1, z.imag)):
            X = np.bincount(sa["family"][hit], weights=x[hit], minlength=n0)
            A = np.bincount(sa["family"][hit], weights=np.abs(z[hit]), minlength=n0)
            # (each contribution rounds to FP32, phases by the fast sine: 2e-6 of |z|)
            assert abs(row[own + 2 * k + c] - X.sum()) <= 2e-6 * A.sum() + 1e-30
            assert abs(row[16 + own + 2 * k + c] - (X * X).sum()) <= 4e-6 * (A * A).sum() + 1e-30


@pytest.mark.parametrize("rep", ["adiabatic", "diabatic"])
@pytest.mark.parametrize("stride,splits", [(1, (4, 3)), (2, (4, 5)), (3, (2, 1, 7)), (50, (1, 6, 49))])
def test_steps_between_outputs(q, rep, stride, splits):
    """Intervals of one, two and more steps, cut by output times and by the
    call's end: the same walkers and rows as the three-launch route."""
    cfg = copy.deepcopy(wl.config(3))
    cfg["model"]["repr"] = rep
    cfg["model"]["hop_scale"] = 20.0
    got = []
    for mem in (0, 1):
        q.set_option(q.OPT_MODES_IN_MEMORY, mem)
        try:
            r = q.SpawnRun(q.Model(cfg["model"]), 300, 60_000, 5, sum(splits) // stride + 1,
                           precision=q.PREC_FP32_BULK)
            r.sample(cfg["init"])
            for n in splits:
                r.propagate(n, cfg["dt"], stride)
        finally:
            q.set_option(q.OPT_MODES_IN_MEMORY, 0)
        got.append(r)
    a, b = got
    assert a.n_live() == b.n_live() > 300
    assert a.status() == b.status()
    sa, sb = a.state(), b.state()
    for key in sa:
        assert np.array_equal(sa[key], sb[key]), key
    assert np.array_equal(a.sums(), b.sums())


@pytest.mark.parametrize("modes", [32, 33, 65])
def test_rows_do_not_depend_on_the_buffer(q, modes):
    """Rows of a many-mode model with a buffer of zeros and one of large numbers:
    only what the observation has written is added up."""
    model = wl.random_lvc2(modes, seed=3, scale=0.1)
    init = wl.sb_init(model, beta=2.0)
    rows = []
    for fill in (0, 0x7E):
        r = q.SpawnRun(q.Model(model), 700, 20_000, 2, 5, precision=q.PREC_FP32_BULK)
        r.obs_buf.fill_(fill)
        r.sample(init)
        r.propagate(8, 0.01, 2)
        rows.append(r.sums())
    assert np.isfinite(rows[0]).all()
    assert np.array_equal(rows[0], rows[1])
