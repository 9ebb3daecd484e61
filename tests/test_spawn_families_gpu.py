"""Sums over families of one walker to thousands: the whole-block form of the
family observation, its limit and the narrower forms beside it, against the same
sums in FP64 from the walkers of the state."""
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


def _contributions(model, st, dia):
    """[walker, 8] complex: the diabatic and the adiabatic block of each walker."""
    E, K, R = model["E"], model["K"], st["R"].astype(np.float64)
    a = 0.5 * (E[0, 0] - E[1, 1]) + R @ (0.5 * (K[:, 0, 0] - K[:, 1, 1]))
    b = E[0, 1] + R @ K[:, 0, 1]
    th = 0.5 * np.arctan2(b, a)
    c, s = np.cos(th), np.sin(th)
    U = np.array([[-s, c], [c, s]])  # U[i, alpha]
    m = (st["m"].astype(np.float64) + st["m_lo"]) * 2.0 ** st["m_exp"]
    z = m * np.exp(-1j * (st["phi"].astype(np.float64) + st["phi_lo"])) * 1j ** st["q"]
    al, be = st["alpha"], st["beta"]
    w = np.arange(al.size)
    own = np.zeros((al.size, 4), dtype=complex)
    own[w, 2 * al + be] = z
    ua, ub = U[:, al, w], U[:, be, w]  # (U is symmetric)
    other = np.stack([z * ua[i] * ub[j] for i in range(2) for j in range(2)], 1)
    return np.concatenate([own, other] if dia else [other, own], 1)


@pytest.mark.parametrize("rep", ["adiabatic", "diabatic"])
# (least: what the largest family has at least)
@pytest.mark.parametrize("n0,cap,steps,modes,least",
                         [(1, 511, 60, 3, 257), (1, 700, 60, 3, 513), (2, 3000, 70, 5, 513),
                          (3, 9000, 80, 1, 513), (300, 60_000, 50, 3, 513), (2, 3000, 70, 40, 513),
                          (300, 4000, 70, 100, 33), (2, 3000, 70, 100, 513)])
def test_families_of_any_size(q, rep, n0, cap, steps, modes, least):
    model = wl.random_lvc2(modes, 3, 0.3)
    model = dict(copy.deepcopy(model), repr=rep, hop_scale=30.0)
    r = q.SpawnRun(q.Model(model), n0, cap, 11, steps + 1, precision=q.PREC_FP32_BULK)
    r.sample(wl.sb_init(model, beta=2.0))
    r.propagate(steps, 0.02, 1)
    st = r.state()
    assert np.bincount(st["family"], minlength=n0).max() >= least
    x = _contributions(model, st, rep == "diabatic")
    row = r.sums()[-1]
    for k in range(8):
        for c, v in ((0, x[:, k].real), (1, x[:, k].imag)):
            X = np.bincount(st["family"], weights=v, minlength=n0)
            A = np.bincount(st["family"], weights=np.abs(x[:, k]), minlength=n0)
            # (FP32 contributions: phases by the fast sine, 2e-6 of each; a and b
            # from FP32 sums over the modes, 2e-6 of the weight)
            M = np.bincount(st["family"], weights=np.abs(x).max(axis=1), minlength=n0)
            assert abs(row[2 * k + c] - X.sum()) <= 2e-6 * A.sum() + 2e-6 * M.sum() + 1e-30
            assert (abs(row[16 + 2 * k + c] - (X * X).sum())
                    <= 8e-6 * ((A + M) * (A + M)).sum() + 1e-30)
