"""The modes-in-memory forms of the FP32-bulk N_s-state kernel (R and P in shared
memory, P alone, neither) at the mode counts where one gives way to the next:
a model with one more mode that couples to nothing runs the next form, and its
other modes, weights, phases, pairs and output sums keep every bit."""
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


def _lvc(ns, n):
    m = wl.random_lvc4(7, n)
    return dict(m, n_states=ns, E=m["E"][:ns, :ns].copy(), K=m["K"][:, :ns, :ns].copy())


def _with_idle_mode(m):
    ns = m["n_states"]
    return dict(m, n_modes=m["n_modes"] + 1, mass=np.append(m["mass"], 1.0),
                omega=np.append(m["omega"], 1.3), K=np.concatenate([m["K"], np.zeros((1, ns, ns))]))


@pytest.mark.parametrize("ns", [3, 4])
@pytest.mark.parametrize("n,walkers", [(3, 389), (32, 128), (32, 389), (64, 1), (64, 389)])
def test_forms_agree_at_their_limits(q, ns, n, walkers):
    model = _lvc(ns, n)
    wide = _with_idle_mode(model)
    steps, stride = 25, 5
    q.set_option(q.OPT_MODES_IN_MEMORY, 1)
    try:
        a = q.Run(q.Model(model), walkers, 3, q.PREC_FP32_BULK, steps // stride + 1)
        a.sample(wl.sb_init(model, beta=2.0))
        st = a.state()
        pad = np.full((walkers, 1), 0.25, dtype=np.float32)
        b = q.Run(q.Model(wide), walkers, 3, q.PREC_FP32_BULK, steps // stride + 1)
        b.load_state(dict(st, R=np.hstack([st["R"], pad]), P=np.hstack([st["P"], pad])), 0)
        for r in (a, b):
            r.propagate(12, 0.01, stride)
            r.propagate(steps - 12, 0.01, stride)
    finally:
        q.set_option(q.OPT_MODES_IN_MEMORY, 0)
    sa, sb = a.state(), b.state()
    assert not np.array_equal(sa["R"], st["R"])
    for key in sa:
        got = sb[key][:, :n] if key in ("R", "P") else sb[key]
        assert np.array_equal(sa[key], got), key
    assert np.array_equal(a.sums(), b.sums())
