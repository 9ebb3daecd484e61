"""FP32-bulk N_s-state solves whose gap and coupling of two states lie so far below
everything else that their squares leave the FP32 range: the walkers stay finite
and move as without that coupling."""
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


def _model(ns, n, coupling):
    E = np.diag([0.0, 0.0] + [1.0 + 0.5 * k for k in range(ns - 2)])
    K = np.zeros((n, ns, ns))
    for j in range(n):
        K[j, 0, 1] = K[j, 1, 0] = coupling * (1 + j)
        K[j, 2, 2] = 0.2 / n  # (state 2 stays above the pair)
    return wl._model(E, K, np.ones(n), np.linspace(0.8, 1.4, n))


@pytest.mark.parametrize("rep", ["adiabatic", "diabatic"])
@pytest.mark.parametrize("coupling", [1e-24, 1e-22, 1e-20, 1e-30, 1e-40])
@pytest.mark.parametrize("ns,n", [(3, 2), (4, 6), (4, 40), (5, 3), (8, 2)])
def test_walkers_stay_finite(q, ns, n, coupling, rep):
    got = []
    for c in (coupling, 0.0):
        model = dict(_model(ns, n, c), repr=rep)
        r = q.Run(q.Model(model), 300, 3, q.PREC_FP32_BULK, 5)
        r.sample(wl.sb_init(model, beta=2.0, state=2))
        r.propagate(40, 0.01, 10)
        st = r.state()
        assert r.status()["n_nonfinite"] == 0
        assert all(np.isfinite(st[k]).all() for k in ("R", "P", "m", "phi"))
        got.append((st, r.observables()))
    (a, oa), (b, ob) = got
    # (the coupling acts on no walker: K_01 is below 1e-18 of the other forces)
    assert np.array_equal(a["R"], b["R"]) and np.array_equal(a["P"], b["P"])
    assert np.isfinite(oa).all()
    assert np.allclose(oa[:, 0], ob[:, 0], atol=1e-6)
