"""The modes-in-memory FP32 kernels choose their form by the ensemble's size: more
tiles than one turn of the grid keep R and P (or P) in shared memory, fewer read
them from the ensemble.  The same walkers in a large and a small ensemble keep
every bit."""
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


@pytest.mark.parametrize("ns,n,rep", [(4, 23, "adiabatic"), (4, 24, "adiabatic"),
                                      (4, 32, "adiabatic"), (4, 33, "adiabatic"),
                                      (4, 64, "adiabatic"), (3, 47, "adiabatic"),
                                      (3, 48, "adiabatic"), (3, 63, "adiabatic"),
                                      (3, 9, "diabatic"), (3, 32, "diabatic")])
def test_walkers_keep_their_bits_in_a_large_ensemble(q, ns, n, rep):
    import torch

    rng = np.random.default_rng(n)
    a = rng.uniform(0, 0.1, (n, ns, ns)) / np.sqrt(n)
    model = wl._model(np.diag(0.4 * np.arange(ns)), a + a.transpose(0, 2, 1), np.ones(n),
                      rng.uniform(0.5, 2.0, n))
    model = dict(model, repr=rep)
    turn = 4 * torch.cuda.get_device_properties(0).multi_processor_count * 128
    states = []
    for walkers in (turn + 57, turn, 300):
        r = q.Run(q.Model(model), walkers, 3, q.PREC_FP32_BULK, 3)
        r.sample(wl.sb_init(model, beta=2.0))
        r.propagate(7, 0.02, 5)
        r.propagate(4, 0.02, 5)
        assert r.status()["n_nonfinite"] == 0
        states.append(r.state())
    for key in states[0]:
        for other in states[1:]:
            assert np.array_equal(states[0][key][:300], other[key][:300]), key
        assert np.array_equal(states[0][key][:turn], states[1][key]), key
