"""FP64 solves across the limits of a launch (256 steps of two states, 16 of more,
three output times): one call and calls of a few steps give the same bits."""
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


def _solve(q, model, walkers, stride, calls):
    r = q.Run(q.Model(model), walkers, 9, q.PREC_FP64, sum(calls) // stride + 1)
    r.sample(wl.sb_init(model, beta=2.0))
    for n in calls:
        r.propagate(n, 0.01, stride)
    return r


@pytest.mark.parametrize("rep", ["adiabatic", "diabatic"])
@pytest.mark.parametrize("ns,n,walkers,stride,steps,cut", [
    (2, 1, 33, 400, 800, 97), (2, 3, 300, 255, 513, 100), (2, 17, 65, 256, 512, 64),
    (2, 5, 40, 1, 20, 3), (2, 2, 257, 100, 700, 31), (3, 2, 33, 50, 100, 7), (4, 6, 65, 16, 48, 5),
    (8, 3, 33, 17, 34, 16), (4, 1, 31, 1, 35, 2)])
def test_one_call_equals_many(q, rep, ns, n, walkers, stride, steps, cut):
    if ns == 2:
        model = wl.random_lvc2(n, 4, 0.3)
    else:
        rng = np.random.default_rng(ns)
        a = rng.uniform(0, 0.1, (n, ns, ns))
        model = wl._model(np.diag(0.4 * np.arange(ns)), a + a.transpose(0, 2, 1), np.ones(n),
                          rng.uniform(0.5, 2.0, n))
    model = dict(model, repr=rep)
    cuts = [cut] * (steps // cut) + ([steps % cut] if steps % cut else [])
    a, b = _solve(q, model, walkers, stride, [steps]), _solve(q, model, walkers, stride, cuts)
    assert a.status() == b.status()
    sa, sb = a.state(), b.state()
    for key in sa:
        assert np.array_equal(sa[key], sb[key]), key
    assert np.array_equal(a.sums(), b.sums())
