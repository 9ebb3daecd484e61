"""The chained FP32 spawning steps with every number of modes in registers, and
captured in a CUDA graph, against the three-launch route (modes in memory)."""
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


def _model(form, n, rep):
    m = (wl.random_lvc2(n, 3, 0.3) if form == "lvc2"
         else wl.spin_boson(0.5, 0.5, *wl.ohmic_modes(n, 0.3, 2.5)))
    return dict(m, repr=rep, hop_scale=8.0)


@pytest.mark.parametrize("rep", ["adiabatic", "diabatic"])
@pytest.mark.parametrize("form", ["lvc2", "spin_boson"])
@pytest.mark.parametrize("n", [2, 5, 8, 9, 16, 17, 31, 32])
def test_every_register_form(q, n, form, rep):
    model = _model(form, n, rep)
    got = []
    for mem in (0, 1):
        q.set_option(q.OPT_MODES_IN_MEMORY, mem)
        try:
            r = q.SpawnRun(q.Model(model), 300, 20_000, 5, 9, precision=q.PREC_FP32_BULK)
            r.sample(wl.sb_init(model, beta=2.0))
            for steps, stride in ((7, 4), (1, 4), (24, 4)):
                r.propagate(steps, 0.02, stride)
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


def test_captured_steps_replay(q):
    """Sampling and 40 chained steps with outputs, captured once: every replay gives
    the rows and walkers of the same calls outside a graph."""
    import torch

    model = _model("lvc2", 3, "adiabatic")
    init = wl.sb_init(model, beta=2.0)

    def calls(r):
        r.sample(init)
        r.propagate(13, 0.02, 5)
        r.propagate(27, 0.02, 5)

    def make():
        return q.SpawnRun(q.Model(model), 700, 50_000, 5, 9, precision=q.PREC_FP32_BULK)

    a = make()
    calls(a)
    rows, st = a.sums(), a.state()
    b = make()
    calls(b)  # (the library's first launches are behind)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        calls(b)
    for _ in range(3):
        b.obs_buf.fill_(0x7E)
        graph.replay()
        torch.cuda.synchronize()
        assert np.array_equal(b.sums(), rows)
        sb = b.state()
        for key in st:
            assert np.array_equal(sb[key], st[key]), key
