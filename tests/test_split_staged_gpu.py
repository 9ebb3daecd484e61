"""The split kernel's next tiles staged in shared memory (two walkers per thread,
65 to 100 modes): several passes a block, ragged last tiles, and warps that hold
few modes or none, against one walker per thread, which loads directly."""
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


@pytest.mark.parametrize("modes", [65, 75, 76, 100])
@pytest.mark.parametrize("form", ["spin_boson", "lvc2"])
@pytest.mark.parametrize("walkers", [64 * 3, 64 * 4 + 1, 64 * 13 + 33])
def test_staged_passes_give_the_same_bits(q, modes, form, walkers):
    model = (wl.spin_boson(1.0, 1.0, *wl.ohmic_modes(modes, 0.25, 5.0)) if form == "spin_boson"
             else wl.random_lvc2(modes, 5, 0.1))
    init = wl.sb_init(model, beta=2.0)
    got = []
    q.set_option(q.OPT_GRID_CAP, 2)  # (two blocks: up to four passes each)
    try:
        for wpt in (1, 2):
            m = q.Model(model)
            m.set_launch_shape(wpt, 0, 0)
            run = q.Run(m, walkers, 6, q.PREC_FP32_BULK, 4)
            run.sample(init)
            run.propagate(7, 0.01, 5)
            run.propagate(9, 0.01, 5)
            got.append((run.sums(), run.state()))
    finally:
        q.set_option(q.OPT_GRID_CAP, 0)
    assert np.array_equal(got[0][0], got[1][0])
    for k in got[0][1]:
        assert np.array_equal(got[0][1][k], got[1][1][k]), k
