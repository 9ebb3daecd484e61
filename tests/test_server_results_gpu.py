"""Results of finished server requests: read together through the staging area,
in several lots when they exceed it, by themselves when one exceeds it."""
import numpy as np
import pytest

from paper_2608_14544_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

STAGE = 1 << 20
ROW2 = (8 * 2 * 2 + 3) * 8  # bytes of one output row with two states
HEAD = 256                  # the header's place before each result


@pytest.fixture(scope="module")
def q():
    import torch

    from paper_2608_14544_gb300 import build, qcl

    build.build()
    torch.cuda.set_device(0)
    return qcl


FULL = (STAGE - HEAD) // ROW2  # rows of the largest two-state result that is staged


@pytest.mark.parametrize("rows", [
    [2, 3, 2],                        # one lot
    [FULL // 2, FULL // 2, FULL // 2, 5],  # more than one lot
    [FULL, 4, FULL],                  # each lot full
    [FULL + 1, 3, FULL + 1],          # one by one, with a staged one between
])
def test_results_through_the_staging_area(q, rows):
    cfg = wl.config(1)
    reqs = [dict(model=cfg["model"], init=cfg["init"], n_traj=257 + 64 * k, seed=11 + k,
                 n_steps=r - 1, dt=cfg["dt"], out_stride=1) for k, r in enumerate(rows)]
    srv = q.Server(1 << 30, quantum_steps=1 << 20)
    ids = [srv.submit(r) for r in reqs]
    for r, n_rows, rid in zip(reqs, rows, ids):
        st, obs = srv.wait(rid)
        assert st == q.REQ_DONE
        run = q.Run(q.Model(r["model"]), r["n_traj"], r["seed"], q.PREC_FP32_BULK, n_rows)
        run.sample(r["init"])
        run.propagate(r["n_steps"], r["dt"], 1)
        want = run.observables()
        assert np.asarray(obs).size == n_rows * (ROW2 // 8)
        # the same kernels on the same inputs, reduced in the same order
        assert np.array_equal(np.asarray(obs).reshape(-1), np.asarray(want).reshape(-1))
    assert srv.stats()["n_error"] == 0
    srv.close()
