"""The batch autotuner times what a step runs on the FP64 pipe, no more."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def kbe():
    import torch
    from paper_2405_08737_gb300 import build as B
    B.build()
    import paper_2405_08737_gb300 as K
    torch.cuda.set_device(0)
    return K


def _batch(kbe, sizes):
    runs = []
    for k, (M, n_t) in enumerate(sizes):
        t, order = W.grid(n_t, 0.05, 0.3, k)
        h = W.goe_h(M, k)
        ctx = kbe.Context(M, n_t)
        ctx.set_grid(t, order)
        ctx.set_model(h, np.linspace(0.2, 0.8, M), W.site_potential(M), None)
        run = kbe.Run(ctx)
        W.free_triangles_torch(h, W.half_filled_rho(h), t, n_t, "cuda", out=(run.L, run.R))
        runs.append(run)
    return runs, kbe.Batch(runs), [s[1] - 1 for s in sizes]


def _close(runs, batch):
    batch.close()
    for r in runs:
        r.ctx.close()


SMALL = [(4, 60)] * 6            # FP64 pipe: (n + 1)^2 M^3 = 2.3e5
LARGE = [(16, 300), (8, 400)]    # tensor cores, 100 times the work of SMALL


def test_large_systems_are_not_timed(kbe):
    """The time of the small systems is the same with large ones beside them
    (on the FP64 pipe those take some 20 times as long)."""
    ms = []
    for sizes in (SMALL, SMALL + LARGE):
        runs, batch, rows = _batch(kbe, sizes)
        block, work, t = batch.autotune(rows, reps=3)
        assert batch.policy() == (block, work)
        ms.append(t)
        _close(runs, batch)
    assert 0 < ms[1] < 2 * ms[0], ms


@pytest.mark.parametrize("rows", ["last", "none"])
def test_nothing_to_tune(kbe, rows):
    import torch
    runs, batch, last = _batch(kbe, LARGE)
    batch.set_policy(128, 18)
    for r in runs:
        r.I.fill_(7.0)
    block, work, ms = batch.autotune(last if rows == "last" else [-1] * len(last), reps=2)
    assert (block, work, ms) == (128, 18, 0.0) and batch.policy() == (128, 18)
    assert all((r.I == 7.0).all() for r in runs)
    batch.step(last)
    batch.sync_status()
    torch.cuda.synchronize()
    _close(runs, batch)
