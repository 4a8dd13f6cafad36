"""Steps over the range of orbital counts: what the launches of a step do at
the sizes where their form changes."""
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


def _run(kbe, M, n, seed=1):
    n_t = n + 1
    t, order = W.grid(n_t, 0.05, 0.3, seed)
    h = W.goe_h(M, seed)
    ctx = kbe.Context(M, n_t)
    ctx.set_grid(t, order)
    ctx.set_model(h, np.linspace(0.2, 0.8, M), W.site_potential(M), None)
    run = kbe.Run(ctx)
    W.free_triangles_torch(h, W.half_filled_rho(h), t, n_t, "cuda", out=(run.L, run.R))
    return ctx, run


def _time_us(f, reps=20):
    import torch
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    best = 1e30
    for _ in range(5):
        f()
        torch.cuda.synchronize()
        e0.record()
        for _ in range(reps):
            f()
        e1.record()
        torch.cuda.synchronize()
        best = min(best, e0.elapsed_time(e1) / reps * 1e3)
    return best


@pytest.mark.parametrize("M", [1, 2, 3, 5, 8, 13, 15, 16, 17, 24, 31, 32, 33, 48, 64])
def test_sweep_finish_over_orbital_counts(kbe, M):
    """Right-hand side and corrector together (a block's threads cover a column)
    and apart: the right-hand side and the corrected row of the formula in
    numpy.  The corrector is linear in the new right-hand side row, so two calls
    whose slices differ by dI give rows that differ by w_c (-i) dI, with one
    weight w_c per column (taken from its first entry), and on the diagonal
    block by w_n times dF - dF^+."""
    import torch
    n = 6
    ctx, run = _run(kbe, M, n)
    rng = np.random.default_rng(M)
    p = W.tri_index(n, 0)
    keep = run.L.clone(), run.R.clone()
    dI = rng.standard_normal((2, n + 1, M, M)) + 1j * rng.standard_normal((2, n + 1, M, M))
    rows, F = [], []
    for k in range(2):
        run.L.copy_(keep[0])
        run.R.copy_(keep[1])
        I = torch.zeros((2, n + 1, M, M), dtype=torch.complex128, device="cuda")
        if k:
            I.copy_(torch.as_tensor(dI, device="cuda"))
        ctx.step_sweep_finish(n, run.L, run.R, I, run.F)
        assert ctx.last_launch_count == (2 if M <= 16 else 3)
        ctx.sync_status()
        F.append(run.F[n % kbe.KBE_RING_ROWS, :, :n + 1].cpu().numpy())
        rows.append([x[p:p + n + 1].cpu().numpy() for x in (run.L, run.R)])
    # F = -i (eps G + I): the new row's sources differ by -i dI
    dF = F[1] - F[0]
    scale = np.abs(dI).max() + np.abs(F[0]).max()
    assert np.abs(dF + 1j * dI).max() < 1e-14 * scale * M
    dL, dR = rows[1][0] - rows[0][0], rows[1][1] - rows[0][1]
    w = (dL[:n, 0, 0] / dF[0, :n, 0, 0]).real[:, None, None]
    assert (w > 0).all()
    size = max(np.abs(r).max() for r in rows[0] + rows[1])
    assert np.abs(dL[:n] - w * dF[0, :n]).max() < 1e-13 * size
    assert np.abs(dR[:n] - w * (dF[1] - dF[0])[:n]).max() < 1e-13 * size
    D = dF[0, n] - dF[0, n].conj().T
    wn = (dL[n, 0, 0] / D[0, 0]).real
    assert np.abs(dL[n] - wn * D).max() < 1e-13 * size and not dR[n].any()
    ctx.close()


def test_sweep_finish_of_large_blocks_is_spread_out(kbe):
    """n = 5, M = 64: 60 us over all entries, 700 us with a block per column; the
    bound lies between them."""
    ctx, run = _run(kbe, 64, 5)
    assert _time_us(lambda: ctx.step_sweep_finish(5, run.L, run.R, run.I, run.F)) < 200.0
    ctx.close()
