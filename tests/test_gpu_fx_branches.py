"""Forms of the larger kernels that the other tests do not reach: history
arrays on 16-byte boundaries, batches of orbital counts that are no multiples of
4, one and two orbitals, the double-float slices of more than 32 orbitals, and
steps captured in a graph (one launch per kernel) against direct ones."""
import numpy as np
import pytest

import oracle
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


def _dev(x):
    import torch
    return torch.as_tensor(np.ascontiguousarray(x), device="cuda")


def _ctx(kbe, M, n, seed):
    t, order = W.grid(n + 1, 0.05, 0.4, seed)
    ctx = kbe.Context(M, n + 1)
    ctx.set_grid(t, order)
    ctx.set_model(W.goe_h(M, seed), np.linspace(0.5, 1.5, M), W.site_potential(M), None)
    return ctx, t, order


@pytest.mark.parametrize("M,n", [(8, 140), (12, 73), (16, 47)])
def test_history_on_16_byte_boundaries(kbe, M, n):
    """The 32-byte loads need 32-byte rows: arrays 16 bytes off give the same bits."""
    import torch
    ctx, t, order = _ctx(kbe, M, n, 3)
    L, R = (_dev(x) for x in W.random_triangles(M, n + 1, 3))
    Sl, Sg = (_dev(x) for x in W.random_rows(M, n, 4))
    out = [torch.zeros((2, n + 1, M, M), dtype=torch.complex128, device="cuda") for _ in range(3)]
    ctx.history_slice(n, L, R, Sl, Sg, out[0])

    def off(x):
        y = torch.zeros(x.numel() + 2, dtype=x.dtype, device="cuda")
        k = 1 if y.data_ptr() % 32 == 0 else 2
        v = y[k:k + x.numel()].view(x.shape)
        v.copy_(x)
        assert v.data_ptr() % 32 == 16
        return v

    ctx.history_slice(n, off(L), off(R), Sl, Sg, out[1])
    ctx.history_slice(n, off(L), R, Sl, Sg, out[2])
    ctx.sync_status()
    assert out[0].abs().max() > 0 and torch.equal(out[0], out[1]) and torch.equal(out[0], out[2])
    ctx.close()


@pytest.mark.parametrize("sizes", [[(5, 230)], [(5, 230), (8, 120), (7, 150)], [(13, 60)],
                                   [(16, 50), (13, 60), (33, 14), (5, 210), (8, 110)], [(2, 1100), (33, 13)]])
def test_batched_tables_of_mixed_orbital_counts(kbe, sizes):
    """All on the tensor cores, multiples of 4 and not in one list: the rows of
    kbe_step to rounding (1e-13 of the row, as the batch tests have it)."""
    import torch
    runs = []
    for batched in (False, True):
        rs = []
        for k, (M, n_t) in enumerate(sizes):
            ctx, t, order = _ctx(kbe, M, n_t - 1, 20 + k)
            h = W.goe_h(M, 20 + k)
            r = kbe.Run(ctx)
            W.free_triangles_torch(h, W.half_filled_rho(h), t, n_t, "cuda", out=(r.L, r.R))
            rs.append(r)
        rows = [s[1] - 1 for s in sizes]
        if batched:
            b = kbe.Batch(rs)
            b.step(rows, P=2)
            b.sync_status()
            b.close()
        else:
            for r, n in zip(rs, rows):
                r.step(n, P=2)
                r.ctx.sync_status()
        runs.append(rs)
    for a, b, (M, n_t) in zip(*runs, sizes):
        p = W.tri_index(n_t - 1, 0)
        for x, y in ((a.L, b.L), (a.R, b.R)):
            assert (x[p:] - y[p:]).abs().max() < 1e-13 * x[p:].abs().max()
        a.ctx.close()
        b.ctx.close()


@pytest.mark.parametrize("M,n", [(1, 4100), (2, 1100)])
def test_one_and_two_orbitals(kbe, M, n):
    """Sampled columns of the longest rows against the sums in numpy: 1e-12 of
    the slice, as in the tests of the other sizes."""
    import torch
    rng = np.random.default_rng(M)
    ntri = W.tri_size(n + 1)
    L, R = (rng.standard_normal((ntri, M, M)) + 1j * rng.standard_normal((ntri, M, M)) for _ in range(2))
    for r in range(n + 1):
        R[W.tri_index(r, r)] = -1j * np.eye(M)
    Sl, Sg = W.random_rows(M, n, 8)
    ctx, t, order = _ctx(kbe, M, n, 6)
    out = torch.zeros((2, n + 1, M, M), dtype=torch.complex128, device="cuda")
    ctx.history_slice(n, _dev(L), _dev(R), _dev(Sl), _dev(Sg), out)
    assert ctx.last_launch_count == 3
    ctx.sync_status()
    got = out.cpu().numpy()
    size = np.abs(got).max()
    wn = kbe.grid_weights(t, order, n)[:, None, None]
    m = np.arange(n + 1)
    for c in [0, 1, 5, 63, 64, 127, 128, 129, n // 2, n - 128, n - 14, n - 13, n - 1, n]:
        p = np.where(m >= c, W.tri_index(m, np.minimum(m, c)), W.tri_index(c, np.minimum(m, c)))
        l, q = L[p], R[p]
        lo = (m < c)[:, None, None]
        adj = lambda x: np.conj(np.swapaxes(x, 1, 2))
        Gl, Gr = np.where(lo, -adj(l), l), np.where(lo, -adj(q), q)
        wc = kbe.grid_weights(t, order, c)[:, None, None]
        Ga = adj(R[W.tri_index(c, 0):W.tri_index(c, 0) + c + 1])
        A = wn * (Sg - Sl)
        for s, (G, S) in enumerate(((Gl, Sl), (Gl + Gr, Sg))):
            ref = np.matmul(A, G).sum(0) + np.matmul(wc * S[:c + 1], Ga).sum(0)
            assert np.abs(got[s, c] - ref).max() < 1e-12 * size, (c, s)
    ctx.close()


@pytest.mark.parametrize("M,n", [(33, 1), (33, 8), (33, 13), (40, 10), (48, 5), (64, 1), (64, 4)])
def test_df64_of_more_than_32_orbitals(kbe, M, n):
    """The untiled kernel below its line to the tensor cores, at the double-float bound of its tests."""
    import torch
    ctx, t, order = _ctx(kbe, M, n, 5)
    L, R = W.random_triangles(M, n + 1, 5)
    Sl, Sg = W.random_rows(M, n, 6)
    out = torch.zeros((2, n + 1, M, M), dtype=torch.complex128, device="cuda")
    ctx.history_slice(n, _dev(L), _dev(R), _dev(Sl), _dev(Sg), out, precision="df64")
    ctx.sync_status()
    ref = oracle.history_slice(t, order, n, L, R, Sl, Sg, nthreads=oracle.threads_available())
    assert np.abs(out.cpu().numpy() - ref).max() < 1e-11 * np.abs(ref).max()
    ctx.close()


# rows that a direct step takes in the cooperative kernel (up to 4096 entries: the
# first ones), on the FP64 pipe and on the tensor cores
@pytest.mark.parametrize("M,n,P", [(1, 30, 2), (2, 5, 1), (2, 200, 2), (2, 1023, 2), (3, 60, 3), (4, 63, 2), (4, 255, 2),
                                   (5, 100, 2), (7, 50, 2), (8, 1, 2), (8, 40, 2), (8, 63, 2), (13, 20, 2), (16, 9, 1),
                                   (16, 15, 2), (24, 5, 2), (26, 3, 2), (32, 3, 1), (32, 3, 2), (45, 1, 2), (8, 64, 2), (8, 140, 2), (17, 20, 2), (24, 30, 1)])
@pytest.mark.parametrize("precision", ["fp64", "df64"])
def test_captured_step_is_the_direct_step(kbe, M, n, P, precision):
    """Bitwise: row n, its right-hand side, the self-energy row and the slice.  (FP64:
    the cooperative kernel against one launch per kernel.)"""
    import torch
    ctx, t, order = _ctx(kbe, M, n, 7)
    h = W.goe_h(M, 7)
    run = kbe.Run(ctx)
    W.free_triangles_torch(h, W.half_filled_rho(h), t, n + 1, "cuda", out=(run.L, run.R))
    g = torch.Generator(device="cuda").manual_seed(3)
    F = torch.randn(run.F.shape, dtype=run.F.dtype, device="cuda", generator=g)
    p = W.tri_index(n, 0)

    def start():
        run.L[p:] = 0
        run.R[p:] = 0
        run.F.copy_(F)
        for x in (run.Sl, run.Sg, run.I):
            x.zero_()

    def result():
        ctx.sync_status()
        return [x.clone() for x in (run.L[p:], run.R[p:], run.F, run.Sl, run.Sg, run.I)]

    start()
    run.step(n, P=P, precision=precision)
    small = precision == "fp64" and (n + 1) * M * M <= 4096 and (M < 24 or M % 8 != 0)
    assert (ctx.last_launch_count == 1) == small
    direct = result()
    start()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        run.step(n, P=P, precision=precision)
    assert ctx.last_launch_count > 1
    for _ in range(2):  # a replay starts from the same state: row n is written anew
        start()
        graph.replay()
        captured = result()
        for a, b in zip(direct, captured):
            assert torch.equal(a, b)
    assert direct[0].abs().max() > 0
    ctx.close()
