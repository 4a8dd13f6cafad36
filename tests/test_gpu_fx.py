"""FP64 history slices on the tensor cores (csrc/history_fx.cu) and the sums of
their adjoint: sizes around its tiles against the oracle, at the FP64 path's
tolerance.

The error of a slice of n + 1 points is below 2^-56 of the largest products per
32 history entries plus FP64 rounding of the sums, well under 1e-12 of the
slice's maximum for the data below (the FP64 pipe's own bound in these tests)."""
import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu
TOL = 1e-12


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


def _setup(kbe, M, n, seed, kind, kmax=5):
    n_t = n + 1
    t, order = W.grid(n_t, 0.05, 0.4, seed, kmax=kmax)
    h = W.goe_h(M, seed)
    if kind == "free":
        L, R = W.free_triangles(h, W.half_filled_rho(h), t)
        Sl, Sg = oracle.sigma_row(oracle.local_U4(np.linspace(0.5, 1.5, M)), n, L, R) if M <= 16 else \
            W.random_rows(M, n, seed)
    else:
        L, R = W.random_triangles(M, n_t, seed)
        Sl, Sg = W.random_rows(M, n, seed + 1)
    if kind == "ramp":  # rows that grow and fall by 2^3 per step: exponents change inside a chunk
        for r in range(n_t):
            s = 2.0 ** (3 * (r % 9))
            L[W.tri_index(r, 0):W.tri_index(r + 1, 0)] *= s
            R[W.tri_index(r, 0):W.tri_index(r, r)] *= s
    ctx = kbe.Context(M, n_t)
    ctx.set_grid(t, order)
    ctx.set_model(h, np.ones(M), W.site_potential(M), None)
    return ctx, t, order, L, R, Sl, Sg


# (n + 1)^2 M^3 above the line where the slice goes to the tensor cores; column
# tiles of 128 / M columns full and ragged, units of 8 entries that span several
# history points or a fraction of one, orbital counts that are no multiple of 4
# or of 8, one to eight parts
@pytest.mark.parametrize("M,n", [(3, 560), (5, 269), (7, 160), (8, 127), (8, 128), (8, 143), (12, 73), (13, 70),
                                 (16, 47), (16, 50), (24, 26), (31, 20), (32, 19), (33, 16), (64, 7)])
@pytest.mark.parametrize("kind", ["free", "random", "ramp"])
def test_slice_sizes(kbe, M, n, kind):
    import torch
    ctx, t, order, L, R, Sl, Sg = _setup(kbe, M, n, 3 * M + n, kind)
    out = torch.zeros((2, n + 1, M, M), dtype=torch.complex128, device="cuda")
    ctx.history_slice(n, _dev(L), _dev(R), _dev(Sl), _dev(Sg), out)
    assert ctx.last_launch_count == 3
    ctx.sync_status()
    ref = oracle.history_slice(t, order, n, L, R, Sl, Sg, nthreads=oracle.threads_available())
    err = np.abs(out.cpu().numpy() - ref).max() / np.abs(ref).max()
    assert err < TOL, err
    ctx.close()


def test_high_orders_and_zero_history(kbe):
    import torch
    M, n = 8, 140
    ctx, t, order, L, R, Sl, Sg = _setup(kbe, M, n, 5, "random", kmax=12)
    out = torch.zeros((2, n + 1, M, M), dtype=torch.complex128, device="cuda")
    ctx.history_slice(n, _dev(L), _dev(R), _dev(Sl), _dev(Sg), out)
    ref = oracle.history_slice(t, order, n, L, R, Sl, Sg, nthreads=oracle.threads_available())
    # order-12 weights differ by about 1e-13 between the library's and the oracle's routes
    assert np.abs(out.cpu().numpy() - ref).max() < 1e-11 * np.abs(ref).max()
    ctx.history_slice(n, _dev(0 * L), _dev(0 * R), _dev(Sl), _dev(Sg), out)
    ctx.sync_status()
    assert not out.abs().any()
    ctx.close()


@pytest.mark.parametrize("M,n", [(3, 560), (5, 269), (8, 128), (12, 73), (16, 47), (33, 16)])
def test_rows_that_start_late(kbe, M, n):
    """Rows of zeros that start inside an accumulation, with values 2^-70 of the
    later ones or with those (the bound of test_slice_sizes)."""
    import torch
    ctx, t, order, L, R, Sl, Sg = _setup(kbe, M, n, 11 * M + n, "random")
    rng = np.random.default_rng(n)
    for x in (L, R):
        x *= rng.choice([0.0, 2.0 ** -70, 1.0], p=[0.45, 0.45, 0.1], size=x.shape)
        x[W.tri_index(n // 2, 0):] *= rng.choice([0.0, 1.0], size=(x.shape[0] - W.tri_index(n // 2, 0), 1, 1))
    out = torch.zeros((2, n + 1, M, M), dtype=torch.complex128, device="cuda")
    ctx.history_slice(n, _dev(L), _dev(R), _dev(Sl), _dev(Sg), out)
    assert ctx.last_launch_count == 3
    ctx.sync_status()
    ref = oracle.history_slice(t, order, n, L, R, Sl, Sg, nthreads=oracle.threads_available())
    assert np.abs(out.cpu().numpy() - ref).max() < TOL * np.abs(ref).max()
    ctx.close()


@pytest.mark.parametrize("M,n", [(5, 269), (8, 128), (13, 70), (16, 47), (24, 26), (33, 16)])
def test_adjoint_is_the_transpose(kbe, M, n):
    """Re<Ibar, I(dS)> = Re<Sbar, dS> for random rows Ibar, dS, which are
    independent of each other (1e-12 of the products' sizes; I is linear in the
    self-energy row and checked against the oracle above)."""
    import torch
    ctx, t, order, L, R, Sl, Sg = _setup(kbe, M, n, 7 * M + n, "random")
    rng = np.random.default_rng(M)
    Ib = _dev(rng.standard_normal((2, n + 1, M, M)) + 1j * rng.standard_normal((2, n + 1, M, M)))
    Ld, Rd, Sld, Sgd = _dev(L), _dev(R), _dev(Sl), _dev(Sg)
    out = torch.zeros_like(Ib)
    ctx.history_slice(n, Ld, Rd, Sld, Sgd, out)
    dSl, dSg = torch.zeros_like(Sld), torch.zeros_like(Sgd)
    dL = torch.zeros((n + 1, M, M), dtype=torch.complex128, device="cuda")
    ctx.adjoint_slice(n, Ld, Rd, Sld, Sgd, Ib, dSl, dSg, dL, torch.zeros_like(dL), n)
    ctx.sync_status()
    lhs = (Ib.conj() * out).sum().real
    rhs = (dSl.conj() * Sld).sum().real + (dSg.conj() * Sgd).sum().real
    size = (dSl.conj() * Sld).abs().sum() + (dSg.conj() * Sgd).abs().sum()
    assert abs(lhs - rhs) < TOL * size
    ctx.close()


@pytest.mark.parametrize("where", ["L", "R", "Sl"])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_non_finite_entries(kbe, where, bad):
    """The same outputs are non-finite as in the sum of two row bands (which
    run on the FP64 pipe), and the status word reports it."""
    import torch
    M, n = 8, 130
    ctx, t, order, L, R, Sl, Sg = _setup(kbe, M, n, 9, "random")
    x = {"L": L, "R": R, "Sl": Sl}[where]
    x[40 if where == "Sl" else W.tri_index(90, 37), 2, 5] = bad
    Ld, Rd, Sld, Sgd = _dev(L), _dev(R), _dev(Sl), _dev(Sg)
    out, part = (torch.zeros((2, n + 1, M, M), dtype=torch.complex128, device="cuda") for _ in range(2))
    ctx.history_slice(n, Ld, Rd, Sld, Sgd, out)
    with pytest.raises(kbe.KBEError) as e:
        ctx.sync_status()
    assert e.value.status == kbe.KBE_ENUMERIC
    total = torch.zeros_like(out)
    for lo, hi in ((0, 60), (60, n + 1)):
        ctx.history_slice_band(n, lo, hi, Ld, Rd, Sld, Sgd, part)
        total += part
    with pytest.raises(kbe.KBEError):
        ctx.sync_status()
    a, b = out.cpu().numpy(), total.cpu().numpy()
    assert np.array_equal(np.isfinite(a), np.isfinite(b)) and not np.isfinite(a).all()
    ok = np.isfinite(b)
    assert np.abs(a[ok] - b[ok]).max() < TOL * np.abs(b[ok]).max()
    ctx.close()


def test_batch_crosses_the_line(kbe):
    """Batched steps whose rows move from the FP64 pipe to the tensor cores
    (M = 8 from n = 98 on; M = 12 and M = 3 stay on either side): the rows of
    kbe_step within 1e-13, whatever set of kernels the graph holds."""
    import torch
    sizes = [(8, 102), (12, 90), (3, 60), (8, 140)]
    first = [95, 84, 54, 134]
    runs = []
    for batched in (False, True):
        rs = []
        for k, (M, n_t) in enumerate(sizes):
            t, order = W.grid(n_t, 0.05, 0.4, 40 + k)
            h = W.goe_h(M, k)
            L, R, F = W.restart_state(h, W.half_filled_rho(h), t, order, first[k], n_t)
            ctx = kbe.Context(M, n_t)
            ctx.set_grid(t, order)
            ctx.set_model(h, np.linspace(0.5, 1.5, M), W.site_potential(M), None)
            r = kbe.Run(ctx)
            r.L.copy_(torch.as_tensor(L, device="cuda"))
            r.R.copy_(torch.as_tensor(R, device="cuda"))
            for j, f in F.items():
                r.F[j % kbe.KBE_RING_ROWS, :, : j + 1] = torch.as_tensor(f, device="cuda")
            rs.append(r)
        b = kbe.Batch(rs) if batched else None
        for q in range(6):
            if batched:
                b.step([f + q for f in first], P=2)
            else:
                for f, r in zip(first, rs):
                    r.step(f + q, P=2)
        if batched:
            b.sync_status()
            b.close()
        runs.append(rs)
    for a, b in zip(*runs):
        for x, y in ((a.L, b.L), (a.R, b.R)):
            assert (x - y).abs().max() < 1e-13 * x.abs().max()
        a.ctx.close()
        b.ctx.close()
