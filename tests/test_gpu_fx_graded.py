"""FP64 slices on the tensor cores (csrc/history_fx.cu) with data whose sizes
vary over the history: the error of each output column, and of each row of
orbitals, against the sizes of its own products, not of the whole slice.

Bound.  An accumulation takes 64 history entries (128 real products) whose
operands share an exponent that lies at most 5 bits above the largest product of
the accumulation and the chunk before it (2 or 3 bits of room and the mantissas'
own).  Dropped digit products and truncated digits cost at most 2^-58 of that per
product, 2^-51 per accumulation, 2^-46 of the largest product in the worst case;
with signs that differ it is about a tenth of it times 2^-5 (sqrt(128) instead of
128 terms, a quarter of the worst size each).  The reference's and the sums' own
rounding stays below 2^-50 of the sum of the products' sizes.  2^-47 of that sum
separates both from a shared exponent that the products do not reach, which loses
2^-40 and more for the data below."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu
BOUND = 2.0 ** -47
LD, CLD = np.longdouble, np.clongdouble


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


def _planes(M, n, L, R, cols):
    """G^<, G^>, G^A of (m, c) for all m and the columns `cols`, in extended
    precision: [m][column][x][b]."""
    Gl, Gg, Ga = (np.zeros((n + 1, len(cols), M, M), CLD) for _ in range(3))
    for k, c in enumerate(cols):
        for m in range(n + 1):
            p = W.tri_index(max(m, c), min(m, c))
            l, q = L[p].astype(CLD), R[p].astype(CLD)
            if m < c:
                l, q = -np.conj(l.T), -np.conj(q.T)
            Gl[m, k], Gg[m, k] = l, l + q
            if m <= c:
                Ga[m, k] = np.conj(R[p].astype(CLD).T)
    return Gl, Gg, Ga


def _adjoint_planes(M, n, L, R, pts):
    """The adjoints of the same for all c and the points `pts`: [c][point][b][x]."""
    Gl, Gg, Ga = (np.zeros((n + 1, len(pts), M, M), CLD) for _ in range(3))
    for k, m in enumerate(pts):
        for c in range(n + 1):
            p = W.tri_index(max(m, c), min(m, c))
            l, q = L[p].astype(CLD), R[p].astype(CLD)
            if m >= c:
                l, q = np.conj(l.T), np.conj(q.T)
            else:
                l, q = -l, -q
            Gl[c, k], Gg[c, k] = l, l + q
            if m <= c:
                Ga[c, k] = R[p].astype(CLD)
    return Gl, Gg, Ga


def _sample(n):
    """Columns: the first and last ones, the middle, and a few between."""
    return sorted({0, 1, n // 7, n // 3, n // 2, (4 * n) // 5, n - 7, n - 2, n - 1, n} & set(range(n + 1)))


def _weights(kbe, t, order, n):
    w = np.zeros((n + 1, n + 1), LD)
    for c in range(n + 1):
        w[c, :c + 1] = kbe.grid_weights(t, order, c)
    return w


def _mm(A, G, out, size):
    """out[k] += sum_m A[m(, k)] G[m, k], size likewise with absolute values."""
    a = np.abs(A).astype(np.float64)
    g = np.abs(G).astype(np.float64)
    per_column = A.ndim == 4
    for m in range(G.shape[0]):
        Am, am = (A[m], a[m]) if per_column else (A[m][None], a[m][None])
        # extended-precision products orbital by orbital (no BLAS for that type)
        for x in range(G.shape[2]):
            out += Am[:, :, x, None] * G[m][:, None, x, :]
        size += np.matmul(am, g[m])


def _setup(kbe, M, n, seed, kind, grow):
    """Random operands; `grow`: the step (a power of two) by which the self-energy
    row grows three times over towards m = n and the history falls with |m - c|."""
    t, order = W.grid(n + 1, 0.05, 0.3, seed)
    L, R = W.random_triangles(M, n + 1, seed)
    Sl, Sg = W.random_rows(M, n, seed + 1)
    m = np.arange(n + 1)
    if kind == "time":
        for r in range(n + 1):
            p = W.tri_index(r, 0)
            f = 2.0 ** (-grow * (r - m[:r + 1]))[:, None, None]
            L[p:p + r + 1] *= f
            R[p:p + r + 1] *= f
        f = 2.0 ** (-3 * grow * (n - m))[:, None, None]
        Sl, Sg = Sl * f, Sg * f
    elif kind == "orbital":  # a row and a column of orbitals smaller than the one before it
        u = 2.0 ** (-grow * np.arange(M) * 30.0 / M)
        f = u[:, None] * u[None, :]
        Sl, Sg = Sl * f, Sg * f
        L, R = L / u[:, None] / u[None, :], R / u[:, None] / u[None, :]
        for r in range(n + 1):
            R[W.tri_index(r, r)] = -1j * np.eye(M)
    elif kind == "filling":  # G^<, Sigma^< far below G^>, Sigma^>
        L, Sl = L * 2.0 ** -40, Sl * 2.0 ** -40
    ctx = kbe.Context(M, n + 1)
    ctx.set_grid(t, order)
    ctx.set_model(W.goe_h(M, seed), np.ones(M), W.site_potential(M), None)
    return ctx, t, order, L, R, Sl, Sg


SIZES = [(3, 560, 0.5), (5, 269, 0.75), (8, 127, 1.0), (12, 73, 2.0), (16, 47, 3.0), (24, 26, 4.0), (33, 16, 8.0)]


@pytest.mark.parametrize("M,n,grow", SIZES)
@pytest.mark.parametrize("kind", ["time", "orbital", "filling"])
def test_graded_slice(kbe, M, n, grow, kind):
    import torch
    ctx, t, order, L, R, Sl, Sg = _setup(kbe, M, n, M + n, kind, grow)
    out = torch.zeros((2, n + 1, M, M), dtype=torch.complex128, device="cuda")
    ctx.history_slice(n, _dev(L), _dev(R), _dev(Sl), _dev(Sg), out)
    assert ctx.last_launch_count == 3
    ctx.sync_status()
    cols = _sample(n)
    Gl, Gg, Ga = _planes(M, n, L, R, cols)
    w = _weights(kbe, t, order, n)
    A = w[n][:, None, None] * (Sg.astype(CLD) - Sl.astype(CLD))
    got = out.cpu().numpy()[:, cols]
    ref, size = np.zeros((2, len(cols), M, M), CLD), np.zeros((2, len(cols), M, M))
    for s, (G, S) in enumerate(((Gl, Sl), (Gg, Sg))):
        _mm(A, G, ref[s], size[s])
        _mm((w[cols].T[:, :, None, None] * S.astype(CLD)[:, None]), Ga, ref[s], size[s])
    err = np.abs(got - ref).astype(np.float64)
    for s in range(2):
        # the largest of each row a of a column against the sizes of that row's products (I^> holds I^<)
        e, z = err[s].max(2), size[:s + 1].max(0).max(2)
        assert (e <= BOUND * z).all(), (s, (e / z).max())
    ctx.close()


@pytest.mark.parametrize("M,n,grow", SIZES)
@pytest.mark.parametrize("kind", ["time", "orbital"])
def test_graded_adjoint(kbe, M, n, grow, kind):
    """The cotangents of the self-energy row: point by point m, with cotangents
    of the slice that grow along c as the history falls."""
    import torch
    ctx, t, order, L, R, Il, Ig = _setup(kbe, M, n, 2 * M + n, kind, grow)
    Ib = np.stack([Il, Ig])
    Sl, Sg = W.random_rows(M, n, 5)
    dSl, dSg = (torch.zeros((n + 1, M, M), dtype=torch.complex128, device="cuda") for _ in range(2))
    dL = torch.zeros((n + 1, M, M), dtype=torch.complex128, device="cuda")
    ctx.adjoint_slice(n, _dev(L), _dev(R), _dev(Sl), _dev(Sg), _dev(Ib), dSl, dSg, dL, torch.zeros_like(dL), n)
    ctx.sync_status()
    pts = _sample(n)
    Gl, Gg, Ga = _adjoint_planes(M, n, L, R, pts)
    w = _weights(kbe, t, order, n)
    A, za = np.zeros((len(pts), M, M), CLD), np.zeros((len(pts), M, M))
    for I, G in ((Il, Gl), (Ig, Gg)):
        _mm(I.astype(CLD), G, A, za)
    wn = w[n][pts][:, None, None]
    for got, I, sign in ((dSl, Il, -1), (dSg, Ig, 1)):
        ref, size = sign * wn * A, np.abs(wn.astype(np.float64)) * za
        _mm(w[:, pts][:, :, None, None] * I.astype(CLD)[:, None], Ga, ref, size)
        e, z = np.abs(got.cpu().numpy()[pts] - ref).astype(np.float64).max(2), size.max(2)
        assert (e <= BOUND * z).all(), (sign, (e / z).max())
    ctx.close()
