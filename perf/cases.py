"""Performance cases of the library: what a solver of the Kadanoff-Baym
equations has it do, through its public Python entry points.

A case is a dict of plain values; ``kind`` names the call:

  run      a whole run from the uncorrelated state in one call (Run.run_steps)
  step     one KBE step of row n on a stored history (Run.step, P sweeps)
  slice    the history integrals of row n alone (Context.history_slice)
  sigma    the second-Born self-energy of every stored block (Context.selfenergy_all)
  dense    the self-energy row n for a four-index interaction (Context.selfenergy_slice)
  adjoint  the vector-Jacobian product of a history slice (Context.adjoint_slice)
  window   a window of steps and its gradient through autograd (window_final_block)
  batch    one batched step of independent systems of uneven sizes (Batch.step)

Histories are those of the model systems of the repository's configurations
(open Hubbard chains, GOE matrices; half filling; seeded nonuniform grids with
orders 1..5): free propagators with a slow decay in t - t', as correlations
give them.  The sizes follow the same configurations (M = 2, N_t = 64; M = 8 and
M = 32, N_t = 1024; M = 16, N_t = 512; batches of M = 4..24), with odd ones
between them.
"""
import math

import numpy as np
import torch

import paper_2405_08737_gb300 as kbe

RING = kbe.KBE_RING_ROWS
DECAY = 0.05   # G(t, t') falls as exp(-DECAY (t - t'))
PULSE = {"E0": 0.5, "t0": 5.0, "sigma": 1.0, "omega": 2.0}
BATCH_M = (4, 8, 12, 16, 24)
MOST_FLOPS = 6.0e11   # of a drawn case: below the batched step's


def listed():
    return [
        # a small molecule or dimer followed from t = 0: every step is tiny, launches and latency are all
        {"name": "run_dimer_m2_n64", "kind": "run", "M": 2, "n_t": 64, "precision": "fp64", "P": 2},
        # one step of a small system by a caller that steps by itself (observables between the steps)
        {"name": "step_fp64_m4_n63", "kind": "step", "M": 4, "n": 63, "precision": "fp64", "P": 2},
        # an odd orbital count early in a run: the middle of the range, nothing a multiple of anything
        {"name": "step_fp64_m5_n333", "kind": "step", "M": 5, "n": 333, "precision": "fp64", "P": 2},
        # the history integrals of the pulse-driven chain's last row, the default precision
        {"name": "slice_fp64_m8_n1023", "kind": "slice", "M": 8, "n": 1023, "precision": "fp64"},
        # the reverse sweep's block: the slice's vector-Jacobian product in the middle of a larger system's run
        {"name": "adjoint_m12_n389_r8", "kind": "adjoint", "M": 12, "n": 389, "rows": 8},
        # the tensor-core form: steps of a long run keep their digit planes
        {"name": "step_split_m8_n1023", "kind": "step", "M": 8, "n": 1023, "precision": "split", "P": 2},
        # the tensor-core form on a large matrix, from a history that was not stepped here
        {"name": "slice_split_m32_n511", "kind": "slice", "M": 32, "n": 511, "precision": "split"},
        # the double-float form
        {"name": "slice_df64_m16_n511", "kind": "slice", "M": 16, "n": 511, "precision": "df64"},
        # self-energy of a whole stored history (restart, analysis): bound by memory
        {"name": "sigma_all_m8_n1024", "kind": "sigma", "M": 8, "n_t": 1024},
        # self-energy row with Coulomb integrals
        {"name": "dense_m16_n255", "kind": "dense", "M": 16, "n": 255},
        # gradients with respect to U and the pulse through the last steps of a run
        {"name": "window_m16_n512_w2", "kind": "window", "M": 16, "n_t": 512, "w": 2, "precision": "fp64", "P": 2},
        # an ensemble of systems advanced together
        {"name": "batch_fp64_s10", "kind": "batch", "n_sys": 10, "mix": 3, "n_lo": 256, "n_hi": 768,
         "precision": "fp64", "P": 2},
    ]


# ------------------------------------------------------------------- ranges --
def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    while True:
        kind = rng.choice(["run", "step", "step", "slice", "slice", "slice", "sigma", "dense", "adjoint", "window",
                           "batch"])
        if kind == "run":
            case = {"M": rng.randint(2, 4), "n_t": rng.randint(24, 96), "precision": "fp64", "P": rng.choice([1, 2, 2, 3])}
        elif kind == "step":
            case = {"M": _log_int(rng, 2, 24), "n": _log_int(rng, 12, 1023),
                    "precision": rng.choice(["fp64", "fp64", "split", "df64"]), "P": 2}
        elif kind == "slice":
            case = {"M": _log_int(rng, 2, 32), "n": _log_int(rng, 12, 1023),
                    "precision": rng.choice(["fp64", "fp64", "split", "df64"])}
        elif kind == "sigma":
            case = {"M": _log_int(rng, 2, 24), "n_t": _log_int(rng, 16, 1024)}
        elif kind == "dense":
            case = {"M": _log_int(rng, 2, 20), "n": _log_int(rng, 12, 511)}
        elif kind == "adjoint":
            case = {"M": _log_int(rng, 2, 16), "n": _log_int(rng, 32, 511), "rows": rng.randint(1, 16)}
        elif kind == "window":
            case = {"M": _log_int(rng, 2, 16), "n_t": _log_int(rng, 40, 512), "w": rng.randint(1, 4),
                    "precision": rng.choice(["fp64", "fp64", "df64"]), "P": rng.choice([1, 2])}
        else:
            case = {"n_sys": rng.randint(2, 12), "mix": rng.randint(0, 10 ** 6), "n_lo": 64, "n_hi": 640,
                    "precision": rng.choice(["fp64", "fp64", "split"]), "P": 2}
        case = {"kind": kind, **case}
        w = work(case)
        if w["flops"] <= MOST_FLOPS and w["bytes"] <= 6.0e9:
            return case


# ------------------------------------------------------------------- inputs --
def _tri(n):
    return n * (n + 1) // 2


def _grid(n_t, dt0, sig, rng):
    z = rng.standard_normal(n_t - 1)
    k = rng.integers(1, 6, size=n_t - 1)
    t = np.zeros(n_t)
    t[1:] = np.cumsum(dt0 * np.exp(sig * z))
    order = np.zeros(n_t, np.int32)
    order[1:] = k
    return t, order


def _model(M, rng, goe=False):
    """(h0, U per orbital, site potential, density matrix of the half-filled free state)."""
    h = np.zeros((M, M), np.complex128)
    if goe:
        A = rng.normal(0.0, 1.0 / math.sqrt(M), size=(M, M))
        h[:] = (A + A.T) / 2
    else:
        for i in range(M - 1):
            h[i, i + 1] = h[i + 1, i] = -1.0
    U = np.full(M, rng.uniform(0.5, 3.0))
    v = np.arange(M) - (M - 1) / 2.0
    e, V = np.linalg.eigh(h)
    occ = V[:, : max(1, M // 2)]
    return h, U, v, (occ @ occ.conj().T).astype(np.complex128)


def _history(h, rho, t, n_rows, L, R):
    """Free two-time functions with a slow decay into the packed triangles L
    = G^<, R = G^R (blocks r (r+1)/2 + c), rows 0..n_rows-1."""
    M = h.shape[0]
    e, V = np.linalg.eigh(h)
    A = torch.as_tensor(np.einsum("ak,rk,bk->rab", V, np.exp(-1j * np.outer(t[:n_rows], e)), V.conj()), device="cuda")
    Ar = 1j * (A @ torch.as_tensor(rho, device="cuda"))
    Ah = A.conj().transpose(1, 2).contiguous()
    tt = torch.as_tensor(t[:n_rows], device="cuda")
    # row lists of about 2^17 / M blocks keep the temporaries small
    r0 = 0
    while r0 < n_rows:
        r1 = r0 + 1
        while r1 < n_rows and (_tri(r1 + 1) - _tri(r0)) * M * M <= 1 << 25:
            r1 += 1
        r = torch.repeat_interleave(torch.arange(r0, r1, device="cuda"),
                                    torch.arange(r0 + 1, r1 + 1, device="cuda"))
        c = torch.arange(_tri(r0), _tri(r1), device="cuda") - r * (r + 1) // 2
        d = torch.exp(-DECAY * (tt[r] - tt[c]))[:, None, None]
        L[_tri(r0):_tri(r1)] = torch.bmm(Ar[r], Ah[c]) * d
        R[_tri(r0):_tri(r1)] = torch.bmm(-1j * A[r], Ah[c]) * d
        r0 = r1
    q = torch.arange(n_rows, device="cuda")
    R[q * (q + 1) // 2 + q] = -1j * torch.eye(M, dtype=torch.complex128, device="cuda")


def _rhs_rows(h, L, R, n):
    """Stored right-hand sides -i h G^s(t_j, t_c) of the rows before n that a step reads."""
    hd = torch.as_tensor(h, device="cuda")
    out = {}
    for j in range(max(0, n - 5), n):
        l, r = L[_tri(j):_tri(j + 1)], R[_tri(j):_tri(j + 1)]
        out[j] = torch.stack([-1j * (hd @ l), -1j * (hd @ (l + r))])
    return out


def _sizes(case):
    """(M, n_t) of the single system of a case."""
    return case["M"], case["n_t"] if "n_t" in case else case["n"] + 1


def _system(M, n_t, rng, goe=False):
    t, order = _grid(n_t, 0.02, 0.4, rng)
    h, U, v, rho = _model(M, rng, goe)
    return {"M": M, "n_t": n_t, "t": t, "order": order, "h": h, "U": U, "v": v, "rho": rho, "pulse": PULSE}


def _batch_sizes(case):
    r = np.random.default_rng(case["mix"])
    return [(int(r.choice(BATCH_M)), int(r.integers(case["n_lo"], case["n_hi"] + 1))) for _ in range(case["n_sys"])]


def _inputs(case, seed):
    """Grid, model and random tensors of a case, on the host, from the seed alone."""
    rng = np.random.default_rng([int(seed), 77])
    kind = case["kind"]
    if kind == "batch":
        return {"systems": [_system(M, n_t, rng) for M, n_t in _batch_sizes(case)]}
    M, n_t = _sizes(case)
    x = _system(M, n_t, rng, goe=M > 24)
    if kind == "run":   # quench of U on the dimer's grid, no pulse
        x["t"], x["order"] = _grid(n_t, 0.05, 0.3, rng)
        x["pulse"] = None
    if kind == "dense":  # integrals of the Coulomb type: (pq|rs) = sum_k B^k_pq B^k_rs
        B = rng.standard_normal((2 * M, M, M))
        B = (B + B.transpose(0, 2, 1)) / 2
        T = np.tensordot(B, B, axes=(0, 0))
        x["U4"] = T / np.mean([T[p, p, p, p] for p in range(M)])
    if kind == "adjoint":
        x["dI"] = rng.standard_normal((2, n_t, M, M)) + 1j * rng.standard_normal((2, n_t, M, M))
    if kind == "window":  # the pulse acts inside the window
        x["pulse"] = dict(PULSE, t0=float(x["t"][-1]) - 0.35)
    return x


def _context(x):
    ctx = kbe.Context(x["M"], x["n_t"])
    ctx.set_grid(x["t"], x["order"])
    ctx.set_model(x["h"], x["U"], x["v"], x["pulse"])
    return ctx


def _stored_run(x):
    """A Run whose rows 0..n_t-1 hold a history and whose ring holds the
    right-hand sides that a step of the last row reads."""
    run = kbe.Run(_context(x))
    _history(x["h"], x["rho"], x["t"], x["n_t"], run.L, run.R)
    for j, f in _rhs_rows(x["h"], run.L, run.R, x["n_t"] - 1).items():
        run.F[j % RING, :, : j + 1] = f
    return run


def _sigma_row(x, run):
    n = x["n_t"] - 1
    run.ctx.selfenergy_slice(n, run.L, run.R, run.Sl, run.Sg)


def prepare(case, seed):
    x = _inputs(case, seed)
    kind = case["kind"]
    s = {"case": case, "x": x}
    if kind == "batch":
        runs = [_stored_run(y) for y in x["systems"]]
        s["runs"], s["batch"] = runs, kbe.Batch(runs)
        s["rows"] = np.array([y["n_t"] - 1 for y in x["systems"]], np.int32)
        return s
    if kind == "run":
        s["run"] = kbe.Run(_context(x))
        return s
    M, n_t = x["M"], x["n_t"]
    if kind == "window":
        ctx = _context(x)
        L, R = ctx.empty_triangle(), ctx.empty_triangle()
        n0 = n_t - case["w"]
        _history(x["h"], x["rho"], x["t"], n0, L, R)
        F = {j: f.cpu() for j, f in _rhs_rows(x["h"], L, R, n0).items()}
        s["window"] = kbe.Window(ctx, L, R, F, n0, n_t, x["h"], x["v"], x["pulse"], P=case["P"],
                                 precision=case["precision"])
        s["U"] = torch.tensor(x["U"], dtype=torch.float64, requires_grad=True)
        s["E0"] = torch.tensor(x["pulse"]["E0"], dtype=torch.float64, requires_grad=True)
        return s
    if kind == "sigma":
        ctx = _context(x)
        s["ctx"] = ctx
        s["L"], s["R"], s["Sl"], s["Sg"] = (ctx.empty_triangle() for _ in range(4))
        _history(x["h"], x["rho"], x["t"], n_t, s["L"], s["R"])
        return s
    run = _stored_run(x)
    s["run"] = run
    if kind == "dense":
        run.ctx.set_interaction(x["U4"])
    if kind in ("slice", "adjoint"):
        _sigma_row(x, run)
    if kind == "adjoint":
        lo = n_t - case["rows"]
        s["lo"] = lo
        s["dI"] = torch.as_tensor(x["dI"], device="cuda")
        s["dSl"], s["dSg"] = run.ctx.empty_rows(), run.ctx.empty_rows()
        s["dL"] = torch.zeros((_tri(n_t) - _tri(lo), M, M), dtype=torch.complex128, device="cuda")
        s["dR"] = torch.zeros_like(s["dL"])
    return s


# --------------------------------------------------------------------- pass --
def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "batch":
        s["batch"].step(s["rows"], P=case["P"], precision=case["precision"])
        out = []
        for r, n in zip(s["runs"], s["rows"]):
            lo, hi = _tri(int(n)), _tri(int(n) + 1)
            out.append([r.L[lo:hi], r.R[lo:hi], r.I.view(-1)[: 2 * (int(n) + 1) * r.ctx.M ** 2]])
        return out
    if kind == "run":
        r = s["run"]
        r.init_uncorrelated(s["x"]["rho"])
        r.run_steps(1, case["n_t"] - 1, P=case["P"], precision=case["precision"])
        return {"L": r.L, "R": r.R}
    if kind == "window":
        blk = kbe.window_final_block(s["U"], s["E0"], s["window"])
        dU, dE0 = torch.autograd.grad(2.0 * blk[0, 0].imag, (s["U"], s["E0"]))
        return {"block": blk.detach(), "dU": dU, "dE0": dE0}
    if kind == "sigma":
        s["ctx"].selfenergy_all(case["n_t"], s["L"], s["R"], s["Sl"], s["Sg"])
        return {"Sl": s["Sl"], "Sg": s["Sg"]}
    r = s["run"]
    n = case["n"]
    if kind == "dense":
        r.ctx.selfenergy_slice(n, r.L, r.R, r.Sl, r.Sg)
        return {"Sl": r.Sl, "Sg": r.Sg}
    if kind == "slice":
        r.ctx.history_slice(n, r.L, r.R, r.Sl, r.Sg, r.I, precision=case["precision"])
        return {"I": r.I}
    if kind == "step":
        r.step(n, P=case["P"], precision=case["precision"])
        lo, hi = _tri(n), _tri(n + 1)
        return {"L": r.L[lo:hi], "R": r.R[lo:hi], "F": r.F[n % RING], "I": r.I}
    s["dL"].zero_()
    s["dR"].zero_()
    r.ctx.adjoint_slice(n, r.L, r.R, r.Sl, r.Sg, s["dI"], s["dSl"], s["dSg"], s["dL"], s["dR"], s["lo"])
    return {"dSl": s["dSl"], "dSg": s["dSg"], "dL": s["dL"], "dR": s["dR"]}


# --------------------------------------------------------------------- work --
def _slice_flops(M, n):
    # term 1 over the 2n + 1 output blocks that a step needs, term 2 over m <= c
    return 8.0 * M ** 3 * (n + 1) * (3 * n + 2)


def _step_work(M, n, P):
    row = 16.0 * (n + 1) * M * M
    # both triangles once, the stored right-hand sides once; rows of L, R and F and the slice written
    return P * _slice_flops(M, n), 2 * 16.0 * _tri(n) * M * M + 10 * row + 6 * row


def work(case):
    kind = case["kind"]
    if kind == "batch":
        w = [_step_work(M, n_t - 1, case["P"]) for M, n_t in _batch_sizes(case)]
        return {"flops": sum(f for f, _ in w), "bytes": sum(b for _, b in w)}
    M, n_t = _sizes(case)
    n = n_t - 1
    row = 16.0 * n_t * M * M
    if kind == "run":
        # the rows are written once; what a step reads stays on the chip at these sizes
        return {"flops": sum(case["P"] * _slice_flops(M, j) for j in range(1, n_t)), "bytes": 2 * 16.0 * _tri(n_t) * M * M}
    if kind == "step":
        f, b = _step_work(M, n, case["P"])
        return {"flops": f, "bytes": b}
    if kind == "slice":
        return {"flops": _slice_flops(M, n), "bytes": 2 * 16.0 * _tri(n_t) * M * M + 4 * row}
    if kind == "sigma":
        return {"flops": 40.0 * _tri(n_t) * M * M, "bytes": 4 * 16.0 * _tri(n_t) * M * M}
    if kind == "dense":
        return {"flops": 2 * 24.0 * M ** 5 * n_t, "bytes": 4 * row + 8.0 * M ** 4}
    if kind == "adjoint":
        # the cotangent of the self-energy row (three sums over m, c) and of the last rows
        rows = case["rows"]
        return {"flops": 24.0 * M ** 3 * n_t ** 2 + 3 * 16.0 * M ** 3 * rows * n_t,
                "bytes": 2 * 16.0 * _tri(n_t) * M * M + 6 * row + 2 * 16.0 * (_tri(n_t) - _tri(n_t - rows)) * M * M}
    # window: the steps, then their recomputation and the slices' adjoints
    f = b = 0.0
    for j in range(n_t - case["w"], n_t):
        sf, sb = _step_work(M, j, case["P"])
        f += 2 * sf + case["P"] * 24.0 * M ** 3 * (j + 1) ** 2
        b += 2 * sb
    return {"flops": f, "bytes": b}


# ------------------------------------------------- the same in 64 bits, plainly --
_GL_X, _GL_W = np.polynomial.legendre.leggauss(8)


def _local(tau, lo, hi):
    """Weights of the interpolatory rule through the nodes tau over [lo, hi]."""
    u = 0.5 * (lo + hi) + 0.5 * (hi - lo) * _GL_X
    w = np.empty(len(tau))
    for i in range(len(tau)):
        p = np.ones_like(u)
        for j in range(len(tau)):
            if j != i:
                p *= (u - tau[j]) / (tau[i] - tau[j])
        w[i] = 0.5 * (hi - lo) * np.dot(_GL_W, p)
    return w


def _weights(t, order):
    """Composite rows w[c, m] of the grid."""
    N = len(t)
    w = np.zeros((N, N))
    for c in range(1, N):
        k = min(int(order[c]), c)
        w[c] = w[c - 1]
        w[c, c - k:c + 1] += _local(t[c - k:c + 1], t[c - 1], t[c])
    return torch.as_tensor(w, device="cuda")


def _plane(T, N):
    """[(m, x), (c, b)] matrix of T over the whole plane: T(m, c), or -T(c, m)^+ above the diagonal."""
    M = T.shape[-1]
    i = torch.arange(N, device=T.device)
    hi, lo = torch.maximum(i[:, None], i[None, :]), torch.minimum(i[:, None], i[None, :])
    X = T[(hi * (hi + 1) // 2 + lo).reshape(-1)].reshape(N, N, M, M)
    X = torch.where((i[:, None] < i[None, :])[:, :, None, None], -X.transpose(2, 3).conj(), X)
    return X.permute(0, 2, 1, 3).reshape(N * M, N * M)


def _slice64(w, L, R, Sl, Sg):
    """I^<, I^> of the last row n = N - 1 from the packed rows 0..n."""
    N, M = Sl.shape[0], Sl.shape[-1]
    n = N - 1
    A1 = (w[n, :N, None, None] * (Sg - Sl)).permute(1, 0, 2).reshape(M, N * M)
    T1 = A1 @ _plane(L[:_tri(N)], N)
    T1g = T1 + A1 @ _plane(R[:_tri(N)], N)
    out = [x.reshape(M, N, M).permute(1, 0, 2) for x in (T1, T1g)]
    i = torch.arange(N, device=L.device)
    t2 = [[], []]
    step = max(1, (1 << 23) // (N * M * M))
    for c0 in range(0, N, step):
        c = i[c0:c0 + step]
        low = i[None, :] <= c[:, None]
        idx = torch.where(low, c[:, None] * (c[:, None] + 1) // 2 + i[None, :], 0)
        wc = torch.where(low, w[c, :N], torch.zeros((), dtype=w.dtype, device=w.device))
        Rc = R[idx.reshape(-1)].reshape(len(c), N, M, M).conj().permute(0, 1, 3, 2).reshape(len(c), N * M, M)
        for s, S in enumerate((Sl, Sg)):
            WS = (wc[:, :, None, None] * S[None]).permute(0, 2, 1, 3).reshape(len(c), M, N * M)
            t2[s].append(torch.bmm(WS, Rc))
    return torch.stack([out[s] + torch.cat(t2[s]) for s in range(2)])


def _sigma64(U, l, g, diag):
    """Self-energy of blocks l = G^<, g = G^>; diag: the index of the equal-time block, or None."""
    uu = (U[:, None] * U[None, :])
    fl, fg = l.conj(), g.conj()
    sg, sl = -uu * g * g * fl, -uu * l * l * fg
    if diag is not None:
        ld, gd = l[diag], g[diag]
        sg = torch.cat([sg[:diag], (uu * gd * gd * ld.transpose(-1, -2))[None], sg[diag + 1:]])
        sl = torch.cat([sl[:diag], (uu * ld * ld * gd.transpose(-1, -2))[None], sl[diag + 1:]])
    return sl, sg


def _field64(p, t):
    return 0.0 if p is None else math.exp(-0.5 * ((t - p["t0"]) / p["sigma"]) ** 2) * math.cos(p["omega"] * t)


def _step64(x, w, L, R, F, n, P, U, E0):
    """Row n from the packed rows 0..n-1 and the right-hand sides F[j]: (L row, R row, F row, slice)."""
    M, t, k = x["M"], x["t"], int(x["order"][n])
    dev = L.device
    eye = -1j * torch.eye(M, dtype=torch.complex128, device=dev)
    h = torch.as_tensor(x["h"], device=dev)
    v = torch.as_tensor(x["v"], device=dev)
    l0, g0 = L[_tri(n - 1):_tri(n)], L[_tri(n - 1):_tri(n)] + R[_tri(n - 1):_tri(n)]

    def adams(Fn):
        new = Fn is not None   # the corrector also uses t_n
        wt = {}
        for q in range(1, min(k, n) + 1):
            wt[q] = _local(t[n - q:n + 1] if new else t[n - q:n], t[n - 1], t[n])
        gl, gg = [], []
        far = max(0, n - k + 1)   # the columns below take all min(k, n) points
        groups = [(0, far, min(k, n))] + [(c, c + 1, n - c) for c in range(far, n)]
        for c0, c1, q in groups:
            if c1 <= c0:
                continue
            al, ag = l0[c0:c1], g0[c0:c1]
            for p, wp in enumerate(wt[q]):
                f = Fn if n - q + p == n else F[n - q + p]
                al, ag = al + wp * f[0, c0:c1], ag + wp * f[1, c0:c1]
            gl.append(al)
            gg.append(ag)
        q = min(k, n)
        d = L[_tri(n) - 1]
        for p, wp in enumerate(wt[q]):
            j = n - q + p
            f = (Fn if j == n else F[j])[0, j]
            d = d + wp * (f - f.transpose(0, 1).conj())
        gl, gg = torch.cat(gl), torch.cat(gg)
        return torch.cat([gl, d[None]]), torch.cat([gg - gl, eye[None]])

    ln, rn = adams(None)
    for _ in range(P):
        Sl, Sg = _sigma64(U, ln, ln + rn, n)
        La, Ra = torch.cat([L[:_tri(n)], ln]), torch.cat([R[:_tri(n)], rn])
        I = _slice64(w, La, Ra, Sl, Sg)
        eps = h + torch.diag(E0 * _field64(x["pulse"], t[n]) * v + U * torch.diagonal(ln[n]).imag)
        Fn = torch.stack([-1j * (eps @ ln + I[0]), -1j * (eps @ (ln + rn) + I[1])])
        ln, rn = adams(Fn)
    return ln, rn, Fn, I


def _triangles(x, n_rows):
    M = x["M"]
    L = torch.zeros((_tri(n_rows), M, M), dtype=torch.complex128, device="cuda")
    R = torch.zeros_like(L)
    _history(x["h"], x["rho"], x["t"], n_rows, L, R)
    return L, R


def _exact_step(x, n, P):
    L, R = _triangles(x, n)
    F = _rhs_rows(x["h"], L, R, n)
    U = torch.as_tensor(x["U"], device="cuda")
    E0 = 0.0 if x["pulse"] is None else x["pulse"]["E0"]
    return _step64(x, _weights(x["t"], x["order"]), L, R, F, n, P, U, E0)


def _exact_dense(x):
    M, n = x["M"], x["n_t"] - 1
    L, R = _triangles(x, n + 1)
    l, g = L[_tri(n):], L[_tri(n):] + R[_tri(n):]
    U4 = torch.as_tensor(x["U4"], device="cuda").to(torch.complex128)
    X = 2.0 * U4.permute(0, 2, 1, 3) - U4   # UEx_jabc = 2 U_jbac - U_jabc
    X = X.permute(0, 2, 1, 3).reshape(M, -1)   # [j, (b, a, c)]
    A = U4.permute(0, 2, 3, 1).reshape(M ** 3, M)   # [(i, d, e), f]

    def one(G, H):   # U_ifde UEx_jabc G_fb G_ea H_cd, H(t', t)
        Y = (A @ G).reshape(M, M, M, M).permute(0, 1, 3, 2).reshape(M ** 3, M)   # [(i, d, b), e]
        Y = (Y @ G).reshape(M, M, M, M).permute(0, 2, 3, 1).reshape(M ** 3, M)   # [(i, b, a), d]
        Z = (Y @ H.transpose(0, 1)).reshape(M, -1)   # [i, (b, a, c)]
        return Z @ X.transpose(0, 1)

    Sl, Sg = [], []
    for c in range(n + 1):
        hl, hg = (l[c], g[c]) if c == n else (-l[c].transpose(0, 1).conj(), -g[c].transpose(0, 1).conj())
        Sl.append(one(l[c], hg))
        Sg.append(one(g[c], hl))
    return torch.stack(Sl), torch.stack(Sg)


def exact(case, seed):
    kind = case["kind"]
    x = _inputs(case, seed)
    if kind == "batch":
        out = []
        for y in x["systems"]:
            ln, rn, _, I = _exact_step(y, y["n_t"] - 1, case["P"])
            out.append([ln, rn, I.reshape(-1)])
        return out
    M, n_t = x["M"], x["n_t"]
    n = n_t - 1
    U = torch.as_tensor(x["U"], device="cuda")
    w = _weights(x["t"], x["order"])
    if kind == "run":
        L = (1j * torch.as_tensor(x["rho"], device="cuda"))[None]
        R = -1j * torch.eye(M, dtype=torch.complex128, device="cuda")[None]
        Sl, Sg = _sigma64(U, L, L + R, 0)
        I = _slice64(w, L, R, Sl, Sg)
        eps = torch.as_tensor(x["h"], device="cuda") + torch.diag(U * torch.diagonal(L[0]).imag)
        F = {0: torch.stack([-1j * (eps @ L + I[0]), -1j * (eps @ (L + R) + I[1])])}
        for j in range(1, n_t):
            ln, rn, Fn, _ = _step64(x, w, L, R, F, j, case["P"], U, 0.0)
            L, R = torch.cat([L, ln]), torch.cat([R, rn])
            F[j] = Fn
        return {"L": L, "R": R}
    if kind == "step":
        ln, rn, Fn, I = _exact_step(x, n, case["P"])
        return {"L": ln, "R": rn, "F": Fn, "I": I}
    if kind == "window":
        n0 = n_t - case["w"]
        L, R = _triangles(x, n0)
        F = _rhs_rows(x["h"], L, R, n0)
        Ud = U.clone().requires_grad_(True)
        Ed = torch.tensor(x["pulse"]["E0"], dtype=torch.float64, device="cuda", requires_grad=True)
        for j in range(n0, n_t):
            ln, rn, F[j], _ = _step64(x, w, L, R, F, j, case["P"], Ud, Ed)
            L, R = torch.cat([L, ln]), torch.cat([R, rn])
        dU, dE0 = torch.autograd.grad(2.0 * L[-1][0, 0].imag, (Ud, Ed))
        return {"block": L[-1].detach(), "dU": dU, "dE0": dE0}
    if kind == "dense":
        Sl, Sg = _exact_dense(x)
        return {"Sl": Sl, "Sg": Sg}
    L, R = _triangles(x, n_t)
    if kind == "sigma":
        uu = U[:, None] * U[None, :]
        l, g = L, L + R
        sg, sl = -uu * g * g * l.conj(), -uu * l * l * g.conj()
        q = torch.arange(n_t, device="cuda")
        q = q * (q + 1) // 2 + q
        ld, gd = l[q], g[q]
        sg[q], sl[q] = uu * gd * gd * ld.transpose(1, 2), uu * ld * ld * gd.transpose(1, 2)
        return {"Sl": sl, "Sg": sg}
    Sl, Sg = _sigma64(U, L[_tri(n):], L[_tri(n):] + R[_tri(n):], n)
    if kind == "slice":
        return {"I": _slice64(w, L, R, Sl, Sg)}
    leaves = [y.detach().requires_grad_(True) for y in (Sl, Sg, L, R)]
    I = _slice64(w, leaves[2], leaves[3], leaves[0], leaves[1])
    dSl, dSg, dL, dR = torch.autograd.grad(I, leaves, torch.as_tensor(x["dI"], device="cuda"))
    q = torch.arange(n_t, device="cuda")
    dR[q * (q + 1) // 2 + q] = 0.0
    lo = _tri(n_t - case["rows"])
    return {"dSl": dSl, "dSg": dSg, "dL": dL[lo:], "dR": dR[lo:]}
