// history_df.cu -- history slice of Eq. (KBE2) (Sec. 2) in double-float
// arithmetic on the FP32 pipe (precision KBE_DF64).
//
// The same sums as history_f64.cu,
//   I^<(n,c) = sum_m A1[m] G^<(m,c) + sum_{m<=c} B^<[m] G^A(m,c),
//   I^>(n,c) = sum_m A1[m] G^>(m,c) + sum_{m<=c} B^>[m] G^A(m,c),
// with A1[m] = w_{n,m} (S^> - S^<)[m], B^s[m] = wbar_m S^s[m] (w_{c,m} S^s[m]
// in the band m > c - K - 1).  With the planes PL(m,c) = L(m,c), Q(m,c) =
// R(m,c) below and on the diagonal and PL = -L(c,m)^+, Q = -R(c,m)^+ above it
// (G^< = PL, G^> = PL + Q, G^A = -Q for m < c), and with the part of the
// settled points that cancels between the terms left out (w_{n,m} = wbar_m
// there; see history_partial_entry), two products per point are summed:
//   I^<       = sum_m A1[m] PL(m,c) - sum_{m<c, settled} B^<[m] Q(m,c) + band^<,
//   I^> - I^< = sum_{m > c - K - 1} A1[m] Q(m,c) + band^> - band^<.
// (The slice n = 511, M = 16 took 6.57 ms with all the products, 4.63 ms with
// these.)
//
// GB300 issues 64 FP32 operations per FP64 operation, so a complex
// multiply-add done as four double-float products (each hi*hi, its FMA
// error and the two cross terms, about 2^-47 relative) with Ogita-Rump-Oishi
// compensated accumulation (a TwoSum per term, the errors in a float tail)
// costs about 48 FP32 operations where FP64 needs 4 DFMA: at the two pipes'
// rates the slice runs about four times faster than on the FP64 pipe, with
// an error of order 1e-14 of the terms' sizes (Sec. 3.2's quadrature and
// the history are FP64 inputs, converted once per use to hi + lo floats).
//
// Layout.  A prep kernel forms A1, B^<, B^> in FP64 (as history_prep) and
// stores them as double-float (float4: re.hi, re.lo, im.hi, im.lo) rows.
// One thread owns one output column entry (c, b) for a group of 2 values of
// a and both s: each history entry it loads is converted once and used for
// its 2 values of a; the self-energy operands are shared by the warp
// (broadcast loads).  The history index m is split into chunks across
// grid.y; per-chunk partials go to the workspace as FP64 and the FP64
// reduction adds them in chunk order (deterministic).

#include <algorithm>

#include "dfloat.cuh"
#include "row_kernels.cuh"

namespace kbe {
namespace {

constexpr int kNA = 2;          // values of a per thread
constexpr int kDfBlock = 128;   // threads per block
// shared memory of a history_df_tiled block: 32 KB (two history points per
// tile at M = 8, seven blocks per SM) measured faster than 64 KB (four
// points, three blocks): 2.14 against 2.72 ms for the slice n = 767, M = 8
constexpr size_t kTileSmem = 32 * 1024;

struct DfArgs {
  int M, MM, n, AG;             // AG = ceil(M / kNA) groups of a
  int chunk_len;
  const double* L;
  const double* R;
  const double* Sl;             // raw row n (band points of term 2)
  const double* Sg;
  const float4* A1;             // double-float rows [n+1][M][M]
  const float4* NB;             // -wbar S^<
  WeightsView w;
  double* dst;                  // partials [chunk][2][n+1][MM] or the output
};

using df::Acc;
using df::c2f;
using df::cconj;
using df::cmac;
using df::cneg;

__global__ void __launch_bounds__(256) history_df_prep(int MM, int n, const double* __restrict__ Sl,
                                                       const double* __restrict__ Sg, WeightsView w,
                                                       float4* __restrict__ A1, float4* __restrict__ NB) {
  const int64_t total = (int64_t)(n + 1) * MM;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int m = (int)(e / MM);
    const double wn = w.at(n, m), wb = w.wbar[m];
    const double2 l = reinterpret_cast<const double2*>(Sl)[e];
    const double2 g = reinterpret_cast<const double2*>(Sg)[e];
    A1[e] = c2f(make_double2(wn * (g.x - l.x), wn * (g.y - l.y)));
    NB[e] = c2f(make_double2(-wb * l.x, -wb * l.y));
  }
}

// One thread's sums for its values of a: I^< and D = I^> - I^< (re, im).
struct Sums {
  Acc lr[kNA], li[kNA], dr[kNA], di[kNA];
  __device__ __forceinline__ Sums() {
#pragma unroll
    for (int k = 0; k < kNA; ++k) lr[k] = li[k] = dr[k] = di[k] = Acc{0.f, 0.f};
  }
};

// History point m, orbital x of column c's entry b: pl, q are the planes'
// values, s1 and nb the operand rows of the thread's first a at stride `as`.
__device__ __forceinline__ void point(const DfArgs& p, Sums& t, int m, int c, int a0, int na, int x, int b, float4 pl,
                                      float4 q, const float4* s1, const float4* nb, int as) {
  if (m <= c - p.w.band_w) {  // settled: the same for I^< and I^>
#pragma unroll
    for (int k = 0; k < kNA; ++k) {
      if (k < na) {
        cmac(t.lr[k], t.li[k], s1[(int64_t)k * as], pl);
        cmac(t.lr[k], t.li[k], nb[(int64_t)k * as], q);
      }
    }
    return;
  }
#pragma unroll
  for (int k = 0; k < kNA; ++k) {
    if (k < na) {
      const float4 v = s1[(int64_t)k * as];
      cmac(t.lr[k], t.li[k], v, pl);
      cmac(t.dr[k], t.di[k], v, q);
    }
  }
  if (m > c) return;
  // term 2 in the band, with the exact weight: w_{c,m} S^s G^A.  Four FP64 operations per a, as many
  // as two weighted values take: they bound the short slices, most of which are band (with S^> - S^< formed
  // first, which takes two more, M = 16, n = 13 took 44 us instead of 41, M = 64, n = 3 157 instead of 146).
  const int M = p.M;
  const double wcm = p.w.at(c, m);
  float4 ga = cneg(q);
  if (m == c)  // G^A(c,c)_xb = conj(R(c,c)_bx)
    ga = cconj(c2f(reinterpret_cast<const double2*>(p.R)[tri(c, c) * p.MM + b * M + x]));
  const double2* sl = reinterpret_cast<const double2*>(p.Sl) + ((int64_t)m * M + a0) * M + x;
  const double2* sg = reinterpret_cast<const double2*>(p.Sg) + ((int64_t)m * M + a0) * M + x;
#pragma unroll
  for (int k = 0; k < kNA; ++k) {
    if (k < na) {
      const double2 vl = sl[(int64_t)k * M], vg = sg[(int64_t)k * M];
      const double2 wl = make_double2(wcm * vl.x, wcm * vl.y);
      cmac(t.lr[k], t.li[k], c2f(wl), ga);
      cmac(t.dr[k], t.di[k], c2f(make_double2(fma(wcm, vg.x, -wl.x), fma(wcm, vg.y, -wl.y))), ga);
    }
  }
}

__device__ __forceinline__ void store_sums(const DfArgs& p, const Sums& t, int chunk, int c, int a0, int na, int b) {
  double2* d = reinterpret_cast<double2*>(p.dst);
  const int64_t stride_s = (int64_t)(p.n + 1) * p.MM;
  const int64_t base = (int64_t)chunk * 2 * stride_s + (int64_t)c * p.MM + b;
#pragma unroll
  for (int k = 0; k < kNA; ++k) {
    if (k < na) {
      const int64_t e = base + (int64_t)(a0 + k) * p.M;
      const double2 l = make_double2((double)t.lr[k].s + (double)t.lr[k].c, (double)t.li[k].s + (double)t.li[k].c);
      d[e] = l;
      d[e + stride_s] = make_double2(l.x + ((double)t.dr[k].s + (double)t.dr[k].c),
                                     l.y + ((double)t.di[k].s + (double)t.di[k].c));
    }
  }
}

__global__ void __launch_bounds__(kDfBlock) history_df_partial(DfArgs p) {
  const int M = p.M, MM = p.MM, n = p.n, AG = p.AG;
  // column blocks from the last column down: the heavier blocks of each
  // chunk (columns past it carry both terms) start first
  const int64_t t = (int64_t)(gridDim.x - 1 - blockIdx.x) * blockDim.x + threadIdx.x;
  if (t >= (int64_t)(n + 1) * AG * M) return;
  const int c = (int)(t / ((int64_t)AG * M));
  const int r = (int)(t - (int64_t)c * AG * M);
  const int ag = r / M, b = r - ag * M;
  const int a0 = ag * kNA;
  const int na = min(kNA, M - a0);
  const int chunk = blockIdx.y;
  const int m0 = chunk * p.chunk_len;
  const int m1 = min(n + 1, m0 + p.chunk_len);

  Sums sum;
  const double2* L = reinterpret_cast<const double2*>(p.L);
  const double2* R = reinterpret_cast<const double2*>(p.R);

  for (int m = m0; m < m1; ++m) {
    // this thread's column b of the planes at (m,c): block (m,c) row x for
    // m >= c; block (c,m) row b, transposed, conjugated and negated, for m < c
    const bool direct = m >= c;
    const int64_t blk = direct ? tri(m, c) * MM : tri(c, m) * MM;
    const float4* a1 = p.A1 + ((int64_t)m * M + a0) * M;
    const float4* nb = p.NB + ((int64_t)m * M + a0) * M;
    for (int x = 0; x < M; ++x) {
      float4 pl, q;
      if (direct) {
        pl = c2f(L[blk + x * M + b]);
        q = c2f(R[blk + x * M + b]);
      } else {
        pl = cneg(cconj(c2f(L[blk + b * M + x])));
        q = cneg(cconj(c2f(R[blk + b * M + x])));
      }
      point(p, sum, m, c, a0, na, x, b, pl, q, a1 + x, nb + x, M);
    }
  }
  store_sums(p, sum, chunk, c, a0, na, b);
}

// Shared-memory form for M <= 32: a block owns CB output columns and AGB
// groups of a; per tile of TM history points it loads the G blocks its
// columns read and the operand rows of its values of a once, converts them
// once (instead of once per thread that reads them), and every thread then
// reads its operands from shared memory.  Same arithmetic in the same order
// per output as history_df_partial.
struct TileGeom {
  int CB, AGB, TM;    // columns, groups of a, history points per block tile
  int col_tiles, ag_tiles;
};

__global__ void __launch_bounds__(kDfBlock) history_df_tiled(DfArgs p, TileGeom tg) {
  extern __shared__ float4 sm[];
  const int M = p.M, MM = p.MM, n = p.n, AG = p.AG;
  const int CB = tg.CB, AGB = tg.AGB, TM = tg.TM, NAB = AGB * kNA;
  float4* sG = sm;                                  // [TM][CB][2][MM]: PL, Q as [x][b]
  float4* sS = sm + (size_t)TM * CB * 2 * MM;       // [TM][2][NAB][M]: A1, -B^< rows
  // column tiles from the last one down (heavier tiles of each chunk first)
  const int bx = (int)(gridDim.x - 1 - blockIdx.x);
  const int ct = bx / tg.ag_tiles, at = bx - ct * tg.ag_tiles;
  const int c_base = ct * CB, ag_base = at * AGB;
  const int a_base = ag_base * kNA;
  const int tid = threadIdx.x;
  const int cl = tid / (AGB * M), rr0 = tid - cl * AGB * M;
  const int agl = rr0 / M, b = rr0 - agl * M;
  const int c = c_base + cl;
  const int a0 = (ag_base + agl) * kNA;
  const bool live = cl < CB && c <= n && ag_base + agl < AG;
  const int na = live ? min(kNA, M - a0) : 0;
  const int chunk = blockIdx.y;
  const int m0 = chunk * p.chunk_len;
  const int m1 = min(n + 1, m0 + p.chunk_len);
  const double2* L = reinterpret_cast<const double2*>(p.L);
  const double2* R = reinterpret_cast<const double2*>(p.R);
  const int nab = min(NAB, M - a_base);  // values of a of this block

  Sums sum;

  for (int mt = m0; mt < m1; mt += TM) {
    const int tm = min(TM, m1 - mt);
    __syncthreads();
    // G blocks of the block's columns: (m, c) read directly for m >= c,
    // (c, m) transposed for m < c
    const int g_items = tm * CB * MM;
    for (int i = tid; i < g_items; i += kDfBlock) {
      const int mi = i / (CB * MM), r = i - mi * CB * MM;
      const int cc = r / MM, e = r - cc * MM;
      const int m = mt + mi, col = c_base + cc;
      if (col > n) continue;
      float4* dst = sG + ((size_t)(mi * CB + cc) * 2) * MM;
      if (m >= col) {
        const int64_t blk = tri(m, col) * MM;
        dst[e] = c2f(L[blk + e]);
        dst[MM + e] = c2f(R[blk + e]);
      } else {
        const int64_t blk = tri(col, m) * MM;   // stored entry (b, x) at e = b M + x
        const int bb = e / M, x = e - bb * M;
        const int et = x * M + bb;
        dst[et] = cneg(cconj(c2f(L[blk + e])));
        dst[MM + et] = cneg(cconj(c2f(R[blk + e])));
      }
    }
    // operand rows of the block's values of a
    const int s_items = tm * 2 * nab * M;
    for (int i = tid; i < s_items; i += kDfBlock) {
      const int mi = i / (2 * nab * M), r = i - mi * 2 * nab * M;
      const int v = r / (nab * M), e = r - v * nab * M;   // e = (a - a_base) M + x
      const float4* src = v == 0 ? p.A1 : p.NB;
      sS[((size_t)(mi * 2 + v) * NAB) * M + e] = src[((int64_t)(mt + mi) * M + a_base) * M + e];
    }
    __syncthreads();
    if (!live) continue;
    for (int mi = 0; mi < tm; ++mi) {
      const int m = mt + mi;
      const float4* g = sG + ((size_t)(mi * CB + cl) * 2) * MM + b;
      const float4* s1 = sS + ((size_t)(mi * 2 + 0) * NAB + (a0 - a_base)) * M;
      const float4* nb = sS + ((size_t)(mi * 2 + 1) * NAB + (a0 - a_base)) * M;
      for (int x = 0; x < M; ++x) point(p, sum, m, c, a0, na, x, b, g[x * M], g[MM + x * M], s1 + x, nb + x, M);
    }
  }
  if (live) store_sums(p, sum, chunk, c, a0, na, b);
}

// Block tiling of history_df_tiled for M orbitals and n + 1 columns, within
// smem_max bytes of shared memory; false for orbital counts it does not take.
bool tile_geom(int M, int n, size_t smem_max, TileGeom* tg, size_t* smem) {
  if (M > 32) return false;
  const int AG = (M + kNA - 1) / kNA, TPC = AG * M;
  if (TPC <= kDfBlock) {
    tg->CB = kDfBlock / TPC;
    tg->AGB = AG;
  } else {
    tg->CB = 1;
    tg->AGB = kDfBlock / M;
  }
  const size_t per_m = ((size_t)tg->CB * 2 * M * M + (size_t)2 * tg->AGB * kNA * M) * sizeof(float4);
  tg->TM = (int)std::max<size_t>(1, std::min<size_t>(8, smem_max / per_m));
  if (per_m > smem_max) return false;
  *smem = per_m * tg->TM;
  tg->col_tiles = (n + 1 + tg->CB - 1) / tg->CB;
  tg->ag_tiles = (AG + tg->AGB - 1) / tg->AGB;
  return true;
}

inline unsigned grid_for(int64_t n, int64_t cap) {
  int64_t b = (n + 255) / 256;
  return (unsigned)(b < 1 ? 1 : (b > cap ? cap : b));
}

}  // namespace

// Workspace as launch_history_f64: the two double-float operand rows take
// the places of A1, Bl (16 bytes per complex either way), then the
// per-chunk partials.
cudaError_t launch_history_df(const HistoryArgs& a, cudaStream_t s, int* launches) {
  const int M = a.M, MM = M * M, n = a.n;
  const int AG = (M + kNA - 1) / kNA;
  const int64_t row = (int64_t)(n + 1) * MM;
  const int64_t threads = (int64_t)(n + 1) * AG * M;
  // enough threads for full occupancy, and chunks of at most ~32 history
  // points so that a block's work stays short
  int64_t want = std::max<int64_t>(((int64_t)sm_count() * 2048 + threads - 1) / threads, (n + 1 + 31) / 32);
  int nchunk = (int)std::min<int64_t>(std::max<int64_t>(want, 1), kMaxSplit);
  if (nchunk > n + 1) nchunk = n + 1;
  const size_t prep_bytes = (size_t)2 * row * 16;
  while (nchunk > 1 && prep_bytes + (size_t)nchunk * 2 * row * 16 > a.part_bytes) --nchunk;
  if (prep_bytes + (nchunk > 1 ? (size_t)nchunk * 2 * row * 16 : 0) > a.part_bytes) return cudaErrorInvalidValue;
  const int chunk_len = (n + 1 + nchunk - 1) / nchunk;
  nchunk = (n + 1 + chunk_len - 1) / chunk_len;

  float4* A1 = reinterpret_cast<float4*>(a.part);
  float4* NB = A1 + row;
  double* partials = a.part + 4 * row;
  int nl = 0;
  history_df_prep<<<grid_for(row, sm_count() * 8), 256, 0, s>>>(MM, n, a.Sl, a.Sg, a.w, A1, NB);
  ++nl;
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) { *launches = nl; return e; }
  DfArgs p{M, MM, n, AG, chunk_len, a.L, a.R, a.Sl, a.Sg, A1, NB, a.w, nchunk == 1 ? a.out : partials};
  TileGeom tg;
  size_t smem = 0;
  const bool tiled = tile_geom(M, n, kTileSmem, &tg, &smem);
  // (no attribute call at or below the default 48 KB, so that the launch can
  // be recorded in a graph capture)
  if (tiled && kTileSmem > 48 * 1024 &&
      (e = cudaFuncSetAttribute(history_df_tiled, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)kTileSmem)) != cudaSuccess) {
    *launches = nl;
    return e;
  }
  if (a.ev_begin) cudaEventRecord(a.ev_begin, s);
  if (tiled) {
    dim3 grid((unsigned)((int64_t)tg.col_tiles * tg.ag_tiles), (unsigned)nchunk);
    history_df_tiled<<<grid, kDfBlock, smem, s>>>(p, tg);
  } else {
    dim3 grid((unsigned)((threads + kDfBlock - 1) / kDfBlock), (unsigned)nchunk);
    history_df_partial<<<grid, kDfBlock, 0, s>>>(p);
  }
  if (a.ev_end) cudaEventRecord(a.ev_end, s);
  ++nl;
  if ((e = cudaGetLastError()) != cudaSuccess) { *launches = nl; return e; }
  int nr = 0;
  e = launch_history_finish(nchunk, row, partials, a.out, a.status, s, &nr);
  *launches = nl + nr;
  return e;
}

}  // namespace kbe
