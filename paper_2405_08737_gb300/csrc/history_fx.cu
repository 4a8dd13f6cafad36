// history_fx.cu -- FP64 history slice of Eq. (KBE2) (Sec. 2) on the 16-bit-float
// tensor cores (tcgen05), by error-free slicing into eight digits per value
// (fx_common.cuh).
//
// The sums are those of history_f64.cu.  With the planes PL(m,c) = L(m,c),
// Q(m,c) = R(m,c) for m >= c and PL = -L(c,m)^+, Q = -R(c,m)^+ for m < c
// (G^< = PL, G^> = PL + Q), A1[m] = w_{n,m} (S^> - S^<)[m], NB[m] = -wbar_m S^<[m]:
//   far  (m <= c - band_w): I^< += A1 PL + NB Q          (both components alike)
//   near (m >  c - band_w): I^< += A1 PL,  D += A1 Q      (I^> = I^< + D)
// and the band of term 2, w_{c,m} S^s R(c,m)^+ for c - band_w < m <= c, is added
// in FP64 by the reduction: two real products of 128-row tiles per history point.
//
// Why: FP64 runs at 1.26 TFLOP/s on this part (152 SMs x 2 FMA), the fp16
// tensor cores at about 1900, so 36 digit products cost a fiftieth of the FP64
// ones.  What bounds it then is the conversion: every history entry is read in
// both orientations and cut into digits with about 30 integer instructions per
// real.  Measured: the slice n = 1023, M = 8 in 0.87 ms, 0.97 with the kernels around
// it, where the same sums on the FP64 pipe (history_f64.cu) take 7.08 ms.
//
// One persistent CTA per SM takes a contiguous range of chunks (32 history
// entries of a 128-row column tile).  A unit is 8 entries, one MMA K step:
//  * 16 converter warps, each owning 8 rows: a lane holds 4 entries of one row
//    of one plane, loaded one unit ahead straight into registers (staging them
//    in shared memory would cost as much of its bandwidth as the digits), finds
//    the row's exponent with its neighbours and writes the digit planes
//    (2 x 32 KB per unit) into a ring of two stages;
//  * one thread copies the small operand's digits of each unit (bulk copies);
//  * one thread issues the MMAs: digit i of the history against the stacked
//    digits 0..7-i of the small operand, so the products of level i + j land in
//    the columns of that level (N = 2 kNA (8 - i));
//  * eight epilogue warps fold a chunk's eight integer levels into one 64-bit
//    integer, and that, scaled, into FP64 sums in registers: two FP64
//    operations per 32 entries of an output.
// A row's exponent holds for the units accumulated together in tensor memory.
// It starts kHeadroom bits above the larger of the unit's and the previous
// chunk's largest entry; a unit that exceeds it nevertheless closes the
// accumulation and starts the next with the larger exponent.
//
// Partial sums go to one slot per (CTA, tile) and are added in CTA order, so
// results are bitwise reproducible.  All waits are bounded.  A row or a small
// operand that holds a non-finite value gives NaN in the outputs it enters, as
// on the FP64 path, and the reduction reports it.

#include <algorithm>
#include <atomic>

#include "fx_common.cuh"
#include "kbe_internal.h"
#include "row_kernels.cuh"
#include "split_common.cuh"

namespace kbe {
namespace {

using namespace fx;
using split::bulk_g2s;
using split::fence_async_smem;
using split::mbar_arrive;
using split::mbar_arrive_expect_tx;
using split::mbar_init;
using split::mbar_try;
using split::smem_u32;
using split::tc_fence_after;
using split::tc_fence_before;
using split::umma_commit;
using split::umma_desc;
using split::umma_f16;
using split::umma_idesc_f16;

constexpr int kNA = 8;                                    // a values per part
constexpr int kN = 2 * kNA;                               // real columns per digit of the small operand
constexpr int kDigPlane = kRows * 2 * kUnitK * 2;         // one digit of one plane: 4 KB
constexpr int kPlane = kDig * kDigPlane;                  // 32 KB
constexpr int kVarBytes = 2 * kDig * (kN / 8) * 128;      // one variant's digits of a unit: 4 KB
constexpr int kExpBytes = 64;                             // exponents of the part's a values (int16), padded
constexpr int kSmallBytes = kExpBytes + 2 * kVarBytes;    // small block of a unit: exponents | A1 | NB
constexpr int kBufCols = kDig * kN;                       // accumulator buffer: 8 levels x kN columns
constexpr int kBufs = 512 / kBufCols;
constexpr int kStages = 2, kBSlots = 4, kExpRing = 32;
constexpr int kEpiWarps = 8;
constexpr int kConvWarps = 16;                            // 8 rows each
constexpr int kMmaWarp = kEpiWarps + kConvWarps, kProdWarp = kMmaWarp + 1;
constexpr int kThreads = (kProdWarp + 1) * 32;
constexpr int kMaxCtas = 160;
constexpr long long kSpinLimit = 1ll << 22;               // polls of the final waits
constexpr long long kWaitCycles = 1ll << 31;              // a work wait gives up after about a second
constexpr size_t kSlotDoubles = 2 * 2 * (size_t)kNA * kRows;  // partial sums of one (CTA, tile): [2][kNA][128] complex
// an epilogue still reading a group's exponents is at most kStages units and
// kBufs + 1 groups behind the converters
static_assert(kStages + kChunkUnits * (kBufs + 1) < kExpRing, "exponent ring");

// What the producer thread hands to the converters and the MMA thread with each
// slot of the small operand's ring: a unit, the end of a segment (a CTA's part
// of a tile: its sums go to `aux`), or the end of the range.
enum DescKind { kUnit = 0, kFlush = 1, kEnd = 2 };
enum DescFlags { kNear = 1, kFirst = 2, kLast = 4, kFresh = 8, kNewTile = 16 };
struct alignas(16) Desc {
  int kap;    // first history entry
  int c0;     // first column of the tile
  int flags;  // kind << 8 | DescFlags (first, last unit of its chunk; no chunk to follow; new tile)
  int aux;    // system of the launch, or the partial slot (flush)
};

enum PostType { kPostSum = 0, kPostFlush = 1, kPostExit = 2 };
struct alignas(16) Post {  // what the MMA thread hands to the epilogue with a buffer
  int type, grp, eidx; // sum group (0: I^<, 1: D), exponent ring index
  int slot;            // partial slot (flush)
  int16_t es[kNA];     // small operand's exponents
};

struct Smem {
  uint8_t stage[kStages][2 * kPlane];
  uint8_t small[kBSlots][kSmallBytes];
  int16_t erow[kExpRing][2][kRows];   // row exponents of a unit, per plane
  Post post[kBufs];
  Desc desc[kBSlots];
  uint64_t full[kStages], empty[kStages], bfull[kBSlots], bempty[kBSlots], accfull[kBufs], accempty[kBufs], mmadone;
  unsigned raise[kStages];            // 1 + the unit whose exponents start a new accumulation
  uint32_t tmem;
  int abort;
};

struct Args {
  Sys one;               // the system of a single-system launch
  const Sys* table;      // or the systems of the launch, in order (device memory)
  int n_sys, G;
  long long total;       // chunk slots of the launch
  double* part;
  int* status;
  long long spin;
};

// Waits for a phase of a barrier, suspended by the hardware between polls (most
// warps of this kernel wait most of the time: polling without suspension took
// a large part of the issue slots).  Gives up after `limit` clock cycles.
__device__ __forceinline__ bool mbar_try_suspend(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\nselp.u32 %0, 1, 0, p;\n}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity), "r"(20000u)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ bool wait_bar(Smem& sm, uint64_t* bar, uint32_t parity, int* status, long long limit) {
  if (mbar_try_suspend(bar, parity)) return true;
  const long long t0 = clock64();
  while (!mbar_try_suspend(bar, parity)) {
    const bool late = clock64() - t0 > limit;
    if (late || *(volatile int*)&sm.abort) {
      if (late) { atomicOr(status, kStatusTimeout); sm.abort = 1; }
      return false;
    }
  }
  return true;
}

// A role's position: chunk slot q of the launch and where it lies.
struct Cursor {
  long long q;
  Walk w;
};
__device__ __forceinline__ const Sys& sys_at(const Args& a, int i) { return a.table ? a.table[i] : a.one; }
__device__ __forceinline__ Cursor cursor_at(const Args& a, long long q) {
  Cursor c;
  int lo = 0, hi = a.n_sys;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (sys_at(a, mid).unit_base <= q) lo = mid; else hi = mid;
  }
  c.q = q;
  walk_to(c.w, sys_at(a, lo), lo, q - sys_at(a, lo).unit_base);
  return c;
}
// The next chunk slot (before `end`, or its place is not evaluated); true when
// it is in another tile or at the end.
__device__ __forceinline__ bool cursor_next(const Args& a, Cursor& c, long long end) {
  if (++c.q >= end) return true;
  const int moved = walk_next(c.w);
  if (moved == 2) walk_to(c.w, sys_at(a, c.w.si + 1), c.w.si + 1, 0);
  return moved != 0;
}

// ---------------------------------------------------------------- prep ---
// fp16 pair (digit of x, digit of y): byte `B` of two digit words, minus 1152
template <int B>
__device__ __forceinline__ uint32_t digit_pair(uint32_t x, uint32_t y) {
  const uint32_t w = (__byte_perm(x, y, B | ((B + 4) << 8)) & 0x00FF00FFu) | 0x64006400u;
  uint32_t r;
  asm("sub.rn.f16x2 %0, %1, %2;" : "=r"(r) : "r"(w), "r"(0x64806480u));
  return r;
}
// digit i of the words (x, y) as an fp16 pair
__device__ __forceinline__ uint32_t digit_of(int i, uint64_t x, uint64_t y) {
  const uint32_t xh = (uint32_t)(x >> 32), xl = (uint32_t)x, yh = (uint32_t)(y >> 32), yl = (uint32_t)y;
  switch (i) {
    case 0: return digit_pair<3>(xh, yh);
    case 1: return digit_pair<2>(xh, yh);
    case 2: return digit_pair<1>(xh, yh);
    case 3: return digit_pair<0>(xh, yh);
    case 4: return digit_pair<3>(xl, yl);
    case 5: return digit_pair<2>(xl, yl);
    case 6: return digit_pair<1>(xl, yl);
    default: return digit_pair<0>(xl, yl);
  }
}
__device__ __forceinline__ uint64_t bytes_of(double v, int E) {
  return digit_bytes((uint32_t)__double2hiint(v), (uint32_t)__double2loint(v), E);
}
__device__ __forceinline__ int field64(double v) { return field_of((uint32_t)__double2hiint(v)); }

// Small operands of chunk kc, part p (grid: chunk x part; warp = a, lane =
// entry of the chunk): A1 and NB with one exponent per a and chunk, in the real
// form of a complex product, columns (a, re): (P.re, -P.im), (a, im): (P.im, P.re)
// over the entry's (re, im).  Layout of a variant of a unit: [K group 2][digit
// 8][column group 2][8 columns][8 reals].
__global__ void __launch_bounds__(32 * kNA) fx_prep(Sys s, const double* __restrict__ Sl,
                                                    const double* __restrict__ Sg, WeightsView w,
                                                    uint8_t* __restrict__ small) {
  const int M = s.M, MM = M * M, n = s.n;
  const int kc = blockIdx.x, p = blockIdx.y, al = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int kap = kc * kChunkK + lane, a = p * kNA + al;
  const int m = div_m(kap, M, s.magic), x = kap - m * M;
  double v[2][2] = {{0.0, 0.0}, {0.0, 0.0}};
  if (m <= n && a < M) {
    const double2 l = reinterpret_cast<const double2*>(Sl)[(size_t)m * MM + a * M + x];
    const double2 g = reinterpret_cast<const double2*>(Sg)[(size_t)m * MM + a * M + x];
    const double wn = w.at(n, m), wb = -w.wbar[m];
    v[0][0] = wn * (g.x - l.x); v[0][1] = wn * (g.y - l.y);
    v[1][0] = wb * l.x; v[1][1] = wb * l.y;
  }
  int E = max(max(field64(v[0][0]), field64(v[0][1])), max(field64(v[1][0]), field64(v[1][1])));
  E = __reduce_max_sync(0xffffffffu, E);
  E = E == 0x7FF ? kNonFinite : max(E, 64);
  const int unit = kc * kChunkUnits + lane / kUnitK, kl = lane % kUnitK;
  uint8_t* blk = small + ((size_t)unit * s.parts + p) * kSmallBytes;
  if (kl == 0) reinterpret_cast<int16_t*>(blk)[al] = (int16_t)E;
  const int kg = kl >> 2, kin = 2 * (kl & 3);
  const int cre = 2 * al, cim = 2 * al + 1;
#pragma unroll
  for (int var = 0; var < 2; ++var) {
    const uint64_t br = bytes_of(v[var][0], E), bi = bytes_of(v[var][1], E);
#pragma unroll
    for (int d = 0; d < kDig; ++d) {
      const uint32_t ri = digit_of(d, br, bi);              // (re, im)
      const uint32_t re = ri & 0xFFFFu, im = ri >> 16;
      uint8_t* base = blk + kExpBytes + var * kVarBytes + (kg * kDig + d) * (kN / 8) * 128 + kin * 2;
      *reinterpret_cast<uint32_t*>(base + (cre >> 3) * 128 + (cre & 7) * 16) = re | ((im ^ 0x8000u) << 16);
      *reinterpret_cast<uint32_t*>(base + (cim >> 3) * 128 + (cim & 7) * 16) = im | (re << 16);
    }
  }
}

// ---------------------------------------------------------- converters ---
// A lane's place in a column tile: its row (c, b) of one plane, and where the
// row's entries lie: `tr` + m M^2 + x for m < c (block (c, m), transposed), and
// `dr` + m (m + 1) / 2 M^2 + x M for m >= c (block (m, c)).
struct Row {
  const double2* tr;
  const double2* dr;
  int c, n, edge;   // column, last history point (-1: no such row), c + shift
  int M;
  uint32_t magic;
};
__device__ __forceinline__ Row row_of(const Sys& s, int c0, int j, int plane) {
  Row r;
  const double2* base = reinterpret_cast<const double2*>(plane ? s.R : s.L);
  r.M = s.M;
  r.magic = s.magic;
  const int cl = div_m(j, r.M, r.magic), b = j - cl * r.M, MM = r.M * r.M;
  r.c = c0 + cl;
  const bool live = cl < s.CT && r.c <= s.n;
  r.n = live ? s.n : -1;
  r.edge = r.c + s.shift;
  r.tr = base + (live ? tri(r.c, 0) * MM + b * r.M : 0);
  r.dr = base + (live ? (int64_t)r.c * MM + b : 0);
  return r;
}
// Four consecutive entries from kap of a row; `mask` has bit i set where entry
// i counts, bit 4 + i where it lies above the diagonal (the entry is then -conj
// of the stored one).  kQuad (M a multiple of 4): the four share their history
// point m; masked entries load something valid instead of branching.
template <bool kQuad>
__device__ __forceinline__ void load_quad(const Row& r, int kap, bool near, double2 z[4], unsigned& mask) {
  const int M = r.M, MM = M * M;
  int m = div_m(kap, M, r.magic), x = kap - m * M;
  if (kQuad) {
    const bool in = m <= r.n && (near ? m > r.edge : m <= r.edge);
    const bool above = m < r.c;
    const double2* p = above ? r.tr + (m * MM + x) : r.dr + (tri(m, 0) * MM + x * M);
    int st = above ? 1 : M;
    if (!in) { p = r.tr; st = 1; }
#pragma unroll
    for (int i = 0; i < 4; ++i) z[i] = __ldg(p + i * st);
    mask = (in ? 15u : 0u) | (above ? 0xF0u : 0u);
    return;
  }
  mask = 0;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const bool in = m <= r.n && (near ? m > r.edge : m <= r.edge);
    const bool above = m < r.c;
    z[i] = make_double2(0.0, 0.0);
    if (in) z[i] = __ldg(above ? r.tr + (m * MM + x) : r.dr + (tri(m, 0) * MM + x * M));
    mask |= ((unsigned)in | ((unsigned)above << 4)) << i;
    if (++x == M) { x = 0; ++m; }
  }
}

// ---------------------------------------------------------------- main ---
template <bool kQuad>
__global__ void __launch_bounds__(kThreads, 1) fx_main(const __grid_constant__ Args a) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  Smem& sm = *reinterpret_cast<Smem*>(smem_raw);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const long long q0 = range_lo(a.total, a.G, blockIdx.x), q1 = range_lo(a.total, a.G, blockIdx.x + 1);

  if (tid == 0) {
    for (int i = 0; i < kStages; ++i) { mbar_init(&sm.full[i], kConvWarps); mbar_init(&sm.empty[i], 1); sm.raise[i] = 0; }
    for (int i = 0; i < kBSlots; ++i) { mbar_init(&sm.bfull[i], 1); mbar_init(&sm.bempty[i], 1); }
    // accfull: the MMA thread's arrival (post written) and its commit; accempty: one lane per epilogue warp
    for (int i = 0; i < kBufs; ++i) { mbar_init(&sm.accfull[i], 2); mbar_init(&sm.accempty[i], kEpiWarps); }
    mbar_init(&sm.mmadone, 1);
    sm.abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == kMmaWarp) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&sm.tmem)), "r"(512)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  fence_async_smem();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = sm.tmem;

  if (warp < kEpiWarps) {
    // --------------------------------------------------------- epilogue --
    // warp = 4 half + quadrant: 32 output rows (tensor-memory lanes), half of
    // the part's a values (kN / 2 columns)
    constexpr int kC = kN / 2;
    const int quad = warp & 3, half = warp >> 2;
    const int j = quad * 32 + lane;
    const uint32_t lane_addr = tmem + ((uint32_t)(quad * 32) << 16) + half * kC;
    double acc[2][kC];
#pragma unroll
    for (int i = 0; i < kC; ++i) acc[0][i] = acc[1][i] = 0.0;
    for (unsigned p = 0;; ++p) {
      const int buf = p % kBufs;
      if (!__all_sync(0xffffffffu, wait_bar(sm, &sm.accfull[buf], (p / kBufs) & 1, a.status, a.spin))) break;
      tc_fence_after();
      const Post& ps = sm.post[buf];
      const int type = ps.type;
      if (type == kPostExit) break;
      if (type == kPostFlush) {
        double2* out = reinterpret_cast<double2*>(a.part + (size_t)ps.slot * kSlotDoubles);
#pragma unroll
        for (int g = 0; g < 2; ++g)
#pragma unroll
          for (int i = 0; i < kC / 2; ++i) {
            out[(g * kNA + half * (kNA / 2) + i) * kRows + j] = make_double2(acc[g][2 * i], acc[g][2 * i + 1]);
            acc[g][2 * i] = acc[g][2 * i + 1] = 0.0;
          }
        __syncwarp();
        if (lane == 0) mbar_arrive(&sm.accempty[buf]);
        continue;
      }
      const int g = ps.grp;
      const int E = sm.erow[ps.eidx][g][j];
      int es[kC / 2];
#pragma unroll
      for (int i = 0; i < kC / 2; ++i) es[i] = ps.es[half * (kNA / 2) + i];
      auto fold = [&](double(&s)[kC]) {
#pragma unroll
        for (int c4 = 0; c4 < kC; c4 += 2) {
          uint32_t r[kDig][2];
#pragma unroll
          for (int d = 0; d < kDig; ++d)
            asm volatile("tcgen05.ld.sync.aligned.32x32b.x2.b32 {%0,%1}, [%2];"
                         : "=r"(r[d][0]), "=r"(r[d][1])
                         : "r"(lane_addr + buf * kBufCols + d * kN + c4));
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
          if (c4 + 2 == kC) {  // every level of this buffer is in registers
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&sm.accempty[buf]);
          }
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            int v[kDig];
#pragma unroll
            for (int d = 0; d < kDig; ++d) v[d] = __float2int_rn(__uint_as_float(r[d][i]));
            // the 64-bit integer sum_l S_l 256^(7-l) / 2^12: |S_0| <= 2^19, |S_1| <= 2^21, |S_2| <= 2^22 and
            // |S_l| <= l 2^21 fit the 32-bit steps, and 2^10 products of 62-bit values stay below 2^(124+7-56-12)
            const uint64_t p01 = (uint64_t)(int64_t)(v[0] * 256 + v[1]), p23 = (uint64_t)(int64_t)(v[2] * 256 + v[3]);
            const int low = v[5] * 16 + ((v[6] + (v[7] >> 8) + 8) >> 4);
            const int64_t t = (int64_t)((p01 << 36) + (p23 << 20) + ((uint64_t)(int64_t)v[4] << 12) + (uint64_t)(int64_t)low);
            // scale 2^(ev + eu - 68 + 12), ev = E - 1022, eu = es - 1022
            const int ex = E + es[(c4 + i) / 2] - 2 * 1022 - 56;
            if (ex >= -1022 && ex <= 1023) {
              s[c4 + i] = fma((double)t, __hiloint2double((ex + 1023) << 20, 0), s[c4 + i]);
            } else if (ex >= kNonFinite - 4096) {
              s[c4 + i] = __longlong_as_double(0x7FF8000000000000ll);
            } else {  // the scale alone leaves the range of FP64
              const int h = ex / 2;
              s[c4 + i] += (double)t * __hiloint2double((h + 1023) << 20, 0) * __hiloint2double((ex - h + 1023) << 20, 0);
            }
          }
        }
      };
      if (g == 0) fold(acc[0]); else fold(acc[1]);
    }
  } else if (warp < kMmaWarp) {
    // ------------------------------------------------------- converters --
    // lane = row (3 bits) | K half q << 3 | plane << 4: a quarter warp writes
    // 128 consecutive bytes of a digit plane
    const int wq = warp - kEpiWarps;
    const int q = (lane >> 3) & 1, plane = lane >> 4;
    const uint32_t dst0 = plane * kPlane + (q * 16 + wq) * 128 + (lane & 7) * 16;
    Row row;
    double2 z[4];
    unsigned mask = 0, d = 0;
    int flags = 0, E = 64, seen = 64;  // of the unit in z; the row's exponent; largest field of the current chunk
    // the next unit's loads; false when there is none
    auto load = [&]() -> bool {
      Desc ds;
      do {
        const int b = d % kBSlots;
        if (!__all_sync(0xffffffffu, wait_bar(sm, &sm.bfull[b], (d / kBSlots) & 1, a.status, a.spin))) return false;
        ds = sm.desc[b];
        ++d;
      } while (ds.flags >> 8 == kFlush);
      flags = ds.flags;
      if (flags >> 8 == kEnd) return false;
      if (flags & kNewTile) row = row_of(sys_at(a, ds.aux), ds.c0, 8 * wq + (lane & 7), plane);
      load_quad<kQuad>(row, ds.kap + 4 * q, flags & kNear, z, mask);
      return true;
    };
    bool more = load();
    for (unsigned u = 0; more; ++u) {
      const int s = u % kStages;
      // exponent of the row (far units: of both planes, which go into one sum)
      int mx = 0;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int h = max(__double2hiint(z[i].x) & 0x7FFFFFFF, __double2hiint(z[i].y) & 0x7FFFFFFF);
        mx = max(mx, h);  // masked entries are zero without kQuad
      }
      if (kQuad && !(mask & 1u)) mx = 0;
      mx >>= 20;
      mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, 8));
      const int other = __shfl_xor_sync(0xffffffffu, mx, 16);
      if (!(flags & kNear)) mx = max(mx, other);
      bool raised = false;
      if (flags & kFirst) {
        const int prev = (flags & kFresh) || seen == 0x7FF ? 0 : seen;
        E = max(max(mx, prev), 64) + kHeadroom;
        seen = mx;
      } else {
        raised = mx > E;
        if (raised) E = mx + kHeadroom;
        seen = max(seen, mx);
      }
      if (mx == 0x7FF) { raised |= E != kNonFinite; E = kNonFinite; }
      const int Ez = kQuad && !(mask & 1u) ? kNonFinite : E;  // a masked quad's digits are zero
      uint64_t br[4], bi[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const uint32_t fl = (mask << (27 - i)) & 0x80000000u;
        br[i] = digit_bytes((uint32_t)__double2hiint(z[i].x) ^ fl, (uint32_t)__double2loint(z[i].x), Ez);
        bi[i] = digit_bytes((uint32_t)__double2hiint(z[i].y), (uint32_t)__double2loint(z[i].y), Ez);
      }
      more = load();  // in flight while this unit's digits are written
      if (!__all_sync(0xffffffffu, wait_bar(sm, &sm.empty[s], ((u / kStages) & 1) ^ 1, a.status, a.spin))) break;
      if (__any_sync(0xffffffffu, raised) && lane == 0) *(volatile unsigned*)&sm.raise[s] = u + 1;
      if (q == 0) sm.erow[u % kExpRing][plane][8 * wq + (lane & 7)] = (int16_t)E;
      uint8_t* dst = sm.stage[s] + dst0;
#pragma unroll
      for (int i = 0; i < kDig; ++i)
        *reinterpret_cast<uint4*>(dst + i * kDigPlane) =
            make_uint4(digit_of(i, br[0], bi[0]), digit_of(i, br[1], bi[1]), digit_of(i, br[2], bi[2]),
                       digit_of(i, br[3], bi[3]));
      fence_async_smem();
      __syncwarp();
      if (lane == 0) mbar_arrive(&sm.full[s]);
    }
  } else if (warp == kProdWarp) {
    // --------------------------------------------------------- producer --
    if (lane == 0) {
      unsigned d = 0;
      // the next slot, its descriptor written; false when the wait ran out
      auto put = [&](int kap, int c0, int flags, int aux) -> bool {
        const int b = d % kBSlots;
        if (!wait_bar(sm, &sm.bempty[b], ((d / kBSlots) & 1) ^ 1, a.status, a.spin)) return false;
        sm.desc[b] = Desc{kap, c0, flags, aux};
        return true;
      };
      bool stop = false;
      Cursor c = cursor_at(a, q0);
      int fresh = kFresh | kNewTile, near = -1;
      while (c.q < q1 && !stop) {
        const Sys& S = sys_at(a, c.w.si);
        if (c.w.near != near) fresh |= kFresh;
        const uint32_t bytes = kExpBytes + (c.w.near ? 1 : 2) * kVarBytes;
        for (int unit = c.w.j0; unit < c.w.j1; ++unit) {
          const int flags = (c.w.near ? kNear : 0) | (unit == c.w.j0 ? kFirst : 0) | (unit + 1 == c.w.j1 ? kLast : 0);
          if (!put(c.w.kc * kChunkK + unit * kUnitK, c.w.c0, kUnit << 8 | flags | fresh, c.w.si)) { stop = true; break; }
          const int b = d % kBSlots;
          mbar_arrive_expect_tx(&sm.bfull[b], bytes);
          bulk_g2s(sm.small[b], S.small + ((size_t)(c.w.kc * kChunkUnits + unit) * c.w.parts + c.w.part) * kSmallBytes,
                   bytes, &sm.bfull[b]);
          ++d;
          fresh = 0;
          near = c.w.near;
        }
        if (stop) break;
        const long long tile = S.tile_base + c.w.T;
        if (cursor_next(a, c, q1)) {
          if (!put(0, 0, kFlush << 8, (int)partial_slot(tile, blockIdx.x))) { stop = true; break; }
          mbar_arrive(&sm.bfull[d++ % kBSlots]);
          fresh = kFresh | kNewTile;
        }
      }
      if (!stop && put(0, 0, kEnd << 8, 0)) mbar_arrive(&sm.bfull[d++ % kBSlots]);
      // the copies already issued must land before the CTA can exit (each slot's last phase)
      for (unsigned k = d > kBSlots ? d - kBSlots : 0; k < d; ++k) {
        long long spins = 0;
        while (!mbar_try(&sm.bfull[k % kBSlots], (k / kBSlots) & 1) && ++spins < kSpinLimit) __nanosleep(64);
        if (spins >= kSpinLimit) atomicOr(a.status, kStatusTimeout);
      }
    }
    __syncwarp();
  } else {
    // -------------------------------------------------------------- MMA --
    if (lane == 0) {
      // A: [digit 8][K group 2][row group 16][8 rows][16 B]; B: [K group 2][digit 8][column group 2][8][16 B]
      const uint64_t a0 = umma_desc(smem_u32(sm.stage[0]), kRows * 16, 128);
      const uint64_t b0 = umma_desc(smem_u32(sm.small[0] + kExpBytes), kDig * (kN / 8) * 128, 128);
      unsigned u = 0, p = 0;
      bool any = false, stop = false, open = false;
      int nb = 0;     // buffers of the open group
      int held = -1;  // slot of a flush descriptor not released yet (every tile has units: one at most)
      auto close = [&]() {
        for (int k = 0; k < nb; ++k) {
          mbar_arrive(&sm.accfull[(p + k) % kBufs]);
          umma_commit(&sm.accfull[(p + k) % kBufs]);
        }
        p += nb;
        open = false;
      };
      // hands a message without sums to the epilogue
      auto message = [&](int type, int slot) -> bool {
        const int buf = p % kBufs;
        if (!wait_bar(sm, &sm.accempty[buf], ((p / kBufs) & 1) ^ 1, a.status, a.spin)) return false;
        sm.post[buf].type = type;
        sm.post[buf].slot = slot;
        mbar_arrive(&sm.accfull[buf]);
        mbar_arrive(&sm.accfull[buf]);
        ++p;
        return true;
      };
      for (unsigned d = 0; !stop; ++d) {
        const int b = d % kBSlots;
        if (!wait_bar(sm, &sm.bfull[b], (d / kBSlots) & 1, a.status, a.spin)) { stop = true; break; }
        const Desc ds = sm.desc[b];
        const int kind = ds.flags >> 8;
        if (kind == kEnd) break;
        if (kind == kFlush) {
          held = b;  // until the next unit is full: then every converter has read past this descriptor
          if (!message(kPostFlush, ds.aux)) stop = true;
          continue;
        }
        const int s = u % kStages;
        const bool near = ds.flags & kNear;
        if (!wait_bar(sm, &sm.full[s], (u / kStages) & 1, a.status, a.spin)) { stop = true; break; }
        if (held >= 0) {
          mbar_arrive(&sm.bempty[held]);
          held = -1;
        }
        const bool begin = (ds.flags & kFirst) || *(volatile unsigned*)&sm.raise[s] == u + 1;
        if (begin) {
          if (open) close();
          nb = near ? 2 : 1;
          const int4 ex = *reinterpret_cast<const int4*>(sm.small[b]);
          for (int g = 0; g < nb && !stop; ++g) {
            const int buf = (p + g) % kBufs;
            if (!wait_bar(sm, &sm.accempty[buf], (((p + g) / kBufs) & 1) ^ 1, a.status, a.spin)) { stop = true; break; }
            Post& ps = sm.post[buf];
            ps.type = kPostSum;
            ps.grp = g;
            ps.eidx = u % kExpRing;
            *reinterpret_cast<int4*>(ps.es) = ex;
          }
          if (stop) break;
          open = true;
        }
        tc_fence_after();
        const uint64_t dPL = a0 + ((uint64_t)(s * 2 * kPlane) >> 4), dQ = dPL + (kPlane >> 4);
        const uint64_t dA = b0 + ((uint64_t)(b * kSmallBytes) >> 4), dB = near ? dA : dA + (kVarBytes >> 4);
        const uint32_t t0 = tmem + (p % kBufs) * kBufCols, t1 = near ? tmem + ((p + 1) % kBufs) * kBufCols : t0;
#pragma unroll
        for (int i = 0; i < kDig; ++i)
          umma_f16(t0 + i * kN, dPL + ((i * kDigPlane) >> 4), dA, umma_idesc_f16(kN * (kDig - i)), !(begin && i == 0));
#pragma unroll
        for (int i = 0; i < kDig; ++i)
          umma_f16(t1 + i * kN, dQ + ((i * kDigPlane) >> 4), dB, umma_idesc_f16(kN * (kDig - i)),
                   !(begin && near && i == 0));
        umma_commit(&sm.empty[s]);
        umma_commit(&sm.bempty[b]);
        any = true;
        ++u;
        if (ds.flags & kLast) close();
      }
      if (!stop) message(kPostExit, 0);
      // every MMA must complete before tensor memory is freed
      if (any) {
        umma_commit(&sm.mmadone);
        long long spins = 0;
        while (!mbar_try(&sm.mmadone, 0) && ++spins < kSpinLimit) __nanosleep(64);
        if (spins >= kSpinLimit) atomicOr(a.status, kStatusTimeout);
      }
    }
    __syncwarp();
  }
  tc_fence_before();
  __syncthreads();
  if (warp == kMmaWarp) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
  }
}

// -------------------------------------------------------------- reduce ---
// Output entry lin = (c, a, b): the partial sums of its tile in CTA order, then
// the band of term 2 in FP64 with its exact weights.
__global__ void __launch_bounds__(256) fx_reduce(Sys s, long long total, int G, const double* __restrict__ part,
                                                 const double* __restrict__ Sl, const double* __restrict__ Sg,
                                                 WeightsView w, double* __restrict__ out, int* status) {
  const int M = s.M, MM = M * M, n = s.n;
  const int64_t lin = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t row = (int64_t)(n + 1) * MM;
  if (lin >= row) return;
  const int c = (int)(lin / MM), ab = (int)(lin - (int64_t)c * MM), a = ab / M, b = ab - a * M;
  const int ct = c / s.CT, T = ct * s.parts + a / kNA;
  const int64_t at = (int64_t)(a % kNA) * kRows + (c - ct * s.CT) * M + b;
  const long long lo = s.unit_base + (long long)T * s.upt, hi = lo + s.upt;
  int i = (int)(lo * G / total);
  while (i > 0 && range_lo(total, G, i) > lo) --i;
  while (range_lo(total, G, i + 1) <= lo) ++i;
  rk::Cd p{0, 0}, d{0, 0}, tl{0, 0}, tg{0, 0};
  for (; i < G && range_lo(total, G, i) < hi; ++i) {
    const double2* q = reinterpret_cast<const double2*>(part + (size_t)partial_slot(s.tile_base + T, i) * kSlotDoubles);
    const double2 x = q[at], y = q[at + kNA * kRows];
    p.re += x.x; p.im += x.y;
    d.re += y.x; d.im += y.y;
  }
  for (int m = max(0, c - w.band_w + 1); m <= c; ++m) {
    const double wcm = w.at(c, m);
    const double* r = s.R + (tri(c, m) * MM + b * M) * 2;
    const double* sl = Sl + ((int64_t)m * MM + a * M) * 2;
    const double* sg = Sg + ((int64_t)m * MM + a * M) * 2;
#pragma unroll 4
    for (int x = 0; x < M; ++x) {
      const rk::Cd rr = rk::ld(r + 2 * x);
      rk::Cd vl = rk::ld(sl + 2 * x), vg = rk::ld(sg + 2 * x);
      vl.re *= wcm; vl.im *= wcm; vg.re *= wcm; vg.im *= wcm;
      rk::mac_cj(tl, vl, rr);
      rk::mac_cj(tg, vg, rr);
    }
  }
  const double2 x = make_double2(p.re + tl.re, p.im + tl.im);
  const double2 y = make_double2(p.re + d.re + tg.re, p.im + d.im + tg.im);
  reinterpret_cast<double2*>(out)[lin] = x;
  reinterpret_cast<double2*>(out)[row + lin] = y;
  if (!(isfinite(x.x) && isfinite(x.y) && isfinite(y.x) && isfinite(y.y))) atomicOr(status, kStatusNumeric);
}

bool make_sys(int M, int n, int band_w, Sys* s) {
  if (M < 1 || M > kMaxNorb || n < 0) return false;
  s->M = M;
  s->n = n;
  s->CT = kRows / M;
  s->cpt = (int)(((long long)(n + 1) * M + kChunkK - 1) / kChunkK);
  s->parts = (M + kNA - 1) / kNA;
  s->tiles = (n + s->CT) / s->CT * s->parts;
  s->upt = s->cpt + kOver;
  s->shift = -band_w;
  s->magic = M == 1 ? 0u : (uint32_t)((0x100000000ull + (unsigned long long)M - 1) / (unsigned long long)M);
  s->unit_base = s->tile_base = 0;
  return true;
}

size_t small_bytes(const Sys& s) { return ((size_t)s.cpt * kChunkUnits * s.parts * kSmallBytes + 255) / 256 * 256; }

int grid_ctas(long long total) { return (int)std::min<long long>(total, std::min(sm_count(), kMaxCtas)); }

}  // namespace

size_t fx_workspace_bytes(int M, int n_max) {
  Sys s;
  if (!make_sys(M, n_max - 1, 1, &s)) return 0;
  return small_bytes(s) + ((size_t)s.tiles + std::min(sm_count(), kMaxCtas)) * kSlotDoubles * sizeof(double);
}

// The kernel's dynamic shared memory exceeds the default limit (set once per device).
cudaError_t fx_prepare() {
  static std::atomic<unsigned long long> done_mask{0};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const unsigned long long bit = 1ull << (dev & 63);
  if (done_mask.load() & bit) return cudaSuccess;
  e = cudaFuncSetAttribute(fx_main<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(Smem));
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(fx_main<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(Smem));
  if (e == cudaSuccess) done_mask.fetch_or(bit);
  return e;
}

cudaError_t launch_history_fx(const HistoryArgs& h, void* work, size_t work_bytes, cudaStream_t st, int* launches) {
  *launches = 0;
  Sys s;
  if (!make_sys(h.M, h.n, h.w.band_w, &s)) return cudaErrorInvalidValue;
  s.L = h.L;
  s.R = h.R;
  uint8_t* small = reinterpret_cast<uint8_t*>(work);
  double* part = reinterpret_cast<double*>(small + small_bytes(s));
  s.small = small;
  const long long total = (long long)s.tiles * s.upt;
  const int G = grid_ctas(total);
  if (small_bytes(s) + ((size_t)s.tiles + G) * kSlotDoubles * sizeof(double) > work_bytes) return cudaErrorInvalidValue;
  cudaError_t e = fx_prepare();
  if (e != cudaSuccess) return e;
  fx_prep<<<dim3(s.cpt, s.parts), 32 * kNA, 0, st>>>(s, h.Sl, h.Sg, h.w, small);
  ++*launches;
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  Args a{};
  a.one = s;
  a.n_sys = 1;
  a.G = G;
  a.total = total;
  a.part = part;
  a.status = h.status;
  a.spin = kWaitCycles;
  if (h.ev_begin) cudaEventRecord(h.ev_begin, st);
  if (s.M % 4 == 0)
    fx_main<true><<<G, kThreads, sizeof(Smem), st>>>(a);
  else
    fx_main<false><<<G, kThreads, sizeof(Smem), st>>>(a);
  if (h.ev_end) cudaEventRecord(h.ev_end, st);
  ++*launches;
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  const int64_t row = (int64_t)(s.n + 1) * s.M * s.M;
  fx_reduce<<<(unsigned)((row + 255) / 256), 256, 0, st>>>(s, total, G, part, h.Sl, h.Sg, h.w, h.out, h.status);
  ++*launches;
  return cudaGetLastError();
}

}  // namespace kbe
