// history_fx.cu -- FP64 history slice of Eq. (KBE2) (Sec. 2) on the 16-bit-float
// tensor cores (tcgen05), by error-free slicing into eight digits per value
// (fx_common.cuh).
//
// The sums are those of history_f64.cu.  With the planes PL(m,c) = L(m,c),
// Q(m,c) = R(m,c) for m >= c and PL = -L(c,m)^+, Q = -R(c,m)^+ for m < c
// (G^< = PL, G^> = PL + Q), A1[m] = w_{n,m} (S^> - S^<)[m], NB[m] = -wbar_m S^<[m]:
//   far  (m <= c - band_w): I^< += A1 PL + NB Q          (both components alike)
//   near (m >  c - band_w): I^< += A1 PL,  D += A1 Q      (I^> = I^< + D)
//   band (c - band_w < m <= c): I^< += S^< w_{c,m} R(c,m)^+,  D += (S^> - S^<) w_{c,m} R(c,m)^+
// -- two real products of 128-row tiles per history point.
//
// The adjoint of the slice (adjoint.cu) has the same form with the roles of c
// and m exchanged.  With J = Ibar^< + Ibar^> and the planes' adjoints in place of
// the planes (signs and the diagonal as noted at load_quad and fx_prep):
//   A1bar[m] = sum_{c < m + band_w} (J PL^+ + Ibar^> Q^+) - sum_{c >= m + band_w} J L(c,m),
//   C[m]     = sum_{c >= m} w_{c,m} J R(c,m),
//   S^>bar[m] = w_{n,m} A1bar[m] + sum_{band} w_{c,m} Ibar^> R(c,m),   S^<bar[m] = C[m] - S^>bar[m]
// (the settled columns as in adj_hist_small): the same far, near and band parts,
// with the sums of the first two scaled by w_{n,m} and wbar_m before the band.
//
// Why: FP64 runs at 1.26 TFLOP/s on this part (152 SMs x 2 FMA), the fp16
// tensor cores at about 1900, so 36 digit products cost a fiftieth of the FP64
// ones.  What bounds it then is the conversion: every history entry is read in
// both orientations and cut into digits with about 30 integer instructions per
// real, and the digit stores (64 KB a unit), the MMA operand reads and the history
// loads share the L1 / shared-memory data pipe (M = 8, n = 1023: issue slots 70%,
// LSU wavefronts 44%, tensor pipe 17%, DRAM 33%).  With NA = 16 the epilogue holds the MMAs back as well.
// Measured, in this kernel: the slice n = 1023, M = 8 in 0.82 ms (7.05 on the FP64
// pipe, history_f64.cu), n = 511, M = 16 in 1.19 ms (14.4).
//
// One persistent CTA per SM takes a contiguous range of chunks (32 history
// entries of a 128-row column tile).  A unit is 8 entries, one MMA K step:
//  * 16 converter warps, each owning 8 rows: a lane holds 4 entries of one row
//    of one plane, loaded one unit ahead straight into registers (staging them
//    in shared memory would cost as much of its bandwidth as the digits), finds
//    the row's exponent with its neighbours and writes the digit planes
//    (2 x 32 KB per unit) into a ring of two stages;
//  * one thread copies the small operand's digits of each unit (bulk copies);
//  * two threads issue the MMAs, one per product of the unit: digit i of the
//    history against the stacked digits 0..7-i of the small operand, so the
//    products of level i + j land in the columns of that level (N = 2 NA (8 - i)
//    for a part of NA rows a);
//  * eight epilogue warps fold the eight integer levels of up to two chunks into
//    one 64-bit integer, and that, scaled, into FP64 sums in registers: two FP64
//    operations per 64 entries of an output.
// Parts of NA = 8 rows a for M <= 8, else 16: a part's conversion of the history
// serves all its rows (two sums of 16 x 8 levels fill tensor memory, so with NA =
// 16 an accumulation waits for the epilogue of the one before).
// One MMA thread instead of two: 0.88 and 1.31 ms for the two slices above.  History
// loads of far quads as 4 x 16 instead of 2 x 32 bytes pass twice through the data pipe.
// A row's exponent holds for the units accumulated together in tensor memory, and
// counts its entries as the small operand scales them (Exps in fx_common.cuh).
// It starts kHeadroom bits above the larger of the unit's and the previous
// chunk's largest entry; a unit that exceeds it nevertheless closes the
// accumulation and starts the next with the larger exponent.  A row that had
// only zeros so far (near the diagonal each column of the tile starts at a point
// of its own) takes its exponent without that, so the sums use the exponents of
// an accumulation's last unit, and starts kStartRoom bits above its first values, which
// may be its smallest.  With an accumulation for each start, which had most near
// the diagonal, and its band entries loaded one by one (for_band), the slice
// M = 8, n = 124 took 85 us instead of 66, M = 5, n = 333 106 instead of 94.
//
// Partial sums go to one slot per (CTA, tile) and are added in CTA order, so
// results are bitwise reproducible.  All waits are bounded.  A row or a small
// operand that holds a non-finite value gives NaN in the outputs it enters, as
// on the FP64 path, and the reduction reports it.

#include <algorithm>
#include <atomic>

#include "history_fx.h"
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

constexpr int kDigPlane = kRows * 2 * kUnitK * 2;         // one digit of one plane: 4 KB
constexpr int kPlane = kDig * kDigPlane;                  // 32 KB
constexpr int kExpBytes = sizeof(Exps);                   // exponents of a part's small operand
constexpr int kStages = 2, kBSlots = 4, kExpRing = 32;
constexpr int kEpiWarps = 8;
constexpr int kConvWarps = 16;                            // 8 rows each
constexpr int kMmaWarp = kEpiWarps + kConvWarps, kProdWarp = kMmaWarp + 1, kMmaWarp2 = kMmaWarp + 2;
constexpr int kThreads = (kProdWarp + 3) * 32;            // whole warpgroups (setmaxnreg): 896
constexpr long long kSpinLimit = 1ll << 22;               // polls of the final waits
constexpr long long kWaitCycles = 1ll << 31;              // a work wait gives up after about a second
template <int NA>
struct Cfg {
  static constexpr int kN = 2 * NA;                              // real columns per digit of the small operand
  static constexpr int kVarBytes = 2 * kDig * (kN / 8) * 128;    // one variant's digits of a unit
  static constexpr int kHalfBytes = kExpBytes + 2 * kVarBytes;   // exponents | variant 0 | variant 1
  static constexpr int kSmallBytes = 2 * kHalfBytes;             // small block of a unit: main half, band half
  static constexpr int kBufCols = kDig * kN;                     // accumulator buffer: 8 levels x kN columns
  static constexpr int kBufs = 512 / kBufCols;
  static constexpr size_t kSlot = slot_complex(NA);              // partial sums of one (CTA, tile): [2][NA][128] complex
  static_assert(kSmallBytes == small_block_bytes(NA) && kHalfBytes % 128 == 0 && kExpBytes % 128 == 0, "small operand layout");
  // an epilogue still reading an accumulation's exponents is at most kStages units
  // and the open and the buffered ones (8 units per two buffers) behind the converters
  static_assert(kStages + kChunkUnits * (kBufs + 2) < kExpRing, "exponent ring");
};

// What the producer thread hands to the converters and the MMA thread with each
// slot of the small operand's ring: a unit, the scaling of an adjoint's sums
// before the band, the end of a segment (a CTA's part of a tile: its sums go to
// partial slot `aux`), or the end of the range.
enum DescKind { kUnit = 0, kScale = 1, kFlush = 2, kEnd = 3 };
enum DescFlags { kFlagNear = 1, kFlagBand = 2, kFirst = 4, kLast = 8, kFresh = 16, kNewTile = 32, kFlagLow = 64 };
struct alignas(16) Desc {
  int kap;    // first history entry
  int c0;     // first column of the tile
  int flags;  // a values of the part << 16 | kind << 8 | DescFlags (first, last unit of its chunk; no chunk to follow; new tile; far points
              // may lie below the diagonal)
  int aux;    // system of the launch; partial slot (flush)
};

__device__ __forceinline__ int kind_of(int flags) { return flags >> 8 & 0xFF; }

struct alignas(16) Post {  // what the MMA thread hands to the epilogue with a buffer
  int type;                // kUnit (sums), kScale, kFlush, kEnd
  int grp, eidx, plane;    // sum group (0: I^<, 1: D), exponent ring index (the last unit's) and plane
  int si, c0, slot;        // system; first column (scale); partial slot (flush)
  int cols;                // a values of the part, plus one
  int16_t es[16];          // small operand's exponents
};

// Registers of the epilogue, converter and other warpgroups (setmaxnreg), whose sum is
// the launch's 896 x 72: an epilogue thread holds 2 NA FP64 sums, a converter 16 words of
// loads, as many of digits and the entries' exponents.  (With 56 for the converters of
// NA = 16 the slice M = 16, n = 511 takes 1.36 ms instead of 1.24, with 104, 64 and 40 the
// slice M = 8, n = 1023 865 us instead of 836.)
template <int NA, bool kQuad>
struct Regs {
  static constexpr int kEpi = NA == 8 && kQuad ? 88 : 104, kConv = NA == 8 && kQuad ? 72 : 64, kMisc = 40;
  static_assert(256 * kEpi + 512 * kConv + 128 * kMisc == kThreads * 72, "register split");
};


template <int NA>
struct Smem {
  uint8_t stage[kStages][2 * kPlane];
  uint8_t small[kBSlots][Cfg<NA>::kHalfBytes];
  int16_t erow[kExpRing][2][kRows];   // row exponents of a unit, per plane
  Post post[Cfg<NA>::kBufs];
  Desc desc[kBSlots];
  uint64_t full[kStages], empty[kStages], bfull[kBSlots], bempty[kBSlots];
  uint64_t accfull[Cfg<NA>::kBufs], accempty[Cfg<NA>::kBufs], mmadone[2];
  unsigned raise[kStages];            // 1 + the unit whose exponents start a new accumulation
  uint32_t tmem;
  int abort;
};

// The systems of a launch: one, by value, or a table and its head in device memory.
struct Args {
  Sys one;
  Head one_head;
  const Sys* table;
  const Head* head;
  int G;
  int withhold;           // failure-path test: the unit of each CTA that its producer does not supply
  long long wait_cycles;  // and the length of its waits (0: no test)
};
__device__ __forceinline__ const Sys& sys_at(const Args& a, int i) { return a.table ? a.table[i] : a.one; }
__device__ __forceinline__ const Head& head_of(const Args& a) { return a.table ? *a.head : a.one_head; }
// last system whose base (one of the Sys members) is at most x
template <class F>
__device__ __forceinline__ int find_sys(const Args& a, long long x, F base) {
  int lo = 0, hi = head_of(a).n_sys;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (base(sys_at(a, mid)) <= x) lo = mid; else hi = mid;
  }
  return lo;
}
__device__ __forceinline__ WeightsView weights_of(const Sys& s) { return WeightsView{s.wbar, s.band, s.band_w}; }

// Lets the next kernel (launch_overlapped) start its setup.
__device__ __forceinline__ void grid_launch_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Waits for a phase of a barrier, suspended by the hardware between polls.
// Gives up after kWaitCycles (kTest: the launch's own), or when another role has.
__device__ __forceinline__ bool try_suspend(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\nselp.u32 %0, 1, 0, p;\n}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity), "r"(20000u)
      : "memory");
  return ok != 0;
}
template <bool kTest>
__device__ __forceinline__ bool wait_bar(const Args& a, int* abort, uint64_t* bar, uint32_t parity, int* status) {
  if (try_suspend(bar, parity)) return true;
  const long long t0 = clock64();
  while (!try_suspend(bar, parity)) {
    const bool late = clock64() - t0 > (kTest ? a.wait_cycles : kWaitCycles);
    if (late || *(volatile int*)abort) {
      if (late) { atomicOr(status, kStatusTimeout); *(volatile int*)abort = 1; }
      return false;
    }
  }
  return true;
}

// ---------------------------------------------------------------- prep ---
// fp16 pair (digit of x, digit of y): byte `B` of two digit words, each put into
// the low mantissa bits of 1024, minus 1152
template <int B>
__device__ __forceinline__ uint32_t digit_pair(uint32_t x, uint32_t y) {
  // bytes (x, y) of B and B ^ 1 side by side: shared by the two digits
  const uint32_t xy = __byte_perm(x, y, (B & 2) | ((B & 2) + 4) << 4 | ((B & 2) + 1) << 8 | ((B & 2) + 5) << 12);
  const uint32_t w = __byte_perm(xy, 0x64646464u, (B & 1) ? 0x4342 : 0x4140);
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

// Small operands of a pair of chunks and a part (grid-stride over them; warp = a,
// a lane has one entry of each chunk): an exponent per entry k, unit half and
// variant (Exps), and with those taken off one exponent per a, pair, half and
// variant (near sums accumulate over the pair), in the real form
// of a complex product: columns (a, re): (P.re, -P.im), (a, im): (P.im, P.re) over
// the entry's (re, im).  Layout of a variant of a unit: [K group 2][digit 8]
// [column group][8 columns][8 reals].  With (l, g) = (S^<, S^>), resp. (Ibar^<, Ibar^>):
//   slice    main w_{n,m} (g - l), -wbar_m l    band l, g - l
//   adjoint  main -(l + g), -g                  band g, l + g
template <int NA>
__global__ void __launch_bounds__(32 * NA) fx_prep(const __grid_constant__ Args a) {
  using C = Cfg<NA>;
  __shared__ int s_ek[2][2][2][kChunkK];  // [half][variant][chunk][entry]: largest field over the rows a
  grid_launch_next();
  grid_wait();
  const int al = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const long long chunks = head_of(a).chunks;
  for (long long ch = blockIdx.x; ch < chunks; ch += gridDim.x) {
    const Sys& s = sys_at(a, find_sys(a, ch, [](const Sys& y) { return y.chunk_base; }));
    const int M = s.M, MM = M * M, n = s.n, parts = s.parts;
    const int pair = (int)((ch - s.chunk_base) / parts), p = (int)(ch - s.chunk_base - (long long)pair * parts);
    const int row = p * NA + al;
    __syncthreads();
    for (int i = threadIdx.x; i < 8 * kChunkK; i += 32 * NA) (&s_ek[0][0][0][0])[i] = 0;
    double2 l[2], g[2];
    double w0[2] = {1.0, 1.0}, w1[2] = {1.0, 1.0};
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const int kap = (2 * pair + k) * kChunkK + lane;
      const int m = div_m(kap, M, s.magic), x = kap - m * M;
      l[k] = g[k] = make_double2(0.0, 0.0);
      if (m <= n && row < M) {
        l[k] = reinterpret_cast<const double2*>(s.Sl)[(size_t)m * MM + row * M + x];
        g[k] = reinterpret_cast<const double2*>(s.Sg)[(size_t)m * MM + row * M + x];
        if (!s.adj) {
          w0[k] = weights_of(s).at(n, m);
          w1[k] = s.wbar[m];
        }
      }
    }
    double2 v[2][2][2];  // [half][variant][chunk]; FP64 arithmetic bounds this kernel, so once
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      if (s.adj) {
        const double2 t = make_double2(l[k].x + g[k].x, l[k].y + g[k].y);
        v[0][0][k] = make_double2(-t.x, -t.y);
        v[0][1][k] = make_double2(-g[k].x, -g[k].y);
        v[1][0][k] = g[k];
        v[1][1][k] = t;
      } else {
        const double2 d = make_double2(g[k].x - l[k].x, g[k].y - l[k].y);
        v[0][0][k] = make_double2(w0[k] * d.x, w0[k] * d.y);
        v[0][1][k] = make_double2(-w1[k] * l[k].x, -w1[k] * l[k].y);
        v[1][0][k] = l[k];
        v[1][1][k] = d;
      }
    }
    __syncthreads();
#pragma unroll
    for (int half = 0; half < 2; ++half)
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        int f[2];
#pragma unroll
        for (int var = 0; var < 2; ++var) {
          f[var] = max(field64(v[half][var][k].x), field64(v[half][var][k].y));
          if (f[var] == 0x7FF) f[var] = 0;
        }
        if (half) f[0] = f[1] = max(f[0], f[1]);
        if (f[0]) atomicMax(&s_ek[half][0][k][lane], f[0]);
        if (f[1]) atomicMax(&s_ek[half][1][k][lane], f[1]);
      }
    __syncthreads();
    const int kl = lane % kUnitK, kg = kl >> 2, kin = 2 * (kl & 3), cre = 2 * al, cim = 2 * al + 1;
#pragma unroll
    for (int half = 0; half < 2; ++half)
#pragma unroll
      for (int var = 0; var < 2; ++var) {
        int ek[2], E = -kNonFinite;
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          ek[k] = s_ek[half][var][k][lane];
          const int f = max(field64(v[half][var][k].x), field64(v[half][var][k].y));
          if (f) E = max(E, f == 0x7FF ? kNonFinite : f - ek[k]);
        }
        E = __reduce_max_sync(0xffffffffu, E);
        if (E == -kNonFinite) E = 0;  // zeros
        const int least = __reduce_max_sync(0xffffffffu, max(ek[0], ek[1])) + 64;
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          if (2 * pair + k >= s.cpt) break;
          const int unit = (2 * pair + k) * kChunkUnits + lane / kUnitK;
          uint8_t* out = s.small + ((size_t)unit * parts + p) * C::kSmallBytes + half * C::kHalfBytes;
          Exps& x = *reinterpret_cast<Exps*>(out);
          if (kl == 0) x.es[var][al] = (int16_t)E;
          const int ek1 = __shfl_down_sync(0xffffffffu, ek[k], 1);
          if (al == 0 && !(kl & 1))
            x.ek[var][kl >> 1] = (uint32_t)ek[k] | (uint32_t)(kl & 2 ? least >> 8 : least & 0xFF) << 12 | (uint32_t)ek1 << 20;
          // zeros (and subnormals) whatever the exponents
          const double2 z = v[half][var][k];
          const uint64_t br = bytes_of(z.x, field64(z.x) ? E + ek[k] : kNonFinite),
                         bi = bytes_of(z.y, field64(z.y) ? E + ek[k] : kNonFinite);
#pragma unroll
          for (int d = 0; d < kDig; ++d) {
            const uint32_t ri = digit_of(d, br, bi);              // (re, im)
            const uint32_t re = ri & 0xFFFFu, im = ri >> 16;
            uint8_t* base = out + kExpBytes + var * C::kVarBytes + (kg * kDig + d) * (C::kN / 8) * 128 + kin * 2;
            *reinterpret_cast<uint32_t*>(base + (cre >> 3) * 128 + (cre & 7) * 16) = re | ((im ^ 0x8000u) << 16);
            *reinterpret_cast<uint32_t*>(base + (cim >> 3) * 128 + (cim & 7) * 16) = im | (re << 16);
          }
        }
      }
  }
}

// ---------------------------------------------------------- converters ---
// A lane's place in a column tile: its row (c, b) of one plane, and where the
// row's entries lie: `tr` + m M^2 + x above the diagonal (m < diag: block (c, m),
// transposed), and `dr` + m (m + 1) / 2 M^2 + x M below it (block (m, c)).
struct Row {
  const double2* tr;
  const double2* dr;
  int n, edge;      // last point (-1: no such row), c + shift
  int diag;         // first point that is read directly: c, in the adjoint c + 1
  int M, wide;      // wide: the plane starts on a 32-byte boundary
  uint32_t magic;
};
__device__ __forceinline__ Row row_of(const Sys& s, int c0, int j, int plane) {
  Row r;
  const double2* base = reinterpret_cast<const double2*>(plane ? s.R : s.L);
  r.M = s.M;
  r.wide = (reinterpret_cast<uintptr_t>(base) & 31u) == 0;
  r.magic = s.magic;
  const int cl = div_m(j, r.M, r.magic), b = j - cl * r.M, MM = r.M * r.M;
  const int c = c0 + cl;
  const bool live = cl < s.CT && c <= s.n;
  r.n = live ? s.n : -1;
  r.edge = c + s.shift;
  r.diag = c + s.adj;
  r.tr = base + (live ? tri(c, 0) * MM + b * r.M : 0);
  r.dr = base + (live ? (int64_t)c * MM + b : 0);
  return r;
}
// m (m + 1) / 2 as one 32 x 32 -> 64 bit product
__device__ __forceinline__ uint64_t tri0(int m) {
  const uint32_t h = (uint32_t)m >> 1, odd = (uint32_t)m & 1u;
  return (uint64_t)(odd ? (uint32_t)m : h) * (odd ? h + 1 : (uint32_t)m + 1);
}
// Four consecutive entries from kap of a row; `mask` has bit i set where entry
// i counts, bit 4 + i where it lies above the diagonal (the entry of the plane is
// then -conj of the stored one).  kQuad (M a multiple of 4): the four share their
// point m; masked entries load something valid instead of branching.  A slice's
// far points (far_tr) all lie above the diagonal.
// Two entries (32 bytes, 32-byte aligned) in one load: a far quad's 64 bytes lie
// in a row of their own, and 16-byte loads of them took as many passes through
// the L1 data pipe, which the digit stores and the MMA operands share, as both.
__device__ __forceinline__ void ldg_pair(const double2* p, double2& x, double2& y) {
  asm("ld.global.nc.v4.f64 {%0,%1,%2,%3}, [%4];" : "=d"(x.x), "=d"(x.y), "=d"(y.x), "=d"(y.y) : "l"(p));
}
template <bool kQuad>
__device__ __forceinline__ void load_quad(const Row& r, int kap, bool near, bool far_tr, double2 z[4], unsigned& mask) {
  const int M = r.M, MM = M * M;
  int m = div_m(kap, M, r.magic), x = kap - m * M;
  if (kQuad) {
    if (far_tr) {
      const bool in = m <= r.edge && r.n >= 0;
      const double2* p = r.tr + (in ? (unsigned)(m * MM + x) : 0u);
      if (r.wide) {
        ldg_pair(p, z[0], z[1]);
        ldg_pair(p + 2, z[2], z[3]);
      } else {
#pragma unroll
        for (int i = 0; i < 4; ++i) z[i] = __ldg(p + i);
      }
      mask = in ? 0xFFu : 0u;
      return;
    }
    const bool in = m <= r.n && (near ? m > r.edge : m <= r.edge);
    const bool above = m < r.diag || !in;
    const double2* p = r.tr + (in ? (unsigned)(m * MM + x) : 0u);
    if (!above) p = r.dr + (tri0(m) * (unsigned)MM + (unsigned)(x * M));
    const unsigned st = above ? 1u : (unsigned)M;
#pragma unroll
    for (int i = 0; i < 4; ++i) z[i] = __ldg(p + i * st);
    mask = (in ? 15u : 0u) | (above ? 0xF0u : 0u);
    return;
  }
  mask = 0;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const bool in = m <= r.n && (near ? m > r.edge : m <= r.edge);
    const bool above = m < r.diag;
    z[i] = make_double2(0.0, 0.0);
    if (in) z[i] = __ldg(above ? r.tr + (m * MM + x) : r.dr + (tri0(m) * (unsigned)MM + (unsigned)(x * M)));
    mask |= ((unsigned)in | ((unsigned)above << 4)) << i;
    if (++x == M) { x = 0; ++m; }
  }
}
// Four entries of the band of term 2 (plane R): w_{c,m} R(c,m)^+ for c - band_w < m
// <= c, in the adjoint w_{m,c} R(m,c) for c <= m < c + band_w.  band_values loads the
// entries, like load_quad a unit ahead; band_weights, when they are converted, their
// weights (which repeat from unit to unit, so they come from the L1 cache).  Loading
// both and multiplying at once, one entry after the other, took 3.0 to 3.8 us a unit where
// a far or near unit takes 1.4 to 1.8, and the CTA that holds a tile's band is the
// last of a short row.
template <class F>
__device__ __forceinline__ void for_band(const Sys& s, const Row& r, int kap, F f) {
  const int M = r.M, c = r.edge - s.shift;
  int m = div_m(kap, M, r.magic), x = kap - m * M;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int d = s.adj ? m - c : c - m;
    f(i, m, x, d, m <= r.n && d >= 0 && d < s.band_w);
    if (++x == M) { x = 0; ++m; }
  }
}
__device__ __forceinline__ void band_values(const Sys& s, const Row& r, int kap, bool live, double2 z[4]) {
  const int M = r.M, MM = M * M, adj = s.adj;
  for_band(s, r, kap, [&](int i, int m, int x, int, bool in) {
    z[i] = make_double2(0.0, 0.0);
    if (in && live) z[i] = __ldg(adj ? r.dr + (tri0(m) * (unsigned)MM + (unsigned)(x * M)) : r.tr + (m * MM + x));
  });
}
__device__ __forceinline__ void band_weights(const Sys& s, const Row& r, int kap, double2 z[4]) {
  const int adj = s.adj, c = r.edge - s.shift;
  for_band(s, r, kap, [&](int i, int m, int, int d, bool in) {
    if (!in) return;  // zero
    const double w = __ldg(s.band + (int64_t)(adj ? m : c) * s.band_w + d);
    z[i] = make_double2(w * z[i].x, adj ? w * z[i].y : -w * z[i].y);
  });
}

// ------------------------------------------------------------ epilogue ---
// Folds the accumulator buffer at `at` into the FP64 sums s of this thread's row
// and half of the a values, and hands the buffer back (empty) once its levels are
// in registers.  kWhole: every a value of the part is in use (otherwise the
// columns past the last one are skipped).  Two columns' levels are read at a time
// and reduced to 64-bit integers before the next two are: a read waits for tensor
// memory about as long as its arithmetic takes, and NA = 16, whose accumulations wait
// for it, has no registers to hold more (one column at a time with its levels converted
// first: M = 12, n = 389 in 549 us instead of 517, M = 16, n = 511 in 1.24 ms instead of 1.21).
template <int NA, bool kWhole>
__device__ __forceinline__ void fold(double (&s)[NA], uint32_t at, int E, int half, const Post& ps, uint64_t* empty) {
  constexpr int kN = 2 * NA, kC = NA, kCols = 2;  // kCols: columns in registers at a time
  const int cols = kWhole ? kC : (ps.cols - half) & ~1;
  uint32_t r[kDig][kCols];
  auto read = [&](int c2) {  // the levels of columns c2, ... in flight
#pragma unroll
    for (int d = 0; d < kDig; ++d)
#pragma unroll
      for (int i = 0; i < kCols; i += 2) {
        const uint32_t p = at + d * kN + 2 * (c2 + i);
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x2.b32 {%0,%1}, [%2];" : "=r"(r[d][i]), "=r"(r[d][i + 1]) : "r"(p));
      }
  };
  read(0);
#pragma unroll
  for (int c2 = 0; c2 < kC; c2 += kCols) {
    if (!kWhole && c2 > 0 && c2 >= cols) continue;
    int es[kCols / 2];
#pragma unroll
    for (int i = 0; i < kCols / 2; ++i) es[i] = ps.es[c2 + 2 * i + half];
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
    int64_t t[kCols];
#pragma unroll
    for (int i = 0; i < kCols; ++i) {
      int v[kDig];
#pragma unroll
      for (int d = 0; d < kDig; ++d) v[d] = __float2int_rn(__uint_as_float(r[d][i]));
      // the 64-bit integer sum_l S_l 256^(7-l) / 2^12: |S_0| <= 2^19, |S_1| <= 2^21, |S_2| <= 2^22 and
      // |S_l| <= l 2^21 fit the 32-bit steps, and 2^10 products of 62-bit values stay below 2^(124+7-56-12)
      const uint64_t p01 = (uint64_t)(int64_t)(v[0] * 256 + v[1]), p23 = (uint64_t)(int64_t)(v[2] * 256 + v[3]);
      const int low = v[5] * 16 + ((v[6] + (v[7] >> 8) + 8) >> 4);
      t[i] = (int64_t)((p01 << 36) + (p23 << 20) + ((uint64_t)(int64_t)v[4] << 12) + (uint64_t)(int64_t)low);
    }
    if (c2 + kCols < cols) {
      read(c2 + kCols);  // while these are scaled
    } else {
      tc_fence_before();
      __syncwarp();
      if ((threadIdx.x & 31) == 0) mbar_arrive(empty);
    }
#pragma unroll
    for (int i = 0; i < kCols; ++i) {
      // scale 2^(ev + eu - 68 + 12), ev = E - 1022, eu = es - 1022 (the entries' own exponents cancel)
      const int ex = E + es[i / 2] - 2 * 1022 - 56;
      if (ex >= -1022 && ex <= 1023) {
        s[c2 + i] = fma((double)t[i], __hiloint2double((ex + 1023) << 20, 0), s[c2 + i]);
      } else if (ex > kFiniteMost) {
        s[c2 + i] = __longlong_as_double(0x7FF8000000000000ll);
      } else {  // the scale alone leaves the range of FP64
        const int h = ex / 2;
        s[c2 + i] += (double)t[i] * __hiloint2double((h + 1023) << 20, 0) * __hiloint2double((ex - h + 1023) << 20, 0);
      }
    }
  }
}

// ---------------------------------------------------------------- main ---
// kTest: a launch whose producers stop at a unit (kbe_debug_withhold_split), an instantiation of its own (with the
// unit and the cycles read from the arguments the slice n = 1023, M = 8 took 858 us instead of 834).
template <int NA, bool kQuad, bool kTest = false>
__global__ void __launch_bounds__(kThreads, 1) fx_main(const __grid_constant__ Args a) {
  using C = Cfg<NA>;
  constexpr int kN = C::kN, kBufs = C::kBufs, kBufCols = C::kBufCols;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  Smem<NA>& sm = *reinterpret_cast<Smem<NA>*>(smem_raw);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

  if (tid == 0) {
    // empty, bempty: both MMA threads
    for (int i = 0; i < kStages; ++i) { mbar_init(&sm.full[i], kConvWarps); mbar_init(&sm.empty[i], 2); sm.raise[i] = 0; }
    for (int i = 0; i < kBSlots; ++i) { mbar_init(&sm.bfull[i], 1); mbar_init(&sm.bempty[i], 2); }
    // accfull: an MMA thread's arrival (post written) and its commit; accempty: one lane per epilogue warp
    for (int i = 0; i < kBufs; ++i) { mbar_init(&sm.accfull[i], 2); mbar_init(&sm.accempty[i], kEpiWarps); }
    mbar_init(&sm.mmadone[0], 1);
    mbar_init(&sm.mmadone[1], 1);
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
  grid_wait();  // the small operands are complete
  const long long total = head_of(a).total;
  const long long q0 = range_lo(total, a.G, blockIdx.x), q1 = range_lo(total, a.G, blockIdx.x + 1);
  int* const status = sys_at(a, 0).status;

  if (warp < kEpiWarps) {
    // --------------------------------------------------------- epilogue --
    // warp = 4 half + quadrant: 32 output rows (tensor-memory lanes), the even
    // or the odd a values of the part (kN / 2 columns)
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(Regs<NA, kQuad>::kEpi));
    constexpr int kC = kN / 2;
    const int quad = warp & 3, half = warp >> 2;
    const int j = quad * 32 + lane;
    const uint32_t lane_addr = tmem + ((uint32_t)(quad * 32) << 16) + 2 * half;  // + 4 (c / 2) + c % 2
    double acc[2][kC];
#pragma unroll
    for (int i = 0; i < kC; ++i) acc[0][i] = acc[1][i] = 0.0;
    unsigned used[2] = {0, 0};  // buffers taken from each MMA thread
    for (int from = 0;;) {      // thread 0's message, or its sum and then thread 1's
      const unsigned k = from ? used[1]++ : used[0]++;
      const int buf = 2 * (k % (kBufs / 2)) + from;
      if (!__all_sync(0xffffffffu, wait_bar<kTest>(a, &sm.abort, &sm.accfull[buf], (k / (kBufs / 2)) & 1, status))) break;
      tc_fence_after();
      const Post& ps = sm.post[buf];
      const int type = ps.type;
      if (type == kEnd) break;
      if (type == kUnit) from ^= 1;
      if (type != kUnit) {
        const Sys& s = sys_at(a, ps.si);
        if (type == kFlush) {
          double2* out = reinterpret_cast<double2*>(s.part) + (size_t)ps.slot * C::kSlot;
#pragma unroll
          for (int g = 0; g < 2; ++g)
#pragma unroll
            for (int i = 0; i < kC / 2; ++i) {
              out[(g * NA + 2 * i + half) * kRows + j] = make_double2(acc[g][2 * i], acc[g][2 * i + 1]);
              acc[g][2 * i] = acc[g][2 * i + 1] = 0.0;
            }
        } else {  // the adjoint's sums, before its band
          const int m = min(ps.c0 + div_m(j, s.M, s.magic), s.n);
          const double wn = weights_of(s).at(s.n, m), wb = -s.wbar[m];
#pragma unroll
          for (int i = 0; i < kC; ++i) {
            acc[0][i] *= wn;
            acc[1][i] *= wb;
          }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&sm.accempty[buf]);
        continue;
      }
      const int g = ps.grp;
      const int E = sm.erow[ps.eidx][ps.plane][j];
      uint64_t* const empty = &sm.accempty[buf];
      const uint32_t at = lane_addr + buf * kBufCols;
      if (ps.cols > NA) {
        if (g == 0) fold<NA, true>(acc[0], at, E, half, ps, empty);
        else fold<NA, true>(acc[1], at, E, half, ps, empty);
      } else {
        if (g == 0) fold<NA, false>(acc[0], at, E, half, ps, empty);
        else fold<NA, false>(acc[1], at, E, half, ps, empty);
      }
    }
  } else if (warp < kMmaWarp) {
    // ------------------------------------------------------- converters --
    // lane = row (3 bits) | K half q << 3 | plane << 4: a quarter warp writes
    // 128 consecutive bytes of a digit plane
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(Regs<NA, kQuad>::kConv));
    const int wq = warp - kEpiWarps;
    const int q = (lane >> 3) & 1, plane = lane >> 4;
    const uint32_t dst0 = plane * kPlane + (q * 16 + wq) * 128 + (lane & 7) * 16;
    Row row;
    double2 z[4];
    unsigned mask = 0, d = 0;
    uint2 ekw = make_uint2(0, 0);  // exponents of the entries in z
    int flags = 0, kap = 0, si = 0, E = 64, seen = 0;  // of the unit in z; the row's exponent; largest field of the current chunk
    // the next unit's loads; false when there is none
    auto load = [&]() -> bool {
      Desc ds;
      do {
        const int b = d % kBSlots;
        if (!__all_sync(0xffffffffu, wait_bar<kTest>(a, &sm.abort, &sm.bfull[b], (d / kBSlots) & 1, status))) return false;
        ds = sm.desc[b];
        ++d;
      } while (kind_of(ds.flags) == kFlush || kind_of(ds.flags) == kScale);
      flags = ds.flags;
      if (kind_of(flags) == kEnd) return false;
      if (flags & kNewTile) row = row_of(sys_at(a, ds.aux), ds.c0, 8 * wq + (lane & 7), plane);
      kap = ds.kap + 4 * q;
      si = ds.aux;
      // (read here and not when the unit is converted: behind the digit stores a read waits long; M = 8, n = 1023 963 us instead of 865)
      ekw = *reinterpret_cast<const uint2*>(
          &reinterpret_cast<const Exps*>(sm.small[(d - 1) % kBSlots])->ek[plane && !(flags & kFlagNear)][2 * q]);
      if (flags & kFlagBand) {
        band_values(sys_at(a, ds.aux), row, kap, plane, z);
        mask = 15u;
      } else {
        load_quad<kQuad>(row, kap, flags & kFlagNear, !(flags & (kFlagNear | kFlagLow)), z, mask);
      }
      return true;
    };
    bool more = load();
    for (unsigned u = 0; more; ++u) {
      const int s = u % kStages;
      if (flags & kFlagBand) band_weights(sys_at(a, si), row, kap, z);
      // exponent of the row, of the entries scaled as the small operand says
      const uint32_t ek[4] = {ekw.x << 20, ekw.x & 0xFFF00000u, ekw.y << 20, ekw.y & 0xFFF00000u};
      uint32_t top = 0, most = 0;  // (a zero counts as 2^-1022: below any product that matters)
#pragma unroll
      for (int i = 0; i < 4; ++i) {  // masked entries are zero without kQuad
        const uint32_t re = (uint32_t)__double2hiint(z[i].x) & 0x7FFFFFFFu, im = (uint32_t)__double2hiint(z[i].y) & 0x7FFFFFFFu;
        most = __vimax3_u32(most, re, im);
        top = __vimax3_u32(top, re + ek[i], im + ek[i]);
      }
      int mx = (int)(top >> 20);
      if (most < 0x100000u || (kQuad && !(mask & 1u))) mx = 0;  // nothing but zeros
      else if (most >= 0x7FF00000u) mx = kNonFinite;
      mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, 8));
      bool raised = false;
      if (flags & kFirst) {
        const int prev = (flags & kFresh) || seen == kNonFinite ? 0 : seen;
        E = max(max(mx, prev), least_of(ekw.x, ekw.y)) + (prev ? kHeadroom : kStartRoom);
        seen = mx;
      } else {
        if (mx > E) { raised = seen > 0; E = mx + (raised ? kHeadroom : kStartRoom); }
        seen = max(seen, mx);
      }
      if (mx == kNonFinite) E = kNonFinite;
      const int Ez = kQuad && !(mask & 1u) ? kNonFinite : E;  // a masked quad's digits are zero
      uint64_t br[4], bi[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const uint32_t fl = (kQuad ? mask << 24 : mask << (27 - i)) & 0x80000000u;
        const uint32_t re = (uint32_t)__double2hiint(z[i].x), im = (uint32_t)__double2hiint(z[i].y);
        // E - ek - field, summed in the order that costs fewer registers (M = 8, n = 1023: 865 -> 836 us; M = 5, n = 333:
        // 226 -> 217 us a step the other way)
        if constexpr (NA == 8 && kQuad) {
          const int Ei = Ez - (int)(ek[i] >> 20);
          br[i] = digit_bytes(re ^ fl, (uint32_t)__double2loint(z[i].x), Ei);
          bi[i] = digit_bytes(im, (uint32_t)__double2loint(z[i].y), Ei);
        } else {
          br[i] = digit_bytes_at(re ^ fl, (uint32_t)__double2loint(z[i].x), Ez - (int)(((re & 0x7FFFFFFFu) + ek[i]) >> 20));
          bi[i] = digit_bytes_at(im, (uint32_t)__double2loint(z[i].y), Ez - (int)(((im & 0x7FFFFFFFu) + ek[i]) >> 20));
        }
      }
      more = load();  // in flight while this unit's digits are written
      if (!__all_sync(0xffffffffu, wait_bar<kTest>(a, &sm.abort, &sm.empty[s], ((u / kStages) & 1) ^ 1, status))) break;
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
  } else {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(Regs<NA, kQuad>::kMisc));
    if (warp == kProdWarp && lane == 0) {
      // ------------------------------------------------------- producer --
      unsigned d = 0;
      // the next slot, its descriptor written; false when the wait ran out
      auto put = [&](int kap, int c0, int flags, int aux) -> bool {
        const int b = d % kBSlots;
        if (!wait_bar<kTest>(a, &sm.abort, &sm.bempty[b], ((d / kBSlots) & 1) ^ 1, status)) return false;
        sm.desc[b] = Desc{kap, c0, flags, aux};
        return true;
      };
      auto message = [&](int kind, int kap, int c0, int aux) -> bool {
        if (!put(kap, c0, kind << 8, aux)) return false;
        mbar_arrive(&sm.bfull[d++ % kBSlots]);
        return true;
      };
      bool stop = false;
      if (q0 < q1) {
        long long q = q0;
        int si = find_sys(a, q0, [](const Sys& y) { return y.unit_base; });
        const Sys* S = &sys_at(a, si);
        Walk w;
        walk_to(w, *S, si, q0 - S->unit_base);
        int fresh = kFresh | kNewTile, cls = -1;
        bool scaled = false, joined = false;
        int units = 0;
        while (q < q1 && !stop) {
          if (w.cls != cls) fresh |= kFresh;
          if (S->adj && !scaled && w.cls == kBand && w.j0 < w.j1) {
            if (!message(kScale, 0, w.c0, si)) break;
            scaled = true;
          }
          // a sum takes one plane, so two chunks (an even one and the next) stay
          // within 2^10 products of 2^14 and are accumulated together
          const bool join = w.cls != kBand && !(w.kc & 1) && q + 1 < q1 &&
                            w.idx + 1 < (w.cls == kFar ? w.nfar : w.nfar + S->cpt - w.first);
          const uint32_t bytes = kExpBytes + (w.cls == kNear ? 1 : 2) * C::kVarBytes;
          const uint8_t* src = S->small + (w.cls == kBand ? C::kHalfBytes : 0) +
                               ((size_t)w.kc * kChunkUnits * S->parts + w.part) * C::kSmallBytes;
          for (int unit = w.j0; unit < w.j1; ++unit) {
            if (kTest && units++ == a.withhold) { stop = true; break; }
            const int flags = (w.cls == kNear ? kFlagNear : 0) | (w.cls == kBand ? kFlagBand : 0) |
                              (unit == w.j0 && !joined ? kFirst : 0) | (unit + 1 == w.j1 && !join ? kLast : 0) |
                              (S->adj ? kFlagLow : 0) | min(NA, S->M - w.part * NA) << 16;
            if (!put(w.kc * kChunkK + unit * kUnitK, w.c0, kUnit << 8 | flags | fresh, si)) { stop = true; break; }
            const int b = d % kBSlots;
            mbar_arrive_expect_tx(&sm.bfull[b], bytes);
            bulk_g2s(sm.small[b], src + (size_t)unit * S->parts * C::kSmallBytes, bytes, &sm.bfull[b]);
            ++d;
            fresh = 0;
            cls = w.cls;
          }
          if (stop) break;
          joined = join;
          const int T = w.T, c0 = w.c0, slot = T + (int)blockIdx.x - S->cta0, sys = si;
          const bool adj = S->adj;
          int moved = 1;
          if (++q < q1) {
            moved = walk_next(w, *S);
            if (moved == 2) {
              S = &sys_at(a, ++si);
              walk_to(w, *S, si, 0);
            }
          }
          if (moved) {
            if (adj && !scaled && !message(kScale, 0, c0, sys)) { stop = true; break; }
            if (!message(kFlush, sys, 0, slot)) { stop = true; break; }
            fresh = kFresh | kNewTile;
            scaled = false;
          }
        }
      }
      if (!stop) message(kEnd, 0, 0, 0);
      // the copies already issued must land before the CTA can exit (each slot's last phase)
      for (unsigned k = d > kBSlots ? d - kBSlots : 0; k < d; ++k) {
        long long spins = 0;
        while (!mbar_try(&sm.bfull[k % kBSlots], (k / kBSlots) & 1) && ++spins < kSpinLimit) __nanosleep(64);
        if (spins >= kSpinLimit) atomicOr(status, kStatusTimeout);
      }
    } else if ((warp == kMmaWarp || warp == kMmaWarp2) && lane == 0) {
      // ----------------------------------------------------- MMA threads --
      // Thread 0 issues the first of a unit's two products, thread 1 the second,
      // each into accumulator buffers of its own: one alone leaves the tensor
      // cores idle between its units.  Both walk the same descriptors; thread
      // `me` takes the buffers me, me + 2, ... in turn.
      // A: [digit 8][K group 2][row group 16][8 rows][16 B]; B: [K group 2][digit 8][column group][8][16 B]
      const int me = warp == kMmaWarp ? 0 : 1;
      const uint64_t a0 = umma_desc(smem_u32(sm.stage[0]), kRows * 16, 128);
      const uint64_t b0 = umma_desc(smem_u32(sm.small[0] + kExpBytes), kDig * (kN / 8) * 128, 128);
      unsigned u = 0, k = 0;  // units; this thread's buffers taken
      bool any = false, stop = false, open = false;
      unsigned held = 0;  // slots (bits) of messages not released yet
      int buf = me;
      auto next_buffer = [&]() {
        ++k;
        buf = 2 * (k % (kBufs / 2)) + me;
      };
      auto wait_buffer = [&]() {
        return wait_bar<kTest>(a, &sm.abort, &sm.accempty[buf], ((k / (kBufs / 2)) & 1) ^ 1, status);
      };
      auto close = [&]() {
        sm.post[buf].eidx = (u - 1) % kExpRing;
        mbar_arrive(&sm.accfull[buf]);
        umma_commit(&sm.accfull[buf]);
        next_buffer();
        open = false;
      };
      // hands a message without sums to the epilogue (thread 0)
      auto message = [&](int type, int si, int c0, int slot) -> bool {
        if (me) return true;
        if (!wait_buffer()) return false;
        Post& ps = sm.post[buf];
        ps.type = type;
        ps.si = si;
        ps.c0 = c0;
        ps.slot = slot;
        mbar_arrive(&sm.accfull[buf]);
        mbar_arrive(&sm.accfull[buf]);
        next_buffer();
        return true;
      };
      for (unsigned d = 0; !stop; ++d) {
        const int b = d % kBSlots;
        if (!wait_bar<kTest>(a, &sm.abort, &sm.bfull[b], (d / kBSlots) & 1, status)) { stop = true; break; }
        const Desc ds = sm.desc[b];
        const int kind = kind_of(ds.flags);
        if (kind == kEnd) break;
        if (kind != kUnit) {
          // released when the next unit is full: then every converter has read
          // past this descriptor (at most a scaling and a flush come in a row,
          // since every tile starts with a unit)
          held |= 1u << b;
          if (!message(kind, kind == kFlush ? ds.kap : ds.aux, ds.c0, ds.aux)) stop = true;
          continue;
        }
        const int s = u % kStages;
        const bool near = ds.flags & kFlagNear, band = ds.flags & kFlagBand;
        if (!wait_bar<kTest>(a, &sm.abort, &sm.full[s], (u / kStages) & 1, status)) { stop = true; break; }
        for (int i = 0; i < kBSlots && held; ++i)
          if (held >> i & 1u) {
            mbar_arrive(&sm.bempty[i]);
            held &= ~(1u << i);
          }
        const bool begin = (ds.flags & kFirst) || *(volatile unsigned*)&sm.raise[s] == u + 1;
        if (begin) {
          if (open) close();
          open = true;
          if (!wait_buffer()) { stop = true; break; }
          Post& ps = sm.post[buf];
          ps.type = kUnit;
          ps.grp = me && (near || band);
          ps.plane = band ? 1 : me;
          ps.cols = (ds.flags >> 16) + 1;
#pragma unroll
          for (int i = 0; i < NA / 8; ++i)
            reinterpret_cast<int4*>(ps.es)[i] =
                reinterpret_cast<const int4*>(reinterpret_cast<const Exps*>(sm.small[b])->es[me && !near])[i];
        }
        tc_fence_after();
        // far: PL x variant 0 and Q x variant 1, both to I^<; near: PL and Q x
        // variant 0 to I^< and D; band: Q x variants 0 and 1 to I^< and D
        const uint64_t x = a0 + ((uint64_t)(s * 2 * kPlane + (me || band ? kPlane : 0)) >> 4);
        const uint64_t v = b0 + ((uint64_t)(b * C::kHalfBytes + (me && !near ? C::kVarBytes : 0)) >> 4);
        const uint32_t t = tmem + buf * kBufCols;
#pragma unroll
        for (int i = 0; i < kDig; ++i)
          umma_f16(t + i * kN, x + ((i * kDigPlane) >> 4), v, umma_idesc_f16(kN * (kDig - i)), !(begin && i == 0));
        umma_commit(&sm.empty[s]);
        umma_commit(&sm.bempty[b]);
        any = true;
        ++u;
        if (ds.flags & kLast) close();
      }
      if (!stop) message(kEnd, 0, 0, 0);
      // every MMA must complete before tensor memory is freed
      if (any) {
        umma_commit(&sm.mmadone[me]);
        long long spins = 0;
        while (!mbar_try(&sm.mmadone[me], 0) && ++spins < kSpinLimit) __nanosleep(64);
        if (spins >= kSpinLimit) atomicOr(status, kStatusTimeout);
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
// Output entries (c, a, b): the partial sums of their tile in CTA order.
template <int NA>
__global__ void __launch_bounds__(256) fx_reduce(const __grid_constant__ Args a) {
  grid_wait();
  const Head& h = head_of(a);
  const long long entries = h.entries, total = h.total;
  for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < entries;
       e += (long long)gridDim.x * blockDim.x) {
    const Sys& s = sys_at(a, find_sys(a, e, [](const Sys& y) { return y.entry_base; }));
    const long long lin = e - s.entry_base;
    const int M = s.M, MM = M * M;
    const int c = rk::div_idx(lin, MM), ab = (int)(lin - (long long)c * MM), row = ab / M, b = ab - row * M;
    const int ct = c / s.CT, T = ct * s.parts + row / NA;
    const int64_t at = (int64_t)(row % NA) * kRows + (c - ct * s.CT) * M + b;
    const long long lo = s.unit_base + (long long)T * s.upt, hi = lo + s.upt;
    double2 p = make_double2(0.0, 0.0), d = p;
    for (int i = cta_of(total, a.G, lo); i < a.G && range_lo(total, a.G, i) < hi; ++i) {
      if (range_lo(total, a.G, i + 1) <= range_lo(total, a.G, i)) continue;
      const double2* q = reinterpret_cast<const double2*>(s.part) + (size_t)(T + i - s.cta0) * Cfg<NA>::kSlot;
      const double2 x = q[at], y = q[at + NA * kRows];
      p.x += x.x; p.y += x.y;
      d.x += y.x; d.y += y.y;
    }
    // slice: I^<, I^> = I^< + D; adjoint: S^>bar, S^<bar = C - S^>bar
    const double2 q = s.adj ? make_double2(d.x - p.x, d.y - p.y) : make_double2(p.x + d.x, p.y + d.y);
    reinterpret_cast<double2*>(s.adj ? s.out1 : s.out0)[lin] = p;
    reinterpret_cast<double2*>(s.adj ? s.out0 : s.out1)[lin] = q;
    if (!s.adj && !(isfinite(p.x) && isfinite(p.y) && isfinite(q.x) && isfinite(q.y))) atomicOr(s.status, kStatusNumeric);
  }
}

// prep, contraction and reduction of the systems of `a`
template <int NA>
cudaError_t enqueue(const Args& a, bool quad, unsigned prep_blocks, unsigned red_blocks, cudaStream_t st, int* launches,
                    cudaEvent_t ev_begin, cudaEvent_t ev_end) {
  cudaError_t e = launch_overlapped(fx_prep<NA>, prep_blocks, 32 * NA, 0, st, a);
  if (e != cudaSuccess) return e;
  ++*launches;
  if (a.wait_cycles) {
    if (ev_begin) cudaEventRecord(ev_begin, st);
    fx_main<NA, false, true><<<a.G, kThreads, sizeof(Smem<NA>), st>>>(a);
    e = cudaGetLastError();
    if (ev_end) cudaEventRecord(ev_end, st);
  } else if (ev_begin) {  // timed: no overlap with the kernels around it
    cudaEventRecord(ev_begin, st);
    if (quad) fx_main<NA, true><<<a.G, kThreads, sizeof(Smem<NA>), st>>>(a);
    else fx_main<NA, false><<<a.G, kThreads, sizeof(Smem<NA>), st>>>(a);
    e = cudaGetLastError();
    cudaEventRecord(ev_end, st);
  } else {
    e = launch_overlapped(quad ? fx_main<NA, true> : fx_main<NA, false>, a.G, kThreads, sizeof(Smem<NA>), st, a);
  }
  if (e != cudaSuccess) return e;
  ++*launches;
  if ((e = launch_overlapped(fx_reduce<NA>, red_blocks, 256, 0, st, a)) != cudaSuccess) return e;
  ++*launches;
  return cudaSuccess;
}

// One system's contraction in its workspace.
cudaError_t launch_one(Sys s, int M, int n, int band_w, int adj, void* work, size_t work_bytes, cudaStream_t st,
                       int* launches, cudaEvent_t ev_begin, cudaEvent_t ev_end, long long withhold = -1,
                       long long spin_limit = 0) {
  *launches = 0;
  if (M < 1 || M > kMaxNorb || n < 0) return cudaErrorInvalidValue;
  const int NA = part_rows(M);
  set_geometry(s, M, n, band_w, adj, NA);
  s.small = reinterpret_cast<uint8_t*>(work);
  s.part = reinterpret_cast<double*>(s.small + small_bytes(s, NA));
  Args a{};
  a.one_head.n_sys = 1;
  a.one_head.total = (long long)s.tiles * s.upt;
  a.one_head.chunks = prep_items(s);
  a.one_head.entries = (long long)(n + 1) * M * M;
  a.G = (int)std::min<long long>(a.one_head.total, sm_count());
  if (small_bytes(s, NA) + ((size_t)s.tiles + a.G) * slot_complex(NA) * 16 > work_bytes) return cudaErrorInvalidValue;
  a.one = s;
  if (withhold >= 0) {
    a.withhold = (int)std::min<long long>(withhold, 1 << 30);
    a.wait_cycles = 256 * std::min<long long>(spin_limit, kWaitCycles / 256);
  }
  cudaError_t e = fx_prepare();
  if (e != cudaSuccess) return e;
  const unsigned prep = (unsigned)std::min<long long>(a.one_head.chunks, 1 << 30);
  const unsigned red = (unsigned)std::min<long long>((a.one_head.entries + 255) / 256, 1 << 30);
  return NA == 8 ? enqueue<8>(a, M % 4 == 0, prep, red, st, launches, ev_begin, ev_end)
                 : enqueue<16>(a, M % 4 == 0, prep, red, st, launches, ev_begin, ev_end);
}

}  // namespace

size_t fx_workspace_bytes(int M, int n_max) {
  if (M < 1 || M > kMaxNorb || n_max < 1) return 0;
  Sys s{};
  const int NA = part_rows(M);
  set_geometry(s, M, n_max - 1, kMaxOrder + 1, 0, NA);
  return small_bytes(s, NA) + ((size_t)s.tiles + sm_count()) * slot_complex(NA) * 16;
}

// The main kernels' dynamic shared memory exceeds the default limit (set once per device).
cudaError_t fx_prepare() {
  static std::atomic<unsigned long long> done_mask{0};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const unsigned long long bit = 1ull << (dev & 63);
  if (done_mask.load() & bit) return cudaSuccess;
  const auto set = [](const void* f, size_t bytes) {
    return cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  };
  e = set((const void*)fx_main<8, true>, sizeof(Smem<8>));
  if (e == cudaSuccess) e = set((const void*)fx_main<8, false>, sizeof(Smem<8>));
  if (e == cudaSuccess) e = set((const void*)fx_main<16, true>, sizeof(Smem<16>));
  if (e == cudaSuccess) e = set((const void*)fx_main<16, false>, sizeof(Smem<16>));
  if (e == cudaSuccess) e = set((const void*)fx_main<8, false, true>, sizeof(Smem<8>));
  if (e == cudaSuccess) e = set((const void*)fx_main<16, false, true>, sizeof(Smem<16>));
  if (e == cudaSuccess) done_mask.fetch_or(bit);
  return e;
}

cudaError_t launch_history_fx(const HistoryArgs& h, void* work, size_t work_bytes, cudaStream_t st, int* launches) {
  Sys s{};
  s.L = h.L;
  s.R = h.R;
  s.Sl = h.Sl;
  s.Sg = h.Sg;
  s.wbar = h.w.wbar;
  s.band = h.w.band;
  s.out0 = h.out;
  s.out1 = h.out + 2 * (size_t)(h.n + 1) * h.M * h.M;
  s.status = h.status;
  return launch_one(s, h.M, h.n, h.w.band_w, 0, work, work_bytes, st, launches, h.ev_begin, h.ev_end, h.withhold,
                    h.spin_limit);
}

cudaError_t launch_fx_table(int NA, bool quad, const Sys* table, const Head* head, cudaStream_t st, int* launches) {
  *launches = 0;
  Args a{};
  a.table = table;
  a.head = head;
  a.G = sm_count();
  const unsigned prep = (unsigned)a.G * (NA == 8 ? 8 : 4), red = (unsigned)a.G * 8;
  return NA == 8 ? enqueue<8>(a, quad, prep, red, st, launches, nullptr, nullptr)
                 : enqueue<16>(a, quad, prep, red, st, launches, nullptr, nullptr);
}

// The Sigma-row cotangents of the slice's adjoint (the sums of adj_hist_small and its reduction).
cudaError_t launch_adjoint_fx(const AdjHistArgs& h, void* work, size_t work_bytes, int* status, cudaStream_t st,
                              int* launches) {
  Sys s{};
  s.L = h.L;
  s.R = h.R;
  s.Sl = h.Ib;
  s.Sg = h.Ib + 2 * (size_t)(h.n + 1) * h.M * h.M;
  s.wbar = h.w.wbar;
  s.band = h.w.band;
  s.out0 = h.dSl;
  s.out1 = h.dSg;
  s.status = status;
  return launch_one(s, h.M, h.n, h.w.band_w, 1, work, work_bytes, st, launches, nullptr, nullptr);
}

}  // namespace kbe
