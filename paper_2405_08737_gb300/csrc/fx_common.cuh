// fx_common.cuh -- geometry and digit conversion of the FP64 history slice on
// the 16-bit-float tensor cores (history_fx.cu).  Everything here runs on the
// host too, so that the walk over the work and the conversion can be checked
// without a GPU.
//
// Operands and products.  A double v with |v| < 2^e becomes the 62-bit integer
// V = trunc(v 2^(62-e)) in eight balanced base-256 digits, V = sum_i d_i
// 256^(7-i), d_0 in [-64, 64], the others in [-128, 127] (|d| <= 128 for the
// negated digits of the small operand): each is exact in fp16, a product of two
// is at most 2^14, and a sum of 2^10 of them is an integer of at most 2^24,
// exact in FP32 in any order.  With the digit products of levels l = i + j =
// 0..7 (36 of the 64), v u = 2^(ev+eu-68) sum_l S_l 256^(7-l): the dropped
// levels weigh at most 2^-59 of 2^(ev+eu), typically 2^-61, where FP64 rounds
// every partial sum at 2^-53 (error-free slicing: Ozaki, Ogita, Oishi & Rump,
// Numer. Algorithms 59 (2012)).
#pragma once

#include <cstdint>

namespace kbe {
namespace fx {

constexpr int kDig = 8;        // digits per value
constexpr int kRows = 128;     // output rows (c, b) of a column tile, one tensor-memory lane each
constexpr int kUnitK = 8;      // complex history entries of a unit (one MMA K step of 16 reals)
constexpr int kChunkUnits = 4; // units accumulated in tensor memory: 2 planes x 64 reals x 8 digit pairs = 2^10 products
constexpr int kChunkK = kUnitK * kChunkUnits;
constexpr int kOver = 6;       // chunks that a column tile visits twice, at most (see Walk)
constexpr int kHeadroom = 2;   // bits between a row's exponent and its first values
constexpr int kNonFinite = 8000;  // exponent of a row or column that holds a non-finite value

// One system's slice as a list of column tiles of CT = 128 / M output columns
// (times parts of the small operand's rows a).
struct Sys {
  const double* L;
  const double* R;
  const uint8_t* small;   // [unit][part][small block]: written by the prep kernel
  int M, n, CT, cpt;      // chunks per pass over the history: ceil((n + 1) M / 32)
  int parts, tiles;       // parts of a; column tiles x parts
  int upt;                // chunk slots per tile: cpt + kOver
  int shift;              // history point m of column c is "near" when m > c + shift, else "far"
  uint32_t magic;         // ceil(2^32 / M) (0 for M = 1): x / M without a division
  long long unit_base;    // first chunk slot and first tile of the system in the launch
  long long tile_base;
};

// x / M for 0 <= x < 2^32 / M
__host__ __device__ __forceinline__ int div_m(int x, int M, uint32_t magic) {
  if (M == 1) return x;
#ifdef __CUDA_ARCH__
  return (int)__umulhi((uint32_t)x, magic);
#else
  return (int)(((uint64_t)(uint32_t)x * magic) >> 32);
#endif
}

// A role's walk over the chunk slots of the launch.  A column tile's chunks come
// in this order: first the far ones (entries with m <= c + shift count, both
// planes into one sum), then the near ones (m > c + shift, one sum per plane).
// The at most kOver chunks that straddle the line are taken once each way, with
// the other side's entries masked; the remaining slots of a tile are empty.
struct Walk {
  // system (copied: every role reads these once per unit)
  int M, n, shift, parts, cpt, CT, upt, tiles;
  uint32_t magic;
  int si;
  // tile
  int T, part, c0;      // tile of the system, its part, first column
  int nfar, far_k;      // far chunks and entries
  int first, near_k;    // first near chunk and entry
  // chunk slot
  int idx;
  int near;             // 0: far, 1: near
  int kc, j0, j1;       // chunk of the history and its units [j0, j1) (empty slot: j0 = j1)

  __host__ __device__ __forceinline__ void set_sys(const Sys& s, int i) {
    M = s.M; n = s.n; shift = s.shift; parts = s.parts; cpt = s.cpt; CT = s.CT; upt = s.upt; tiles = s.tiles;
    magic = s.magic;
    si = i;
  }
  // position T, c0 and part are set
  __host__ __device__ __forceinline__ void tile_start() {
    const int c1 = c0 + CT - 1 < n ? c0 + CT - 1 : n;
    const int far_m = c1 + shift < n ? c1 + shift : n;                 // last far point of the tile
    const int near_m = c0 + shift + 1 > 0 ? c0 + shift + 1 : 0;        // its first near point
    far_k = far_m < 0 ? 0 : (far_m + 1) * M;
    nfar = (far_k + kChunkK - 1) / kChunkK;
    near_k = near_m * M;
    first = near_m > n ? cpt : near_k / kChunkK;
  }
  __host__ __device__ __forceinline__ void chunk_start() {
    near = idx >= nfar;
    kc = near ? first + idx - nfar : idx;
    const int end = near ? (n + 1) * M : far_k;
    const int u = (end - kc * kChunkK + kUnitK - 1) / kUnitK;
    j1 = kc >= cpt ? 0 : (u < kChunkUnits ? u : kChunkUnits);
    j0 = near && kc == first && kc < cpt ? (near_k - kc * kChunkK) / kUnitK : 0;
  }
};
__host__ __device__ __forceinline__ void walk_to(Walk& w, const Sys& s, int i, long long slot) {
  w.set_sys(s, i);
  w.T = (int)(slot / s.upt);
  w.idx = (int)(slot - (long long)w.T * s.upt);
  const int ct = w.T / s.parts;
  w.part = w.T - ct * s.parts;
  w.c0 = ct * s.CT;
  w.tile_start();
  w.chunk_start();
}
// The next slot of the launch; 1: of another tile, 2: past the system's last
// tile (the caller moves to the next system, if any).
__host__ __device__ __forceinline__ int walk_next(Walk& w) {
  int moved = 0;
  if (++w.idx == w.upt) {
    w.idx = 0;
    if (++w.T == w.tiles) return 2;
    if (++w.part == w.parts) {
      w.part = 0;
      w.c0 += w.CT;
    }
    w.tile_start();
    moved = 1;
  }
  w.chunk_start();
  return moved;
}

// Chunk slots [lo, hi) of CTA i of G over `total` slots, and the slot of the
// partial sums of tile `tile` (counted over the launch) in CTA i: unique, since
// CTAs take contiguous ranges.
__host__ __device__ __forceinline__ long long range_lo(long long total, int G, int i) { return total * i / G; }
__host__ __device__ __forceinline__ long long partial_slot(long long tile, int i) { return tile + i; }

// Biased exponent field of the high word of a double.
__host__ __device__ __forceinline__ int field_of(uint32_t hi) { return (int)((hi >> 20) & 0x7FFu); }

// Digits of v for exponent field E (every |v| < 2^(E - 1022)), as the bytes
// d_i + 128 of a 64-bit word, d_0 on top.  Values more than 2^62 below the
// exponent (zeros and, for E < 64, everything below 2^-1020) give 0.
__host__ __device__ __forceinline__ uint64_t digit_bytes(uint32_t hi, uint32_t lo, int E) {
  int t = E - field_of(hi);
  t = t < 63 ? t : 63;
  const uint64_t m = ((uint64_t)((hi & 0xFFFFFu) | 0x100000u) << 32) | lo;
  const uint64_t V = (m << 9) >> t;
  const uint64_t sg = (uint64_t)((int64_t)(int32_t)hi >> 31);  // 0 or all ones
  return (V ^ sg) + 0x8080808080808080ull - sg;
}

}  // namespace fx
}  // namespace kbe
