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
//
// Exponents are shared: by a history row (c, b) over an accumulation of up to 64
// entries k = (m, x), by a row a of the small operand A over the same.  Entries are
// scaled first, A(a,k) by 1 / s_k and the history by s_k = max_a |A(a,k)| (Exps), so
// 2^(ev+eu) is at most 2^5 times r_a max_k s_k |G(k,c,b)| with r_a = max_k |A(a,k)| / s_k
// <= 1: the largest product of the accumulation and of the chunk before it, whose
// exponent the row starts from.  Per accumulation the error is then at most 2^-46 of
// that product, typically 2^-53.  It is the output's own largest product where the rows a
// differ by a factor each; where they do not, it is that of a larger row of the part.
#pragma once

#include <cstdint>

namespace kbe {
namespace fx {

constexpr int kDig = 8;        // digits per value
constexpr int kRows = 128;     // output rows (c, b) of a column tile, one tensor-memory lane each
constexpr int kUnitK = 8;      // complex history entries of a unit (one MMA K step of 16 reals)
constexpr int kChunkUnits = 4; // units of a chunk; two chunks of a plane accumulate: 128 reals x 8 digit pairs = 2^10
constexpr int kChunkK = kUnitK * kChunkUnits;
constexpr int kOver = 6;       // chunks that a column tile visits twice, at most (see Walk)
// Bits between a row's exponent and its first values, after a chunk of them and at a start.
// A bit more of either saves accumulations closed early and costs accuracy (rms error of slices
// n = 60..400 in units of the slice 4.8e-17, with 3 bits after a chunk 5.3e-17, with 5 at a start 6.2e-17; M = 16,
// n = 511 1237 us, 1205 and 1203 with both; FP64 sums: 12.6e-17).
constexpr int kHeadroom = 2, kStartRoom = 3;
constexpr int kNonFinite = 8000;  // exponent of a row or column that holds a non-finite value
constexpr int kFiniteMost = 2100; // no sum of two exponents of finite values scales by more than 2^this

// Exponents of a half of a unit's small block, ahead of its digits.  An entry k of
// the small operand is scaled by 2^-ek (its largest value over the rows a of the
// part), the history entry it meets by 2^ek: then a history row's exponent holds
// the largest of its products, whatever the two sizes do along the history, over
// the orbitals or between the two variants.  With exponents of the operands alone a column's
// error was up to 6e-10 of its own products for a self-energy that rises by 2^24 and a
// history that falls by 2^8 a point (M = 33), 5e-6 for G^< and Sigma^< 2^-40 of G^> and
// Sigma^>, and all of it for orbitals of very different sizes.
struct Exps {
  int16_t es[2][16];    // of row a, per variant
  uint32_t ek[2][4];    // of entries 2i and 2i + 1 in bits 0-11 and 20-31 of word i, per variant (the band's
                        // variants share one); bits 12-19 of words i and i + 1 (i even) hold `least`, the least
                        // exponent of a history row: its zeros lie 63 bits below it at every entry
  uint32_t pad[8];      // to 128 bytes: the digits' core matrices behind it stay in one line each
};
// `least` of the words 2q, 2q + 1
__host__ __device__ __forceinline__ int least_of(uint32_t w0, uint32_t w1) {
  return (int)((w0 >> 12 & 0xFFu) | (w1 >> 4 & 0xFF00u));
}

// Values of a per part, bytes of a part's small operand of one unit (two halves
// of exponents and two variants of 8 digits x 16 reals x 2 NA columns),
// complex entries of a partial slot.
__host__ __device__ constexpr int part_rows(int M) { return M <= 8 ? 8 : 16; }
__host__ __device__ constexpr int small_block_bytes(int NA) {
  return 2 * ((int)sizeof(Exps) + 2 * kDig * 2 * NA * 2 * kUnitK * 2);
}
__host__ __device__ constexpr int slot_complex(int NA) { return 2 * NA * kRows; }

// One system's contraction as a list of column tiles of CT = 128 / M output
// columns (times parts of NA rows a of the small operand).  For the slice the
// output columns are the c of I(n, c) and the contracted points the m; for its
// adjoint the other way round (the row m of a Sigma cotangent, summed over c).
struct Sys {
  const double* L;
  const double* R;
  const double* Sl;       // operand rows: Sigma^<, Sigma^> (slice) or Ibar^<, Ibar^> (adjoint), [n+1][M][M]
  const double* Sg;
  const double* wbar;     // composite weights (WeightsView)
  const double* band;
  double* out0;           // I^< and I^>, or the cotangents of Sigma^< and Sigma^>
  double* out1;
  uint8_t* small;         // [unit][part][small block]: written by the prep kernel
  double* part;           // partial sums, [tile + CTA - cta0][slot]
  int* status;
  int M, n, CT, cpt;      // chunks per pass over the history: ceil((n + 1) M / 32)
  int parts, tiles;       // parts of a; column tiles x parts
  int upt;                // chunk slots per tile
  int band_w;
  int adj;                // 0: slice, 1: adjoint
  int shift;              // point m of column c is "near" when m > c + shift, else "far"
  uint32_t magic;         // ceil(2^32 / M) (0 for M = 1): x / M without a division
  int cta0;               // first CTA of the launch that takes slots of this system
  long long unit_base;    // first chunk slot of the system in the launch
  long long chunk_base;   // first chunk x part (prep) and first output entry (reduction)
  long long entry_base;
};
struct Head {             // the systems of a launch
  int n_sys;
  long long total;        // chunk slots
  long long chunks, entries;
};

// Geometry of a system (the pointers and bases are the caller's): NA values of a per part.
__host__ __device__ __forceinline__ void set_geometry(Sys& s, int M, int n, int band_w, int adj, int NA) {
  s.M = M;
  s.n = n;
  s.CT = kRows / M;
  s.cpt = (int)(((long long)(n + 1) * M + kChunkK - 1) / kChunkK);
  s.parts = (M + NA - 1) / NA;
  s.tiles = (n + s.CT) / s.CT * s.parts;
  // the far and near passes overlap in at most kOver chunks; the band points of a tile's columns
  s.upt = s.cpt + kOver + ((s.CT - 1 + band_w) * M + kChunkK - 1) / kChunkK + 1;
  s.band_w = band_w;
  s.adj = adj;
  s.shift = adj ? band_w - 1 : -band_w;
  s.magic = M == 1 ? 0u : (uint32_t)((0x100000000ull + (unsigned long long)M - 1) / (unsigned long long)M);
  s.cta0 = 0;
  s.unit_base = s.chunk_base = s.entry_base = 0;
}
// Bytes of the small operands, rounded up to a 256-byte boundary (the partial sums follow).
__host__ __device__ __forceinline__ size_t small_bytes(const Sys& s, int NA) {
  return ((size_t)s.cpt * kChunkUnits * s.parts * small_block_bytes(NA) + 255) / 256 * 256;
}
// Prep items of a system: pairs of chunks x parts.
__host__ __device__ __forceinline__ long long prep_items(const Sys& s) { return (long long)((s.cpt + 1) / 2) * s.parts; }

// x / M for 0 <= x < 2^32 / M
__host__ __device__ __forceinline__ int div_m(int x, int M, uint32_t magic) {
  if (M == 1) return x;
#ifdef __CUDA_ARCH__
  return (int)__umulhi((uint32_t)x, magic);
#else
  return (int)(((uint64_t)(uint32_t)x * magic) >> 32);
#endif
}

enum Class { kFar = 0, kNear = 1, kBand = 2 };

// The walk over the chunk slots of a system.  A column tile's chunks come in
// this order: the far ones (entries with m <= c + shift count), the near ones
// (m > c + shift), and the band of term 2 (its own weights w_{c,m}).  The at most kOver chunks that straddle the
// line between far and near are taken once each way, with the other side's
// entries masked; the remaining slots of a tile are empty.
struct Walk {
  int si, T, part, c0;  // system of the launch, its tile, the tile's part and first column
  int nfar, far_k;      // far chunks and entries
  int first, near_k;    // first near chunk and entry
  int band0, band1;     // entries of the band
  int idx;              // chunk slot of the tile
  int cls;
  int kc, j0, j1;       // chunk of the history and its units [j0, j1) (empty slot: j0 = j1)

  // T, c0 and part are set
  __host__ __device__ __forceinline__ void tile_start(const Sys& s) {
    const int c1 = c0 + s.CT - 1 < s.n ? c0 + s.CT - 1 : s.n;
    const int far_m = c1 + s.shift < s.n ? c1 + s.shift : s.n;          // last far point of the tile
    const int near_m = c0 + s.shift + 1 > 0 ? c0 + s.shift + 1 : 0;     // its first near point
    far_k = far_m < 0 ? 0 : (far_m + 1) * s.M;
    nfar = (far_k + kChunkK - 1) / kChunkK;
    near_k = near_m * s.M;
    first = near_m > s.n ? s.cpt : near_k / kChunkK;
    band0 = s.adj ? c0 * s.M : near_k;
    band1 = s.adj ? far_k : (c1 + 1) * s.M;
  }
  __host__ __device__ __forceinline__ void chunk_start(const Sys& s) {
    const int nnear = s.cpt - first;
    int beg = 0, end = far_k;
    cls = kFar;
    kc = idx;
    if (idx >= nfar) {
      cls = kNear;
      kc = first + idx - nfar;
      beg = near_k;
      end = (s.n + 1) * s.M;
    }
    if (idx >= nfar + nnear) {
      cls = kBand;
      kc = band0 / kChunkK + idx - nfar - nnear;
      beg = band0;
      end = band1;
    }
    const int lo = beg - kc * kChunkK, hi = end - kc * kChunkK;
    j0 = lo > 0 ? lo / kUnitK : 0;
    j1 = hi > 0 ? (hi + kUnitK - 1) / kUnitK : 0;
    if (j1 > kChunkUnits) j1 = kChunkUnits;
    if (j1 < j0) j1 = j0;
  }
};
__host__ __device__ __forceinline__ void walk_to(Walk& w, const Sys& s, int i, long long slot) {
  w.si = i;
  w.T = (int)(slot / s.upt);
  w.idx = (int)(slot - (long long)w.T * s.upt);
  const int ct = w.T / s.parts;
  w.part = w.T - ct * s.parts;
  w.c0 = ct * s.CT;
  w.tile_start(s);
  w.chunk_start(s);
}
// The next slot; 1: of another tile, 2: past the system's last tile (the
// caller moves to the next system, if any).
__host__ __device__ __forceinline__ int walk_next(Walk& w, const Sys& s) {
  int moved = 0;
  if (++w.idx == s.upt) {
    w.idx = 0;
    if (++w.T == s.tiles) return 2;
    if (++w.part == s.parts) {
      w.part = 0;
      w.c0 += s.CT;
    }
    w.tile_start(s);
    moved = 1;
  }
  w.chunk_start(s);
  return moved;
}

// Chunk slots [range_lo(i), range_lo(i + 1)) of CTA i of G over `total` slots.
__host__ __device__ __forceinline__ long long range_lo(long long total, int G, int i) { return total * i / G; }
// First CTA whose range ends beyond slot q (0 <= q < total).
__host__ __device__ __forceinline__ int cta_of(long long total, int G, long long q) {
  int i = (int)(q * G / total);
  while (i > 0 && range_lo(total, G, i) > q) --i;
  while (range_lo(total, G, i + 1) <= q) ++i;
  return i;
}

// Biased exponent field of the high word of a double.
__host__ __device__ __forceinline__ int field_of(uint32_t hi) { return (int)((hi >> 20) & 0x7FFu); }

// Digits of v for exponent field E (every |v| < 2^(E - 1022)), as the bytes
// d_i + 128 of a 64-bit word, d_0 on top.  Values more than 2^62 below the
// exponent give 0 (so zeros and subnormals need E >= 63).
__host__ __device__ __forceinline__ uint64_t digit_bytes_at(uint32_t hi, uint32_t lo, int t) {  // t = E - field
  t = t < 63 ? t : 63;
  const uint64_t m = ((uint64_t)((hi & 0xFFFFFu) | 0x100000u) << 32) | lo;
  const uint64_t V = (m << 9) >> t;
  const uint64_t sg = (uint64_t)((int64_t)(int32_t)hi >> 31);  // 0 or all ones
  return (V ^ sg) + 0x8080808080808080ull - sg;
}
__host__ __device__ __forceinline__ uint64_t digit_bytes(uint32_t hi, uint32_t lo, int E) {
  return digit_bytes_at(hi, lo, E - field_of(hi));
}

}  // namespace fx
}  // namespace kbe
