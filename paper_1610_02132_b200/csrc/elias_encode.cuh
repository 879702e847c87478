// What the encoders of Elias messages share (elias_encode.cu: the general pipeline, elias_encode_small.cu: problems
// of a few tiles): the workspace, code lengths and code words, where a CTA's run of strings begins, bit writers.
#pragma once

#include "elias_common.cuh"

namespace qsgd {
namespace elias {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;

// CTAs of the length kernel whose sums are also added up together, so that a CTA of the scatter kernel finds its run's start
// and the payload's length by at most one load per group and per CTA of its own group. Beyond kManyCtas CTAs the sums of as many
// groups are added up once more: without them every CTA reads all groups, up to 128 KB in each of a million (n = 2^32, d = 2080,
// s = 16, dense code 103 -> 32 ms; 2^28 2.10 -> 1.97).
constexpr uint32_t kSumGroup = 64;
constexpr uint32_t kManyCtas = 4u * kSumGroup * kSumGroup;
__host__ __device__ inline uint32_t sum_groups(uint32_t ctas) { return (ctas + kSumGroup - 1u) / kSumGroup; }
// Words of the groups' sums and, behind them, of the groups' groups.
__host__ __device__ inline uint32_t sum_words(uint32_t ctas) {
  return sum_groups(ctas) + (ctas > kManyCtas ? sum_groups(sum_groups(ctas)) : 0u);
}

struct Teams {
  uint32_t lpb;               // lanes per bucket (power of two, <= 32)
  uint32_t seg;               // coordinates per lane
  uint32_t nbc;               // buckets per CTA
};

// Lanes get whole blocks of 64 coordinates, so that their ranges begin on word boundaries; where d is no power of two
// the last lanes of a team have less or nothing.
inline Teams make_teams(uint32_t d) {
  Teams t;
  t.lpb = 1;
  while (t.lpb < 32u && t.lpb * 64u < d) t.lpb <<= 1;
  t.seg = ((d + t.lpb - 1u) / t.lpb + 63u) & ~63u;
  t.nbc = kWarps * (32 / t.lpb);
  return t;
}

struct EliasWs {
  uint8_t* fixed;             // fixed-width intermediate
  uint32_t* len;              // L_b
  uint32_t* lane_rec;         // per lane of every bucket team: its bits | (previous nonzero + 1) << 16
  uint32_t* cta_sums;         // per scatter CTA: sum of its buckets' lengths
  uint64_t* group_sums;       // the same per group of CTAs, and per group of groups (sum_words)
  uint32_t* tile_sums;        // the same per tile, and per group of tiles: where len, lane_rec and the sums of the CTAs, which
  uint64_t* tile_groups;      // tiles do without, would be
  size_t bytes;
};

constexpr uint32_t kTileCoords = 16u * kThreads;      // a tile: whole buckets, at most this many coordinates
inline uint32_t tile_buckets(uint32_t d) { return kTileCoords / d; }

// Quantizing and measuring in one kernel: at most kSmallTiles tiles, whose lengths every CTA of the scatter kernel
// adds up.
constexpr uint32_t kSmallTiles = 1000;

// Beyond them, and with a bucket map: by teams (a lane walks 64 coordinates or more: less work per coordinate) or by tiles (a thread
// has 16: shorter walks, less staging per CTA, so more of them resident)? Whole encodes measured both ways, teams against tiles (us).
// Levels above 15, where a symbol costs most. Code'_s: 97 / 70 at n = 17 M, d = 4096, s = 64, 58 / 44 at 8 M, s = 255. Code_s, 4200
// encodes of 3 to 120 M: tiles take 0.8 to 0.99 of the speed of teams on average up to d = 3328 from 8 M on (61 M, d = 512, s = 22, a
// mixture of two scales 190 / 254; 76 M, d = 1024 248 / 325), 1.02 to 1.37 of it at d = 3584 to 4096, where a lane walks 128
// coordinates and a tile is nearly full. Levels up to 15: Code'_s 191 / 239 at 67 M, d = 1024, s = 3 and 60 / 69 at 17 M, d = 128,
// s = 15; Code_s 142 / 204 at 60 M, d = 512, s = 15. Up to 1000 tiles always by tiles: teams do not fill the GPU.
inline bool use_tiles(uint64_t n, uint32_t d, uint32_t s, bool dense) {
  return n <= kSmallTiles * 4096ull || (s > 15u && (dense || d >= 3584u));
}
inline bool use_small(uint64_t n, uint32_t d, const BucketMap& map) {
  return !map.src && n <= kSmallTiles * (uint64_t)(tile_buckets(d) * d);
}

inline EliasWs carve(uint8_t* ws, uint64_t n, uint32_t d, uint32_t s) {
  const FixedLayout L = make_fixed_layout(n, d, s);
  const Teams tm = make_teams(d);
  EliasWs w;
  size_t o = 0;
  w.fixed = ws + o; o += align16(L.total);
  w.len = reinterpret_cast<uint32_t*>(ws + o); o += align16(4 * L.B);
  w.lane_rec = reinterpret_cast<uint32_t*>(ws + o); o += align16(4 * L.B * tm.lpb);
  const uint64_t ctas = (L.B + tm.nbc - 1) / tm.nbc;
  w.cta_sums = reinterpret_cast<uint32_t*>(ws + o);
  w.group_sums = reinterpret_cast<uint64_t*>(ws + o + ((4 * ctas + 7) & ~7ull)); o += align16(8 * (ctas + 1));
  w.tile_sums = w.len;        // at most B of them
  w.tile_groups = reinterpret_cast<uint64_t*>(w.cta_sums);     // at most 8 tiles to a scatter CTA: fewer words than CTAs
  o += 32;                    // (the size that callers reckon with)
  w.bytes = o;
  return w;
}

// Code table indexed by the bit length m of the integer (1 .. 16), kept in shared memory so that
// lanes with different m read it without divergence:
//   bits 0..7 prefix value P(m), bits 8..15 total code length, bit 17 set for m = 1 (whose code is
//   the single bit 0: the generic formula would leave a 1 in bit 1, this bit removes it).
__device__ __forceinline__ void fill_code_table(uint32_t* tab) {
  const uint32_t m = threadIdx.x;
  if (m < 17) {
    uint32_t pv = 0;
    if (m > 8) pv = (3u << 4) | (m - 1u);
    else if (m > 4) pv = (2u << 3) | (m - 1u);
    else if (m > 2) pv = m - 1u;
    const uint32_t len = m <= 1 ? 1u : m + 1u + elias_prefix_len(m);
    tab[m] = pv | (len << 8) | (m == 1 ? (2u << 16) : 0u);
  }
}

__device__ __forceinline__ uint32_t bit_length(uint32_t k) { return 32u - (uint32_t)__clz((int)k); }

// |Elias(k)| from the table.
__device__ __forceinline__ uint32_t tab_len(const uint32_t* tab, uint32_t k) {
  return (tab[bit_length(k)] >> 8) & 0xFFu;
}

// Elias(k), right-aligned; *len receives its length.
__device__ __forceinline__ uint32_t tab_code(const uint32_t* tab, uint32_t k, uint32_t* len) {
  const uint32_t m = bit_length(k);
  const uint32_t e = tab[m];
  *len = (e >> 8) & 0xFFu;
  return ((((e & 0xFFu) << m) | k) << 1) ^ (e >> 16);
}

// Bit j of the result is set iff field j of the level word is nonzero (32 / LB fields).
template <int LB>
__device__ __forceinline__ uint32_t nonzero_mask(uint32_t w) {
  if (LB == 1) return w;
  if (LB == 2) {
    uint32_t y = (w | (w >> 1)) & 0x55555555u;
    y = (y | (y >> 1)) & 0x33333333u;
    y = (y | (y >> 2)) & 0x0F0F0F0Fu;
    y = (y | (y >> 4)) & 0x00FF00FFu;
    return (y | (y >> 8)) & 0xFFFFu;
  }
  if (LB == 4) {
    uint32_t y = w | (w >> 1);
    y = (y | (y >> 2)) & 0x11111111u;
    y = (y | (y >> 3)) & 0x03030303u;
    y = (y | (y >> 6)) & 0x000F000Fu;
    return (y | (y >> 12)) & 0xFFu;
  }
  uint32_t y = w | (w >> 4);
  y |= y >> 2;
  y = (y | (y >> 1)) & 0x01010101u;
  y = (y | (y >> 7)) & 0x00030003u;
  return (y | (y >> 14)) & 0xFu;
}

struct LaneSummary {
  uint32_t bits;      // bits of this lane's codes, excluding the gap code of its first nonzero
  int32_t first;      // first nonzero position in the lane's range, -1 if none
  int32_t last;       // last nonzero position, -1 if none
};

// `bits` plus the sum over the nonzero fields of one level word of 1 + |Elias(level)| (sign bit and level code),
// without a loop: |Elias(level)| grows by 1, 2, 3, 1, 4, 1, 1, 1 when the level reaches 1, 2, 4, 8,
// 16, 32, 64, 128 (Appendix A.2 lengths 1, 3, 6, 7, 11, 12, 13, 14), so the per-field sum is a weighted
// count of "level >= 2^j" masks, added up across the fields of the word.
template <int LB>
__device__ __forceinline__ uint32_t add_level_code_bits(uint32_t w, uint32_t bits) {
  if (LB == 1) return bits + 2u * (uint32_t)__popc(w);
  if (LB == 2) {
    const uint32_t b1 = (w >> 1) & 0x55555555u;
    return bits + 2u * (uint32_t)(__popc(b1 | (w & 0x55555555u)) + __popc(b1));
  }
  if (LB == 4) {
    const uint32_t t3 = w >> 3;
    const uint32_t ge8 = t3 & 0x11111111u;
    const uint32_t ge4 = (t3 | (w >> 2)) & 0x11111111u;
    const uint32_t ge2 = (ge4 | (w >> 1)) & 0x11111111u;
    const uint32_t ge1 = (ge2 | w) & 0x11111111u;
    const uint32_t x = ge8 + 3u * ge4 + 2u * (ge1 + ge2);              // at most 8 per nibble
    return __dp4a((x & 0x0F0F0F0Fu) + ((x >> 4) & 0x0F0F0F0Fu), 0x01010101u, bits);
  }
  const uint32_t ge128 = (w >> 7) & 0x01010101u;
  const uint32_t ge64 = (ge128 | (w >> 6)) & 0x01010101u;
  const uint32_t ge32 = (ge64 | (w >> 5)) & 0x01010101u;
  const uint32_t ge16 = (ge32 | (w >> 4)) & 0x01010101u;
  const uint32_t ge8 = (ge16 | (w >> 3)) & 0x01010101u;
  const uint32_t ge4 = (ge8 | (w >> 2)) & 0x01010101u;
  const uint32_t ge2 = (ge4 | (w >> 1)) & 0x01010101u;
  const uint32_t ge1 = (ge2 | w) & 0x01010101u;
  return __dp4a(2u * (ge1 + ge2) + 3u * ge4 + ge8 + 4u * ge16 + ge32 + ge64 + ge128, 0x01010101u, bits);   // at most 15 per byte
}

// 1 + |Elias(level + 1)| of the dense code's symbols.
template <int LB> struct SymbolLengths { uint8_t of[1u << LB]; };
template <int LB>
__device__ __forceinline__ void fill_symbol_lengths(SymbolLengths<LB>& t) {
  for (uint32_t l = threadIdx.x; l < (1u << LB); l += kThreads) {
    const uint32_t m = 32u - (uint32_t)__clz((int)(l + 1u));
    t.of[l] = (uint8_t)(m <= 1u ? 2u : m + 2u + elias_prefix_len(m));
  }
}
// ... summed over the fields of one level word.
template <int LB>
__device__ __forceinline__ uint32_t symbol_bits(const SymbolLengths<LB>& t, uint32_t w, uint32_t count) {
  constexpr uint32_t kFields = 32u / LB, kMask = (1u << LB) - 1u;
  if constexpr (LB == 1) {                                // two bits, or four
    const uint32_t there = count >= 32u ? 0xFFFFFFFFu : (1u << count) - 1u;
    return 2u * min(count, 32u) + 2u * (uint32_t)__popc(w & there);
  } else {
    uint32_t bits = 0;
#pragma unroll
    for (uint32_t f = 0; f < kFields; ++f) {
      const uint32_t l = t.of[(w >> (f * LB)) & kMask];
      bits += f < count ? l : 0u;
    }
    return bits;
  }
}

// Sum of |Elias(gap)| over the set bits of a 64-coordinate block except the lowest, gap = distance to
// the previous set bit, without a loop: P = "some set bit lies 1 .. 2^b - 1 positions below" is built
// by doubling, and the set bits whose gap has bit length b are those in P_b but not in P_(b-1).
__device__ __forceinline__ uint32_t gap_code_bits(unsigned long long m) {
  unsigned long long prev = 0ull, P = m << 1;
  uint32_t bits = (uint32_t)__popcll(m & P);                            // gap 1: code "0"
  prev = P; P = P | (m << 2) | (P << 2);
  bits += 3u * (uint32_t)__popcll(m & P & ~prev);                       // gaps 2 .. 3
  prev = P; P = P | (m << 4) | (P << 4);
  bits += 6u * (uint32_t)__popcll(m & P & ~prev);                       // gaps 4 .. 7
  prev = P; P = P | (m << 8) | (P << 8);
  bits += 7u * (uint32_t)__popcll(m & P & ~prev);                       // gaps 8 .. 15
  prev = P; P = P | (m << 16) | (P << 16);
  bits += 11u * (uint32_t)__popcll(m & P & ~prev);                      // gaps 16 .. 31
  prev = P; P = P | (m << 32) | (P << 32);
  bits += 12u * (uint32_t)__popcll(m & P & ~prev);                      // gaps 32 .. 63
  return bits;
}

// The same for the 16 coordinates of a small problem's thread: gaps of at most 15.
__device__ __forceinline__ uint32_t gap_code_bits16(uint32_t m) {
  uint32_t prev = 0u, P = m << 1;
  uint32_t bits = (uint32_t)__popc(m & P);
  prev = P; P = P | (m << 2) | (P << 2);
  bits += 3u * (uint32_t)__popc(m & P & ~prev);
  prev = P; P = P | (m << 4) | (P << 4);
  bits += 6u * (uint32_t)__popc(m & P & ~prev);
  prev = P; P = P | (m << 8) | (P << 8);
  return bits + 7u * (uint32_t)__popc(m & P & ~prev);
}

// The lanes' ranges are multiples of 64 coordinates, so every level word this lane reads holds only its
// own coordinates (or, in the last bucket, coordinates past the end of the vector).
template <int LB>
__device__ __forceinline__ LaneSummary summarize_sparse(const uint32_t* tab, const uint32_t* __restrict__ lwb,
                                                        uint32_t c_lo, uint32_t c_hi) {
  // Blocks of 64 coordinates, no loop over the nonzeros: code lengths come from counting. Fields
  // past the end of the vector are zero in the fixed-width layout, so a ragged c_hi needs no mask
  // beyond not reading words that start past it.
  LaneSummary s{0u, -1, -1};
  constexpr uint32_t kFields = 32u / LB;
  for (uint32_t c0 = c_lo; c0 < c_hi; c0 += 64u) {
    const uint32_t* wp = lwb + ((c0 * LB) >> 5);
    unsigned long long m = 0ull;
    uint32_t bits = 0;
#pragma unroll
    for (uint32_t j = 0; j < 2u * LB; ++j) {
      const uint32_t w = (c0 + j * kFields < c_hi) ? __ldg(wp + j) : 0u;
      m |= (unsigned long long)nonzero_mask<LB>(w) << (j * kFields);
      bits = add_level_code_bits<LB>(w, bits);
    }
    if (m) {
      const int32_t lowest = (int32_t)c0 + __ffsll((long long)m) - 1;
      if (s.first < 0) s.first = lowest;
      else bits += tab_len(tab, (uint32_t)(lowest - s.last));          // gap across two blocks of this lane
      s.last = (int32_t)c0 + 63 - __clzll((long long)m);
      s.bits += bits + gap_code_bits(m);
    }
  }
  return s;
}

// Fields past the end of the vector are zero in the fixed-width layout but are not coordinates: the count stops at c_hi.
template <int LB>
__device__ __forceinline__ uint32_t summarize_dense(const SymbolLengths<LB>& lengths, const uint32_t* __restrict__ lwb,
                                                    uint32_t c_lo, uint32_t c_hi) {
  uint32_t bits = 0;
  constexpr uint32_t kFields = 32u / LB;
  for (uint32_t c0 = c_lo; c0 < c_hi; c0 += 64u) {
    const uint32_t* wp = lwb + ((c0 * LB) >> 5);
    uint32_t w[2u * LB];
#pragma unroll
    for (uint32_t j = 0; j < 2u * LB; ++j) w[j] = c0 + j * kFields < c_hi ? __ldg(wp + j) : 0u;
    const uint32_t left = c_hi - c0;
    if (left >= 64u) {
#pragma unroll
      for (uint32_t j = 0; j < 2u * LB; ++j) bits += symbol_bits<LB>(lengths, w[j], kFields);
    } else {
#pragma unroll
      for (uint32_t j = 0; j < 2u * LB; ++j) bits += symbol_bits<LB>(lengths, w[j], left > j * kFields ? left - j * kFields : 0u);
    }
  }
  return bits;
}

// Position of the last nonzero in the team's lanes before this one (-1 if none).
__device__ __forceinline__ int32_t prev_nonzero_before_lane(int32_t last, uint32_t tl, uint32_t lpb) {
  int32_t run = last;                           // inclusive max-scan of `last` inside the team
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int32_t t = __shfl_up_sync(0xffffffffu, run, o, 32);
    if ((uint32_t)o < lpb && tl >= (uint32_t)o) run = max(run, t);
  }
  const int32_t excl = __shfl_up_sync(0xffffffffu, run, 1, 32);
  return tl == 0 ? -1 : excl;
}

struct BucketParams {
  const float* A;
  const uint32_t* sign;
  const uint32_t* level;
  uint64_t n;
  uint32_t d;
  uint64_t B;
  uint32_t lpb, seg, nbc;
};

// Bits of this lane's part of its bucket's string (the scale's 32 bits go with team lane 0).
template <int LB, bool DENSE, class Lengths>
__device__ __forceinline__ uint32_t lane_bits(const uint32_t* tab, const Lengths& lengths, const uint32_t* __restrict__ lwb, uint32_t lpb,
                                              uint32_t c_lo, uint32_t c_hi, uint32_t tl, bool live,
                                              int32_t* prev_out) {
  uint32_t bits = 0;
  int32_t prev = -1;
  if constexpr (DENSE) {
    if (live) bits = summarize_dense<LB>(lengths, lwb, c_lo, c_hi);
  } else {
    LaneSummary s{0u, -1, -1};
    if (live) s = summarize_sparse<LB>(tab, lwb, c_lo, c_hi);
    prev = prev_nonzero_before_lane(s.last, tl, lpb);
    bits = s.bits + (s.first >= 0 ? tab_len(tab, (uint32_t)(s.first - prev)) : 0u);
  }
  if (live && tl == 0) bits += 32u;
  *prev_out = prev;
  return bits;
}

// Sum over the lanes of a team (every lane of the team receives it).
__device__ __forceinline__ uint32_t team_sum(uint32_t v, uint32_t lpb) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const uint32_t t = __shfl_xor_sync(0xffffffffu, v, o);
    if ((uint32_t)o < lpb) v += t;
  }
  return v;
}

// Sizes of the whole message: the info words, the capacity check. False: it does not fit, nothing is written.
__device__ __forceinline__ bool fix_geometry(uint64_t total, uint64_t B, size_t out_capacity, uint64_t* out_bits,
                                             uint32_t* status_dev, bool report, uint64_t* payload_bytes) {
  const uint64_t pay = align16((total + 7) / 8), bytes = pay + 8 * (B + 1);
  const bool ok = bytes <= out_capacity;
  if (report && threadIdx.x == 0) {
    out_bits[0] = total; out_bits[1] = pay; out_bits[2] = bytes; out_bits[3] = 0;
    if (!ok) atomicOr(status_dev, QSGD_DEV_CAPACITY);
  }
  *payload_bytes = pay;
  return ok;
}

// By one thread of each CTA of a length kernel: its sum to those of its groups.
__device__ __forceinline__ void add_to_groups(uint64_t* groups, uint32_t sum) {
  atomicAdd(reinterpret_cast<unsigned long long*>(groups) + blockIdx.x / kSumGroup, (unsigned long long)sum);
  if (gridDim.x > kManyCtas)
    atomicAdd(reinterpret_cast<unsigned long long*>(groups) + sum_groups(gridDim.x) + blockIdx.x / (kSumGroup * kSumGroup), (unsigned long long)sum);
}

// By one warp: the first payload bit of this CTA's run, and the payload's length.
__device__ __forceinline__ void find_start(const uint32_t* sums, const uint64_t* groups, uint64_t* start, uint64_t* all) {
  const uint32_t lane = threadIdx.x & 31, mine = blockIdx.x / kSumGroup, count = sum_groups(gridDim.x);
  const bool many = gridDim.x > kManyCtas;
  uint64_t before = 0, total = 0;
  // the coarsest sums, all of them; of the finer ones those in front of this CTA in its own group
  const uint64_t* top = many ? groups + count : groups;
  const uint32_t tops = many ? sum_groups(count) : count, own = many ? mine / kSumGroup : mine;
  for (uint32_t i = lane; i < tops; i += 32u) {
    const uint64_t v = __ldg(top + i);
    total += v;
    before += i < own ? v : 0ull;
  }
  if (many)
    for (uint32_t i = own * kSumGroup + lane; i < mine; i += 32u) before += __ldg(groups + i);
  for (uint32_t i = mine * kSumGroup + lane; i < blockIdx.x; i += 32u) before += __ldg(sums + i);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    before += __shfl_xor_sync(0xffffffffu, before, o);
    total += __shfl_xor_sync(0xffffffffu, total, o);
  }
  if (lane == 0) { *start = before; *all = total; }
}

// Whole code words of what is met most, their bits from bit 31 down and their length in bits 0 .. 4: sign and level (entry
// level | negative << LB), and gaps below 64. At most 27 bits together.
template <int LB, bool DENSE>
struct CodeWords {
  uint32_t level[2u << LB];
  uint32_t gap[DENSE ? 1 : 64];
};
template <int LB, bool DENSE>
__device__ __forceinline__ void fill_code_words(CodeWords<LB, DENSE>& words) {
  constexpr uint32_t kLevels = 2u << LB, kMask = (1u << LB) - 1u;
  for (uint32_t k = threadIdx.x; k < kLevels + (DENSE ? 0u : 64u); k += kThreads) {
    const bool is_level = k < kLevels;
    const uint32_t v = is_level ? (k & kMask) + (DENSE ? 1u : 0u) : k - kLevels;
    uint32_t ln = 0, code = v ? elias_code(v, &ln) : 0u;
    if (is_level && v) { code |= (k >> LB) << ln; ++ln; }
    const uint32_t e = v ? code << (32u - ln) | ln : 0u;
    if (is_level) words.level[k] = e;
    else words.gap[k - kLevels] = e;
  }
}

// Lane-private writer into the CTA's staging words in shared memory: the bits of the word at `at` gather in `acc`.
struct StageWriter {
  uint32_t at, acc, n;
  __device__ __forceinline__ void begin(uint32_t* words, uint32_t start_bit) {
    at = (uint32_t)__cvta_generic_to_shared(words) + (start_bit >> 5) * 4u; acc = 0u; n = start_bit & 31u;
  }
  // `len` <= 31 bits from bit 31 of c down; below them c is zero
  __device__ __forceinline__ void put(uint32_t c, uint32_t len) {
    acc |= c >> n;
    n += len;
    if (n >= 32u) {
      asm volatile("red.shared.or.b32 [%0], %1;" ::"r"(at), "r"(acc) : "memory");
      at += 4u;
      n -= 32u;
      acc = c << (len - n);
    }
  }
  // The same without a branch, for lanes that put one symbol after the other and come to a word's end at different times.
  __device__ __forceinline__ void put_even(uint32_t c, uint32_t len) {
    acc |= c >> n;
    n += len;
    asm volatile("{\n\t.reg .pred p;\n\t.reg .u32 t;\n\tsetp.ge.u32 p, %2, 32;\n\t@p red.shared.or.b32 [%0], %1;\n\t@p add.u32 %0, %0, 4;\n\t"
                 "and.b32 %2, %2, 31;\n\tsub.u32 t, %4, %2;\n\t@p shl.b32 %1, %3, t;\n\t}"
                 : "+r"(at), "+r"(acc), "+r"(n) : "r"(c), "r"(len) : "memory");
  }
  __device__ __forceinline__ void put_word(uint32_t c) {
    asm volatile("red.shared.or.b32 [%0], %1;" ::"r"(at), "r"(acc | c >> n) : "memory");
    at += 4u;
    acc = __funnelshift_l(0u, c, 32u - n) & (n ? 0xFFFFFFFFu : 0u);
  }
  __device__ __forceinline__ void finish() {
    if (n) asm volatile("red.shared.or.b32 [%0], %1;" ::"r"(at), "r"(acc) : "memory");
  }
};

// One nonzero: gap, then sign and level (entry `idx` of words.level), in one piece but for gaps from 64 on, whose code goes ahead.
template <int LB>
__device__ __forceinline__ void put_entry(StageWriter& bw, const uint32_t* tab, const CodeWords<LB, false>& words, uint32_t gap, uint32_t idx) {
  if (gap >= 64u) {
    uint32_t gl;
    const uint32_t gcode = tab_code(tab, gap, &gl);
    bw.put(gcode << (32u - gl), gl);
    gap = 0u;                                            // nothing of it is left
  }
  const uint32_t l = words.level[idx], g = words.gap[gap];
  bw.put((g & ~31u) | __funnelshift_r(l & ~31u, 0u, g), (g + l) & 31u);
}

inline uint32_t host_elias_len(uint32_t k) {
  uint32_t len = 1;
  while (k > 1) {
    uint32_t m = 0;
    for (uint32_t t = k; t; t >>= 1) ++m;
    len += m;
    k = m - 1;
  }
  return len;
}

// Staging: the longest strings that the fields of a CTA's buckets can make, plus the shared lead-in word.
template <bool DENSE>
inline size_t stage_bytes(uint32_t buckets, uint32_t d, uint32_t s) {
  const uint32_t most = (1u << level_bits_for(s)) - 1u;
  const uint32_t per = DENSE ? 1 + host_elias_len(most + 1) : 2 + host_elias_len(most);
  const size_t run_bits = (size_t)buckets * (32 + (size_t)d * per);
  return ((run_bits + 31) / 32 + 4) * 4;
}

// ---- tiles: 16 coordinates a thread ------------------------------------------------------------------
// The team kernels give a lane 64 coordinates or more, which is what makes them cheap per coordinate; on a
// problem that does not fill the GPU their time is that serial walk (13 to 22 us of scatter whatever n up
// to 10^6). Here a thread takes 16 coordinates, a CTA a tile of whole buckets of at most 4096
// coordinates, and what a lane needs of its predecessors (the last nonzero of its bucket, the bits in
// front of it) comes from scans over the CTA. Three times the instructions per coordinate of a sparse
// bucket, a quarter of the chain.

// What one thread holds of its 16 coordinates.
template <int LB>
struct Piece {
  static constexpr int kWords = LB == 8 ? 4 : LB == 4 ? 2 : 1;
  uint32_t level[kWords];     // 16 fields of LB bits
  uint32_t sign;              // 16 bits
  uint32_t c0;                // position of the first in its bucket
  uint32_t bucket;            // bucket in the tile
  uint32_t count;             // coordinates that exist: 0 .. 16
};

template <int LB>
__device__ __forceinline__ uint32_t piece_level(const Piece<LB>& q, uint32_t j) {   // j is a constant after unrolling
  return (q.level[(j * LB) >> 5] >> ((j * LB) & 31u)) & ((1u << LB) - 1u);
}

// Piece of this thread in tile blockIdx.x, from the fixed-width fields; with plain loads, since they may have
// been written by this very kernel.
template <int LB>
__device__ __forceinline__ Piece<LB> load_piece(const BucketParams& p) {
  Piece<LB> q;
  const uint32_t local = threadIdx.x * 16u;               // first coordinate in the tile
  const uint32_t tile = p.nbc * p.d;
  const uint64_t i0 = (uint64_t)blockIdx.x * tile + local;
  q.bucket = local / p.d;
  q.c0 = local - q.bucket * p.d;
  q.count = local < tile && i0 < p.n ? (uint32_t)min((uint64_t)16u, p.n - i0) : 0u;
  q.sign = 0u;
#pragma unroll
  for (int j = 0; j < Piece<LB>::kWords; ++j) q.level[j] = 0u;
  if (q.count) {                                          // fields past the end of the vector are zero
    const uint64_t slot = i0 >> 4;
    q.sign = reinterpret_cast<const uint16_t*>(p.sign)[slot];
    if (LB == 8) {
      const uint4 w = reinterpret_cast<const uint4*>(p.level)[slot];
      q.level[0] = w.x; q.level[1] = w.y; q.level[2] = w.z; q.level[3] = w.w;
    } else if (LB == 4) {
      const uint2 w = reinterpret_cast<const uint2*>(p.level)[slot];
      q.level[0] = w.x; q.level[1] = w.y;
    } else if (LB == 2) {
      q.level[0] = p.level[slot];
    } else {
      q.level[0] = reinterpret_cast<const uint16_t*>(p.level)[slot];
    }
  }
  return q;
}

// Bit j: level j is nonzero.
template <int LB>
__device__ __forceinline__ uint32_t piece_mask(const Piece<LB>& q) {
  uint32_t m = 0;
#pragma unroll
  for (int j = 0; j < Piece<LB>::kWords; ++j) m |= nonzero_mask<LB>(q.level[j]) << (j * (32 / LB));
  return m;
}

// Scans over the CTA, one barrier each: the largest key, or the sum, in front of this thread (0 for the
// first).
__device__ __forceinline__ uint32_t cta_max_before(uint32_t key, uint32_t* warp_slots) {
  const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t t = __shfl_up_sync(0xffffffffu, key, o);
    if (lane >= (uint32_t)o) key = max(key, t);
  }
  if (lane == 31) warp_slots[warp] = key;
  __syncthreads();
  uint32_t before = __shfl_up_sync(0xffffffffu, key, 1);
  if (lane == 0) before = 0u;
#pragma unroll
  for (int w = 0; w < kWarps; ++w)
    if ((uint32_t)w < warp) before = max(before, warp_slots[w]);
  return before;
}
__device__ __forceinline__ uint32_t cta_sum_before(uint32_t v, uint32_t* warp_slots, uint32_t* total) {
  const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t inc = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t t = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= (uint32_t)o) inc += t;
  }
  if (lane == 31) warp_slots[warp] = inc;
  __syncthreads();
  uint32_t before = inc - v, all = 0;
#pragma unroll
  for (int w = 0; w < kWarps; ++w) {
    if ((uint32_t)w < warp) before += warp_slots[w];
    all += warp_slots[w];
  }
  *total = all;
  return before;
}

// Last nonzero of the piece's bucket in front of the piece (-1: none). One CTA barrier.
template <int LB>
__device__ __forceinline__ int32_t nonzero_before(const Piece<LB>& q, uint32_t mask, uint32_t* warp_slots) {
  // bucket number above position + 1: the largest key in front is the nearest nonzero, if of this bucket
  const uint32_t at = mask ? q.c0 + 32u - (uint32_t)__clz((int)mask) : 0u;
  const uint32_t before = cta_max_before((q.bucket + 1u) << 13 | at, warp_slots);
  return before >> 13 == q.bucket + 1u ? (int32_t)(before & 8191u) - 1 : -1;
}

// Bits of the piece's part of its bucket's string (with the scale's 32 where the bucket starts).
template <int LB, bool DENSE, class Lengths>
__device__ __forceinline__ uint32_t piece_bits(const uint32_t* tab, const Lengths& lengths, const Piece<LB>& q, uint32_t mask, int32_t prev) {
  uint32_t bits = q.count && q.c0 == 0u ? 32u : 0u;
  if constexpr (DENSE) {
    constexpr uint32_t kFields = LB == 1 ? 16u : 32u / LB;
#pragma unroll
    for (uint32_t j = 0; j < Piece<LB>::kWords; ++j)
      bits += symbol_bits<LB>(lengths, q.level[j], q.count > j * kFields ? q.count - j * kFields : 0u);
    return bits;
  }
  if (mask) {
#pragma unroll
    for (int j = 0; j < Piece<LB>::kWords; ++j) bits = add_level_code_bits<LB>(q.level[j], bits);
    bits += gap_code_bits16(mask);
    bits += tab_len(tab, q.c0 + (uint32_t)__ffs((int)mask) - 1u - (uint32_t)prev);
  }
  return bits;
}

// Assembles the piece's codes at bit `bit` of the CTA's staging words.
template <int LB, bool DENSE>
__device__ __forceinline__ void emit_piece(const uint32_t* tab, const CodeWords<LB, DENSE>& words, uint32_t* stage, uint32_t bit,
                                           const Piece<LB>& q, uint32_t mask, int32_t prev, float A) {
  constexpr uint32_t kMask = (1u << LB) - 1u;
  StageWriter bw;
  bw.begin(stage, bit);
  if (q.c0 == 0u) bw.put_word(__float_as_uint(A));
  if constexpr (DENSE) {
#pragma unroll
    for (uint32_t j = 0; j < 16; ++j) {
      const uint32_t e = j < q.count ? words.level[piece_level<LB>(q, j) | ((q.sign >> j) & 1u) << LB] : 0u;
      bw.put_even(e & ~31u, e & 31u);
    }
  } else {
    while (mask) {                                 // once per nonzero of the busiest lane
      const uint32_t j = (uint32_t)__ffs((int)mask) - 1u;
      mask &= mask - 1u;
      const uint32_t pos = q.c0 + j;
      uint32_t w = q.level[0];
      if (LB == 8) {
        const uint32_t lo = j & 4u ? q.level[1 % Piece<LB>::kWords] : q.level[0];
        const uint32_t hi = j & 4u ? q.level[3 % Piece<LB>::kWords] : q.level[2 % Piece<LB>::kWords];
        w = j & 8u ? hi : lo;
      } else if (LB == 4) {
        w = j & 8u ? q.level[1 % Piece<LB>::kWords] : q.level[0];
      }
      put_entry<LB>(bw, tab, words, pos - (uint32_t)prev, (__funnelshift_r(w, 0u, LB * j) & kMask) | ((q.sign >> j) & 1u) << LB);
      prev = (int32_t)pos;
    }
  }
  bw.finish();
}

// Flushes a CTA's run of strings, assembled in `stage` from bit `lead` of the first word on, to the payload words
// gw[0 ..]. Every word is stored once and whole: a word that two runs share is the first one's, which knows
// what follows -- the next run begins with the 32 bits of its first bucket's scale. The last run clears the
// padding behind it.
__device__ __forceinline__ void flush_run(uint32_t* __restrict__ gw, const uint32_t* stage, uint32_t lead, uint32_t span,
                                          bool last_run, const float* next_scale, uint32_t words_left) {
  const uint32_t nwords = (lead + span + 31u) >> 5, r = (lead + span) & 31u;
  for (uint32_t j = threadIdx.x + (lead ? 1u : 0u); j < nwords; j += kThreads) {
    uint32_t v = stage[j];
    if (j == nwords - 1u && r && !last_run) v |= __float_as_uint(*next_scale) >> r;
    gw[j] = v;
  }
  if (last_run)
    for (uint32_t j = nwords + threadIdx.x; j < words_left; j += kThreads) gw[j] = 0u;
}

// elias_encode_small.cu
int launch_tile_scatter(const BucketParams& bp, const EliasWs& w, uint32_t s, bool dense, uint8_t* out, size_t out_capacity,
                        uint64_t* out_bits, uint32_t* status_dev, cudaStream_t stream);
int launch_elias_encode_small(const float* g, uint64_t n, uint32_t d, uint32_t s, int norm_kind, bool dense, uint64_t seed,
                              uint32_t step, uint32_t worker, uint8_t* out, size_t out_capacity, uint64_t* out_bits,
                              const EliasWs& w, uint32_t* status_dev, cudaStream_t stream);

}  // namespace elias
}  // namespace qsgd
