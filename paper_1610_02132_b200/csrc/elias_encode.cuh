// What the encoders of Elias messages share (elias_encode.cu: the general pipeline, elias_encode_small.cu: problems
// of a few tiles): the workspace, code lengths and code words, the scan of the CTAs' lengths, bit writers.
#pragma once

#include "elias_common.cuh"

namespace qsgd {
namespace elias {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;

struct Ctrl {                 // control block at the end of the workspace
  uint64_t total_bits;
  uint64_t payload_bytes;
  uint32_t ok;                // 1 when the message fits out_capacity
  uint32_t arrived;           // CTAs of the length kernel that have published their sum
};

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
  uint64_t* cta_sums;         // per scatter CTA: sum of its buckets' lengths, then exclusive prefix
  uint64_t* tile_sums;        // the same per tile, where len and lane_rec, which tiles do without, would be
  Ctrl* ctrl;
  size_t bytes;
};

constexpr uint32_t kTileCoords = 16u * kThreads;      // a tile: whole buckets, at most this many coordinates
inline uint32_t tile_buckets(uint32_t d) { return kTileCoords / d; }

// Quantizing and measuring in one kernel: at most kSmallTiles tiles, whose lengths every CTA of the scatter kernel
// adds up.
constexpr uint32_t kSmallTiles = 1000;

// By teams (a lane walks 64 coordinates or more: less work per coordinate) or by tiles (a thread has 16: done
// sooner)? Whole encodes measured both ways on three input families, teams against tiles (us). Tiles in two kernels:
// 20.4 / 8.8 at n = 2^20, 18.5 to 26.4 / 17.5 to 21.9 at 3 * 2^20, 20.2 to 28.0 / 20.6 to 26.5 at 1000 tiles
// (d = 512, s = 15); beyond 1000 tiles, where they take three kernels, only for levels above 15: Code_s up to
// 6 * 2^20 coordinates 0.43 to 1.17 of the time by teams, Code'_s with d > 1024 (128 coordinates a lane) up to 20 * 2^20
// 0.66 to 1.15. Code'_s with smaller levels, whose symbols cost a lane little, 0.87 to 1.34 from there on (n = 19 M,
// d = 4096, s = 1: 74 / 98).
inline bool use_tiles(uint64_t n, uint32_t d, uint32_t s, bool dense) {
  if (n <= kSmallTiles * 4096ull) return true;
  const uint64_t m = s <= 15u ? 0u : !dense ? 6u : d > 1024u ? 20u : 0u;
  return n <= m << 20;
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
  w.cta_sums = reinterpret_cast<uint64_t*>(ws + o); o += align16(8 * (ctas + 1));
  w.tile_sums = reinterpret_cast<uint64_t*>(w.len);     // tiles + 1 <= B + 1 of them: 4 B bytes of len, at least 4 B of lane_rec, 16 of cta_sums
  w.ctrl = reinterpret_cast<Ctrl*>(ws + o); o += align16(sizeof(Ctrl));
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

// Sum over the nonzero fields of one level word of 1 + |Elias(level)| (sign bit and level code),
// without a loop: |Elias(level)| grows by 1, 2, 3, 1, 4, 1, 1, 1 when the level reaches 1, 2, 4, 8,
// 16, 32, 64, 128 (Appendix A.2 lengths 1, 3, 6, 7, 11, 12, 13, 14), so the per-field sum is a weighted
// count of "level >= 2^j" masks, added up across the fields of the word.
template <int LB>
__device__ __forceinline__ uint32_t level_code_bits(uint32_t w) {
  if (LB == 1) return 2u * (uint32_t)__popc(w);
  if (LB == 2) {
    const uint32_t b1 = (w >> 1) & 0x55555555u;
    return 2u * (uint32_t)(__popc(b1 | (w & 0x55555555u)) + __popc(b1));
  }
  if (LB == 4) {
    const uint32_t t3 = w >> 3;
    const uint32_t ge8 = t3 & 0x11111111u;
    const uint32_t ge4 = (t3 | (w >> 2)) & 0x11111111u;
    const uint32_t ge2 = (ge4 | (w >> 1)) & 0x11111111u;
    const uint32_t ge1 = (ge2 | w) & 0x11111111u;
    const uint32_t x = ge8 + 3u * ge4 + 2u * (ge1 + ge2);              // at most 8 per nibble
    const uint32_t y = (x & 0x0F0F0F0Fu) + ((x >> 4) & 0x0F0F0F0Fu);
    return (y * 0x01010101u) >> 24;
  }
  const uint32_t ge128 = (w >> 7) & 0x01010101u;
  const uint32_t ge64 = (ge128 | (w >> 6)) & 0x01010101u;
  const uint32_t ge32 = (ge64 | (w >> 5)) & 0x01010101u;
  const uint32_t ge16 = (ge32 | (w >> 4)) & 0x01010101u;
  const uint32_t ge8 = (ge16 | (w >> 3)) & 0x01010101u;
  const uint32_t ge4 = (ge8 | (w >> 2)) & 0x01010101u;
  const uint32_t ge2 = (ge4 | (w >> 1)) & 0x01010101u;
  const uint32_t ge1 = (ge2 | w) & 0x01010101u;
  const uint32_t x = 2u * (ge1 + ge2) + 3u * ge4 + ge8 + 4u * ge16 + ge32 + ge64 + ge128;   // at most 15 per byte
  return (x * 0x01010101u) >> 24;
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
      bits += level_code_bits<LB>(w);
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

// Whole level words are loaded once and their fields taken from the register (fields past the end of the
// vector are zero in the fixed-width layout but are not coordinates: the count stops at c_hi).
template <int LB>
__device__ __forceinline__ uint32_t summarize_dense(const uint32_t* tab, const uint32_t* __restrict__ lwb,
                                                    uint32_t c_lo, uint32_t c_hi) {
  uint32_t bits = 0;
  constexpr uint32_t kFields = 32u / LB, kMask = (1u << LB) - 1u;
  for (uint32_t c0 = c_lo; c0 < c_hi; c0 += 64u) {
    const uint32_t* wp = lwb + ((c0 * LB) >> 5);
#pragma unroll
    for (uint32_t j = 0; j < 2u * LB; ++j) {
      const uint32_t cw = c0 + j * kFields;                 // first coordinate of this word
      if (cw >= c_hi) break;
      const uint32_t w = __ldg(wp + j);
      const uint32_t cnt = min(kFields, c_hi - cw);
      if (cnt == kFields) {
#pragma unroll
        for (uint32_t f = 0; f < kFields; ++f) bits += 1u + tab_len(tab, ((w >> (f * LB)) & kMask) + 1u);
      } else {
        for (uint32_t f = 0; f < cnt; ++f) bits += 1u + tab_len(tab, ((w >> (f * LB)) & kMask) + 1u);
      }
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

struct ScanArgs {              // what the last CTA of the length kernel needs for the scan
  uint64_t ctas;
  size_t out_capacity;
  Ctrl* ctrl;
  uint64_t* out_bits;
  uint32_t* status_dev;
};

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
template <int LB, bool DENSE>
__device__ __forceinline__ uint32_t lane_bits(const uint32_t* tab, const uint32_t* __restrict__ lwb, uint32_t lpb,
                                              uint32_t c_lo, uint32_t c_hi, uint32_t tl, bool live,
                                              int32_t* prev_out) {
  uint32_t bits = 0;
  int32_t prev = -1;
  if (DENSE) {
    if (live) bits = summarize_dense<LB>(tab, lwb, c_lo, c_hi);
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

// ---- scan of the per-CTA sums, run by the CTA of the length kernel that finishes last ------------
__device__ __forceinline__ uint64_t block_exclusive_scan(uint64_t v, uint64_t* total) {
  __shared__ uint64_t warp_sums[32];
  const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  uint64_t inc = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint64_t t = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= (uint32_t)o) inc += t;
  }
  if (lane == 31) warp_sums[warp] = inc;
  __syncthreads();
  uint64_t before = 0, all = 0;
  for (uint32_t w = 0; w < nwarps; ++w) {
    const uint64_t t = warp_sums[w];
    if (w < warp) before += t;
    all += t;
  }
  __syncthreads();
  *total = all;
  return before + inc - v;
}

// In place: cta_sums[c] becomes the first payload bit of CTA c's run, cta_sums[ctas] the payload
// length. Also: message geometry and capacity check. Called by all threads of one CTA.
__device__ __forceinline__ void scan_cta_sums(uint64_t* cta_sums, uint64_t ctas, uint64_t B, size_t out_capacity,
                                              Ctrl* ctrl, uint64_t* out_bits, uint32_t* status_dev) {
  // every thread owns a contiguous chunk of the sums: one block-wide scan in total
  const uint64_t chunk = (ctas + blockDim.x - 1) / blockDim.x;
  const uint64_t lo = min((uint64_t)threadIdx.x * chunk, ctas), hi = min(lo + chunk, ctas);
  uint64_t mine = 0;
#pragma unroll 8
  for (uint64_t i = lo; i < hi; ++i) mine += __ldcg(cta_sums + i);
  uint64_t total;
  uint64_t run = block_exclusive_scan(mine, &total);
  if (threadIdx.x == 0) {
    const uint64_t pay = align16((total + 7) / 8);
    const uint64_t total_bytes = pay + 8 * (B + 1);
    const bool ok = total_bytes <= out_capacity;
    ctrl->total_bits = total;
    ctrl->payload_bytes = pay;
    ctrl->ok = ok ? 1u : 0u;
    out_bits[0] = total; out_bits[1] = pay; out_bits[2] = total_bytes; out_bits[3] = 0;
    if (!ok) atomicOr(status_dev, QSGD_DEV_CAPACITY);
    cta_sums[ctas] = total;
  }
#pragma unroll 8
  for (uint64_t i = lo; i < hi; ++i) {
    const uint64_t v = __ldcg(cta_sums + i);
    cta_sums[i] = run;
    run += v;
  }
}

// Whole code words (code | length << 16) of the integers met most: every level, and gaps below 64.
template <int LB>
struct CodeWords {
  uint32_t level[1u << LB];
  uint32_t gap[64];
};
template <int LB>
__device__ __forceinline__ void fill_code_words(CodeWords<LB>& words) {
  for (uint32_t k = threadIdx.x; k < (1u << LB) + 64u; k += kThreads) {
    const uint32_t v = k < (1u << LB) ? k : k - (1u << LB);
    uint32_t ln = 0;
    const uint32_t code = v ? elias_code(v, &ln) : 0u;
    (k < (1u << LB) ? words.level[v] : words.gap[v]) = code | (ln << 16);
  }
}

// Lane-private writer into the CTA's staging words in shared memory.
struct StageWriter {
  uint32_t* words;
  uint32_t widx;
  uint64_t buf;
  uint32_t nbuf;
  __device__ __forceinline__ void begin(uint32_t* w, uint32_t start_bit) {
    words = w; widx = start_bit >> 5; buf = 0; nbuf = start_bit & 31;
  }
  __device__ __forceinline__ void put(uint32_t code, uint32_t len) {   // len in [1, 32]
    buf |= (uint64_t)code << (64 - nbuf - len);
    nbuf += len;
    if (nbuf >= 32) {
      atomicOr(words + widx, (uint32_t)(buf >> 32));
      ++widx; buf <<= 32; nbuf -= 32;
    }
  }
  __device__ __forceinline__ void finish() {
    if (nbuf) atomicOr(words + widx, (uint32_t)(buf >> 32));
  }
};

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

// Staging: the longest legal strings of a CTA's buckets, plus the shared lead-in word.
template <bool DENSE>
inline size_t stage_bytes(uint32_t buckets, uint32_t d, uint32_t s) {
  const uint32_t per = DENSE ? 1 + host_elias_len(s + 1) : 2 + host_elias_len(s);
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
template <int LB, bool DENSE>
__device__ __forceinline__ uint32_t piece_bits(const uint32_t* tab, const Piece<LB>& q, uint32_t mask, int32_t prev) {
  uint32_t bits = q.count && q.c0 == 0u ? 32u : 0u;
  if (DENSE) {
#pragma unroll
    for (uint32_t j = 0; j < 16; ++j)
      if (j < q.count) bits += 1u + tab_len(tab, piece_level<LB>(q, j) + 1u);
    return bits;
  }
  if (mask) {
#pragma unroll
    for (int j = 0; j < Piece<LB>::kWords; ++j) bits += level_code_bits<LB>(q.level[j]);
    bits += gap_code_bits16(mask);
    bits += tab_len(tab, q.c0 + (uint32_t)__ffs((int)mask) - 1u - (uint32_t)prev);
  }
  return bits;
}

// Assembles the piece's codes at bit `bit` of the CTA's staging words.
template <int LB, bool DENSE>
__device__ __forceinline__ void emit_piece(const uint32_t* tab, const CodeWords<LB>& words, uint32_t* stage, uint32_t bit,
                                           const Piece<LB>& q, uint32_t mask, int32_t prev, float A) {
  StageWriter bw;
  bw.begin(stage, bit);
  if (q.c0 == 0u) bw.put(__float_as_uint(A), 32);
  if (DENSE) {
#pragma unroll
    for (uint32_t j = 0; j < 16; ++j) {
      if (j >= q.count) break;
      uint32_t ln;
      const uint32_t code = tab_code(tab, piece_level<LB>(q, j) + 1u, &ln);
      bw.put((((q.sign >> j) & 1u) << ln) | code, ln + 1u);
    }
  } else {
    while (mask) {                                 // once per nonzero of the busiest lane
      const uint32_t j = (uint32_t)__ffs((int)mask) - 1u;
      mask &= mask - 1u;
      const uint32_t pos = q.c0 + j, gap = pos - (uint32_t)prev;
      uint32_t level, gcode, gl;
      if (LB == 8) {
        const uint32_t lo = j & 4u ? q.level[1 % Piece<LB>::kWords] : q.level[0];
        const uint32_t hi = j & 4u ? q.level[3 % Piece<LB>::kWords] : q.level[2 % Piece<LB>::kWords];
        level = ((j & 8u ? hi : lo) >> (8u * (j & 3u))) & 0xFFu;
      } else if (LB == 4) {
        level = (q.level[j >> 3 ? 1 % Piece<LB>::kWords : 0] >> (4u * (j & 7u))) & 15u;
      } else {
        level = (q.level[0] >> (LB * j)) & ((1u << LB) - 1u);
      }
      if (gap < 64u) {
        const uint32_t e = words.gap[gap];
        gcode = e & 0xFFFFu;
        gl = e >> 16;
      } else {
        gcode = tab_code(tab, gap, &gl);
      }
      const uint32_t e = words.level[level], ll = e >> 16;
      const uint32_t lcode = (e & 0xFFFFu) | (((q.sign >> j) & 1u) << ll);
      if (gl + ll + 1u <= 32u) {                   // gap, sign and level in one piece (the rule)
        bw.put((gcode << (ll + 1u)) | lcode, gl + ll + 1u);
      } else {
        bw.put(gcode, gl);
        bw.put(lcode, ll + 1u);
      }
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
int launch_tile_scatter(const BucketParams& bp, const EliasWs& w, uint32_t s, bool dense, uint8_t* out, cudaStream_t stream);
int launch_elias_encode_small(const float* g, uint64_t n, uint32_t d, uint32_t s, int norm_kind, bool dense, uint64_t seed,
                              uint32_t step, uint32_t worker, uint8_t* out, size_t out_capacity, uint64_t* out_bits,
                              const EliasWs& w, uint32_t* status_dev, cudaStream_t stream);

}  // namespace elias
}  // namespace qsgd
