// Decode-and-aggregate, Elias path, for problems with too few strings to give every lane of the GPU one of
// its own: a team of up to 32 lanes shares a string. (Section 3.1 for the string, Appendix A.2 and A.3 for
// the codes, Algorithm 1 for the sum and the step.)
//
// A string can only be read front to back, but a reader that starts at the wrong bit usually falls into
// step with the right one after a few symbols (the self-synchronisation of variable-length codes used for
// parallel Huffman decoding: Weissenberger & Schmidt, ICPP 2018). Lane t of a team owns the t-th part of
// the string's bits. It starts kWarmUp bits ahead of its part, reads up to the first symbol that starts in
// it, then reads its part through, counting positions. Its start is right when it is where lane t - 1
// ended; where it is not, the lane reads its part again from there, and so on until all agree. Lane 0 is
// right from the start and every round makes at least one more lane right, so T rounds always suffice
// (the time of reading the string by one lane); two or three are the rule. (A lane keeps two readings, so that a lane in
// front of it that turns out wrong costs it no third one.) A scan of the counts gives
// every lane the position its part starts at, and a last reading writes one code per coordinate (level,
// sign) into the string's row in shared memory. Then all threads add the rows in ascending k.
//
// Latency is what counts here: one string of 4096 dense symbols read by one lane is 300 us, whatever else
// the GPU does. So the strings are read where they are, a word ahead of the need: a copy of them in shared memory costs
// half of the resident warps (8 workers, n = 16.8 M, s = 64, d = 4096, dense code, which streams read now: 375 us with it,
// 283 without; Code_s with d = 1024: 693 and 630; only the smallest problems, which leave most of the GPU idle, lose: 17.8 and
// 18.7 us at n = 100 K). The rest is the number of instructions: the dense code is read three table entries to a window, for 10
// instructions per symbol against 30 with one entry at a time (412 -> 279 us there).
#include <type_traits>

#include "elias_decode.cuh"

namespace qsgd {

namespace {

constexpr uint32_t kThreads = 256, kMostThreads = 1024;       // (the latter where strings are shared by several warps)
template <bool DENSE> constexpr uint32_t kWarmUp = DENSE ? 96 : 64;      // bits: 75-98 % of the starts are then right
constexpr uint32_t kLeastPart = 64;               // bits of a string that are worth a lane
constexpr uint32_t kSplitBits = 120;              // ... that a lane has where a string is shared by several warps
constexpr uint32_t kDenseBits = 10;
constexpr uint32_t kFewBits = 7;                  // bits per symbol of a string from which on a table entry rarely holds one
constexpr uint32_t kRowPad = 16;                  // bytes between rows: teams at similar positions use other banks

constexpr uint32_t kLanesPerSm = 1024;            // lanes that fill an SM well enough
constexpr size_t kMostBytes = 108u << 10;         // shared memory of a CTA: two of them fit on an SM

// One code per coordinate: level | negative << kSignShift. s <= 15: 5 bits, the lane index of the value in a
// shuffle table; s <= 127: 8 bits; else 9 bits, in 16.
enum CodeWidth { kNibble = 0, kByte = 1, kWide = 2 };
template <int WIDTH> struct CodeOf {
  using type = uint8_t;
  static constexpr uint32_t kSignShift = WIDTH == kNibble ? 4u : 7u;
};
template <> struct CodeOf<kWide> {
  using type = uint16_t;
  static constexpr uint32_t kSignShift = 8u;
};

struct TeamParams {
  PeerSet peers;
  uint32_t K;
  uint32_t Kc;            // peers per pass
  uint64_t n;
  uint32_t d;
  uint32_t s;
  uint64_t B;
  float* out;             // acc (overwritten) or x (updated in place)
  float c;                // eta / K
  float minus_zero;       // add_product2
  uint32_t* status;
  uint32_t T;             // lanes per string, a power of two
  uint32_t split;         // SPLIT: warps per string, of 32 lanes each
  uint32_t buckets;       // per CTA and pass
  uint32_t row_bytes;
  Regime when;
  BucketMap map;
};

// Where in its row the code of a position lies. The lanes of a team write at positions a fixed distance
// apart (128 with 4096 coordinates and 32 lanes: one bank for all), so the pieces that the sum reads at
// once (8 codes) are permuted inside each block of 128 bytes by the number of the block.
// (The dense code stores whole words, at places as irregular as the lengths of the parts: it needs no permutation.)
template <bool DENSE, int WIDTH>
__device__ __forceinline__ uint32_t place(uint32_t pos) {       // in bytes
  if (DENSE) return WIDTH == kWide ? 2u * pos : pos;
  if (WIDTH == kWide) { const uint32_t a = 2u * pos; return a ^ ((a >> 3) & 0x70u); }
  return pos ^ ((pos >> 4) & 0x78u);
}

template <bool DENSE>
struct Tables {
  uint2 code[kCodeEntries];
  // Code_s, s <= 15: what follows a gap (tail_entry). Code'_s: what the next 10 bits hold, up to three symbols of
  // levels <= 7 (kWide: two): their length in bits 0-3, their number in bits 5-6, their codes in bytes 1, 2 and 3
  // (kWide: level | negative << 7); 0 when they hold none. Bit 4 is 0: an entry is a shift by its length as it is.
  uint32_t symbol[DENSE ? 1u << kDenseBits : kTailEntries];
  // Code'_s, for a reader that only counts: up to three symbols of those 10 bits, or the one that they start. Their
  // length in bits 0-4, that of the first of several in bits 8-11, of the first two of three in bits 12-15, their number
  // from bit 20 on. Fields of three entries can be added.
  uint32_t count[DENSE ? 1u << kDenseBits : 1u];
};

// One symbol of the dense code by the general table: level and number of bits.
__device__ __forceinline__ uint32_t dense_symbol(const uint2* code, uint32_t w, uint32_t* bits, uint32_t* closing) {
  const uint32_t x = w << 1;
  const uint2 c = code[x >> 25];
  const uint32_t body = code_body(c);
  *bits = body + 2u;
  *closing = x << body;                           // top bit: has to be 0
  return code_value(x, c) - 1u;
}

// Reads symbols from bit `from` to the first one that starts at or behind bit `until` (both counted from
// bit 0 of words[0]; `end`: first bit behind the string). Returns where that is; *sum: the gaps or, in the
// dense code, the symbols passed. What is no symbol (the reader is out of step, or the string is
// malformed) still moves it on.
template <bool DENSE, int WIDTH>
__device__ __forceinline__ uint32_t walk(const Tables<DENSE>& tab, const uint32_t* words, uint32_t from, uint32_t until,
                                         uint32_t end, uint32_t* sum) {
  *sum = 0;
  if (from >= until) return from;
  Window in;
  in.open(words, from);
  const uint32_t origin = from & ~31u;
  const uint32_t stop = until - origin, last = end - origin;
  uint32_t n = 0;
  if constexpr (DENSE) {
    auto look = [&](uint32_t w) { return tab.count[w >> (32 - kDenseBits)]; };
    while (in.bp + 31u <= stop) {                 // three entries to a window
      uint32_t w = in.peek();
      const uint32_t e0 = look(w);
      w = __funnelshift_l(0u, w, e0);
      const uint32_t e1 = look(w), e01 = e0 + e1;
      w = __funnelshift_l(0u, w, e1);
      uint32_t e = e01 + look(w);
      // long symbols: what the window does not hold is left for the next
      if ((e01 & 0xFFu) > 32u - kDenseBits || (e & 0xFFu) > 31u) e = (e01 & 0xFFu) > 31u ? e0 : e01;
      in.drop_even(e & 31u, last);
      n += e >> 20;
    }
    while (in.bp < stop) {                        // the symbols that start in front of it
      const uint32_t e = look(in.peek()), room = stop - in.bp;
      const uint32_t one = (e >> 8) & 15u, two = (e >> 12) & 15u;
      in.drop_even(one >= room ? one : two >= room ? two : e & 31u, last);
      n += one >= room ? 1u : two >= room ? 2u : e >> 20;
    }
  } else {
    while (in.bp < stop) {
      const uint32_t w = in.peek();
      const uint2 e = tab.code[w >> 25];
      const uint32_t body = code_body(e);
      n += code_value(w, e);
      if (WIDTH == kNibble) {
        const uint32_t tail = tab.symbol[(w << body) >> (32 - kTailBits)];
        in.drop(tail ? body + (tail >> 8) : body + 1u, last);
      } else {
        const uint32_t y = in.peek_at(body) << 2;
        in.drop(body, last);
        in.drop(code_body(tab.code[y >> 25]) + 3u, last);
      }
    }
  }
  *sum = n;
  return origin + in.bp;
}

// The last reading of the dense code. Codes are gathered in a word, and stored a word at a time. A word that two lanes
// have codes for is the one's that its first code belongs to: that lane reads on until it has the word, the others leave
// their part of it out. What a lane passes behind its part is checked by the lane that it belongs to.
// `few`: most symbols are too long for an entry of the table, which is then not asked for more than one at a time.
template <int WIDTH>
__device__ __forceinline__ uint32_t emit_dense(const Tables<true>& tab, const uint32_t* words, uint32_t from, uint32_t until,
                                               uint32_t end, uint32_t at, uint32_t db, uint32_t s, bool few, uint8_t* row) {
  constexpr uint32_t kBits = WIDTH == kWide ? 16u : 8u;
  if (from >= until) return 0u;
  Window in;
  in.open(words, from);
  const uint32_t origin = from & ~31u;
  const uint32_t stop = until - origin, last = end - origin;
  const uint32_t full = kBits * db;
  uint32_t q = kBits * at;                        // the next position, in bits of the row
  const uint32_t mine = (q + 31u) & ~31u;
  uint32_t addr = (uint32_t)__cvta_generic_to_shared(row) + (q >> 5) * 4u;   // of the word under way
  uint32_t bad = 0, codes = 0;
  auto gather = [&](uint32_t more, uint32_t width) {
    codes |= __funnelshift_l(0u, more, q);        // (the shift takes q mod 32)
    const uint32_t over = __funnelshift_l(more, 0u, q), next = q + width;
    // the word is whole, and it is mine
    asm volatile("{\n\t.reg .pred p, m;\n\t.reg .u32 x;\n\txor.b32 x, %2, %3;\n\tand.b32 x, x, 32;\n\tsetp.ne.u32 p, x, 0;\n\t"
                 "setp.ge.and.u32 m, %3, %4, p;\n\t@m st.shared.u32 [%1], %0;\n\t@p mov.u32 %0, %5;\n\t@p add.u32 %1, %1, 4;\n\t}"
                 : "+r"(codes), "+r"(addr) : "r"(q), "r"(next), "r"(mine + 32u), "r"(over) : "memory");
    q = next;
  };
  auto entry = [&](uint32_t e) {                  // the codes of an entry; none of the entry 0
    if (WIDTH == kWide) {
      const uint32_t x = __byte_perm(e, 0u, 0x4241);
      gather((x & 0x00070007u) | (x & 0x00800080u) << 1, (e >> 1) & 48u);
    } else {
      gather(e >> 8, (e >> 2) & 24u);
    }
  };
  auto width_of = [&](uint32_t e) { return WIDTH == kWide ? (e >> 1) & 48u : (e >> 2) & 24u; };
  auto single = [&](uint32_t w) {                 // one symbol, with every check
    uint32_t bits, closing;
    const uint32_t level = dense_symbol(tab.code, w, &bits, &closing);
    bad |= closing;
    if (level > s) return (uint32_t)QSGD_DEV_LEVEL;
    if (q >= full) return (uint32_t)QSGD_DEV_OVERRUN;                        // more symbols than coordinates
    gather(level | (level ? (w >> 31) << CodeOf<WIDTH>::kSignShift : 0u), kBits);
    in.drop_even(bits, last);
    return 0u;
  };
  if (!few) {
    while (in.bp + 3u * kDenseBits <= stop && q + 96u <= full) {             // three entries to a window
      uint32_t w = in.peek(), bits = 0, e = 0;
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        e = tab.symbol[w >> (32 - kDenseBits)];
        w = __funnelshift_l(0u, w, e);
        bits += e & 15u;
        entry(e);
      }
      in.drop_even(bits, last);
      if (e == 0u) {
        const uint32_t err = single(in.peek());
        if (err) return err;
      }
    }
  }
  // the rest; and on while the word under way is mine, has codes, and there are more
  while (in.bp < stop || ((q & 31u) != 0u && q > mine && q < full && in.bp < last)) {
    const uint32_t w = in.peek();
    const uint32_t e = few ? 0u : tab.symbol[w >> (32 - kDenseBits)];
    if (e == 0u || q + width_of(e) > full) {
      const uint32_t err = single(w);
      if (err) return err;
    } else {
      entry(e);
      in.drop_even(e & 15u, last);
    }
  }
  if ((q & 31u) != 0u && q > mine) asm volatile("st.shared.u32 [%0], %1;" ::"r"(addr), "r"(codes) : "memory");
  return bad >> 31 ? QSGD_DEV_OVERRUN : 0u;
}

// The last reading of Code_s: the same part, every check, one code per coordinate into the row. `at`: position of
// the last nonzero in front of the part.
template <int WIDTH>
__device__ __forceinline__ uint32_t emit(const Tables<false>& tab, const uint32_t* words, uint32_t from, uint32_t until,
                                         uint32_t end, uint32_t at, uint32_t db, uint32_t s, uint8_t* row) {
  using Code = typename CodeOf<WIDTH>::type;
  auto put = [&](uint32_t pos, uint32_t code) { *reinterpret_cast<Code*>(row + place<false, WIDTH>(pos)) = (Code)code; };
  constexpr uint32_t kSignShift = CodeOf<WIDTH>::kSignShift;
  if (from >= until) return 0u;
  Window in;
  in.open(words, from);
  const uint32_t origin = from & ~31u;
  const uint32_t stop = until - origin, last = end - origin;
  uint32_t bad = 0;
  while (in.bp < stop) {
    const uint32_t w = in.peek();
    const uint2 e = tab.code[w >> 25];
    const uint32_t body = code_body(e);
    at += code_value(w, e);
    if (WIDTH == kNibble) {
      const uint32_t y = w << body, tail = tab.symbol[y >> (32 - kTailBits)];
      if (tail == 0u) return y >> 31 ? QSGD_DEV_OVERRUN : in.bp + body + 2u > last ? QSGD_DEV_OVERRUN : QSGD_DEV_LEVEL;
      if (at >= db) return QSGD_DEV_POSITION;
      put(at, tail);
      in.drop(body + (tail >> 8), last);
    } else {
      const uint32_t y = in.peek_at(body), z = y << 2;
      const uint2 c = tab.code[z >> 25];
      const uint32_t level = code_value(z, c), lb = code_body(c);
      bad |= y | (z << lb);                     // the two closing bits
      if (at >= db) return QSGD_DEV_POSITION;
      if (level > s) return QSGD_DEV_LEVEL;
      put(at, level | (((y >> 30) & 1u) << kSignShift));
      in.drop(body, last);
      in.drop(lb + 3u, last);
    }
  }
  return bad >> 31 ? QSGD_DEV_OVERRUN : 0u;
}

// Reads a part in MARKS pieces and keeps where each piece ended, so that a lane that has to read its part
// again from another bit can stop at the first mark where it falls into step with its first reading.
constexpr uint32_t kLeastPiece = 96;      // bits
template <uint32_t MARKS>
struct Marks {
  uint32_t pos[MARKS];        // first symbol at or behind the mark
  uint32_t sum[MARKS];        // positions from the part's start up to there
};

// By the lanes of `mask`, which wait for one another at the marks: left to itself the compiler let them read some of the pieces one
// lane after the other (Code_s, n = 729 K, d = 4096, s = 15, K = 8, max-norm: 35 -> 53 us).
template <bool DENSE, int WIDTH, uint32_t MARKS>
__device__ __forceinline__ void read_part(const Tables<DENSE>& tab, const uint32_t* words, uint32_t start, uint32_t lo, uint32_t hi,
                                          uint32_t end, bool again, uint32_t mask, Marks<MARKS>& m) {
  const uint32_t piece = max((hi - lo + MARKS - 1u) / MARKS, kLeastPiece);
  uint32_t pos = start, sum = 0;
  bool apart = true;                                // not in step with the first reading
#pragma unroll
  for (uint32_t q = 0; q < MARKS; ++q) {
    __syncwarp(mask);
    if (apart) {
      uint32_t n;
      pos = walk<DENSE, WIDTH>(tab, words, pos, q == MARKS - 1u ? hi : min(lo + (q + 1u) * piece, hi), end, &n);
      sum += n;
      if (again && pos == m.pos[q]) {               // from here on: the rest differs by the count only
        const uint32_t more = sum - m.sum[q];
#pragma unroll
        for (uint32_t r = 0; r < MARKS; ++r)
          if (r >= q) m.sum[r] += more;
        apart = false;
      } else {
        m.pos[q] = pos;
        m.sum[q] = sum;
      }
    }
  }
  __syncwarp(mask);
}

// SPLIT: a string is shared by several warps of a CTA that has a warp for every part of its strings.
// CTAs that an SM has to hold, 0 for the compiler's choice. Code'_s, whose loops hold most, is faster with all registers that they
// want (s = 255, d = 512, K = 32 27.5 -> 25.8 us), Code_s with levels above 127 with 40 a thread and six CTAs (d = 512, K = 5 41 -> 39).
template <bool DENSE, int WIDTH, bool SPLIT> constexpr uint32_t kLeastCtas = SPLIT ? 0 : DENSE ? 1 : WIDTH == kWide ? 6 : 0;

template <bool DENSE, int WIDTH, bool FUSED, bool SPLIT, uint32_t MARKS>
__global__ void __launch_bounds__(SPLIT ? kMostThreads : kThreads, kLeastCtas<DENSE, WIDTH, SPLIT>) decode_elias_teams_kernel(const __grid_constant__ TeamParams p) {
  using Code = typename CodeOf<WIDTH>::type;
  constexpr uint32_t kLevels = 1u << CodeOf<WIDTH>::kSignShift;
  extern __shared__ __align__(16) uint8_t tsm[];
  __shared__ Tables<DENSE> tab;
  __shared__ float xi[2 * kLevels];                     // +-(level / s) by code
  __shared__ uint32_t warp_end[SPLIT ? kMostThreads / 32 : 1], warp_sum[SPLIT ? kMostThreads / 32 : 1];
  const uint32_t tid = threadIdx.x, lane = tid & 31, threads = SPLIT ? blockDim.x : kThreads;
  const float sf = (float)p.s;
  for (uint32_t i = tid; i < kCodeEntries; i += threads) tab.code[i] = code_entry(i);
  if (DENSE) {
    for (uint32_t i = tid; i < (1u << kDenseBits); i += threads) {
      const uint32_t w = i << (32 - kDenseBits);
      uint32_t used = 0, held = 0, ends = 0, codes = 0, small = 0, small_bits = 0;
      while (held < 3u) {
        const uint32_t x = w << used;
        uint32_t v, len;
        if (!elias_from_window(x << 1, v, len) || used + 1u + len > kDenseBits) break;
        if (held) ends |= used << (4u * held + 4u);
        used += 1u + len;
        if (small == held && held < (WIDTH == kWide ? 2u : 3u) && v - 1u <= min(p.s, 7u)) {
          codes |= ((v - 1u) | (v > 1u ? (x >> 31) << (WIDTH == kNibble ? 4 : 7) : 0u)) << (8u * held + 8u);
          small = held + 1u;
          small_bits = used;
        }
        ++held;
      }
      tab.symbol[i] = small ? codes | small_bits | (small << 5) : 0u;
      // (a longer one than 22 bits is of no level <= 255)
      tab.count[i] = held ? used | ends | (held << 20) : min(code_body(code_entry((w << 1) >> 25)) + 2u, 22u) | (1u << 20);
    }
  } else if (WIDTH == kNibble) {
    for (uint32_t i = tid; i < kTailEntries; i += threads) tab.symbol[i] = tail_entry(i, p.s);
  }
  for (uint32_t i = tid; i < 2u * kLevels; i += threads) {
    const float q = __fdiv_rn((float)(i & (kLevels - 1u)), sf);
    xi[i] = i & kLevels ? -q : q;
  }

  // rows[bucket][peer] of one pass over the peers | with several passes, the sums so far | the scales
  const uint32_t most = p.buckets * p.Kc;
  float* sums = reinterpret_cast<float*>(tsm + (size_t)most * p.row_bytes);
  float* scales = sums + (p.Kc < p.K ? p.buckets * p.d : 0u);
  const uint32_t T = SPLIT ? 32u : p.T, t = lane & (T - 1u);
  // SPLIT: warp w has part w / strings of string w % strings, so that the first parts, which have work whatever the length,
  // lie on all of an SM's schedulers; warps beyond that help with the tables and the sums only
  const uint32_t warp = tid >> 5, part = SPLIT ? warp / most : 0u;
  const uint32_t team = SPLIT ? warp % most : tid / T, teams = SPLIT ? most : kThreads / T;
  const uint32_t tt = part * 32u + t, TT = SPLIT ? 32u * p.split : T;     // this lane among the string's lanes
  const uint64_t groups = (p.B + p.buckets - 1) / p.buckets;
  chain_wait();                                         // the messages come from the kernels ahead
  if (!DENSE && p.when.lo && mean_below(p.when.lo, p.peers, p.K, p.B)) return;

  for (uint64_t grp = blockIdx.x; grp < groups; grp += gridDim.x) {
    const uint64_t b0 = grp * p.buckets;
    const uint32_t nb = (uint32_t)min((uint64_t)p.buckets, p.B - b0);
    for (uint32_t k0 = 0; k0 < p.K; k0 += p.Kc) {
      const uint32_t kc = min(p.Kc, p.K - k0), rows = p.buckets * kc;
      for (uint32_t i = tid; i < rows * (p.row_bytes >> 4); i += threads)
        reinterpret_cast<uint4*>(tsm)[i] = make_uint4(0u, 0u, 0u, 0u);
      __syncthreads();

      // ---- the strings, one per team and pass -------------------------------------------------------
      for (uint32_t j0 = 0; j0 < rows; j0 += teams) {
        const uint32_t j = j0 + team;
        const uint32_t g = j / kc, k = j - g * kc;         // k: in this pass
        const uint64_t b = b0 + g;
        const bool mine = j < rows && g < nb && tt < TT;
        StringRef ref;
        ref.words = nullptr; ref.lo = 0; ref.total = 0; ref.err = 0;
        uint32_t db = 0;
        const uint32_t* words = nullptr;
        if (mine) {
          db = (uint32_t)min((uint64_t)p.d, p.n - b * p.d);
          ref = string_ref(p.peers, k0 + k, b, p.B, db);
          if (!ref.err) words = ref.words + (ref.lo >> 5);
        }
        const bool reads = mine && ref.err == 0u;
        const uint32_t first = (uint32_t)(ref.lo & 31u) + 32u, end = first + ref.total;   // bits behind the scale
        // Parts of equal length, not shorter than kLeastPart. In the dense code the symbols of the levels 0, 1 and 2 are 2,
        // 4 and 4 bits long, and a reader that starts an odd number of bits from the front of a string of such levels is
        // out of step to the end of its part: where the symbols are short, parts have an even length (n = 33.5 M, d = 4096,
        // K = 8, 2-norm: 2361 -> 423 us at s = 15, 1851 -> 371 at s = 1).
        // SPLIT: a string that is shorter than was likely goes by fewer lanes, as without: more of them would start out of step.
        // So does one of symbols that are 2.75 to 3.25 bits on average, in which a warp that starts out of step often stays so
        // (n = 14 K, d = 2048, s = 32, K = 5, 3.03 bits: 19 us by 32 lanes, 27 by 64; outside that range
        // 64 lanes are 5 to 40 % faster).
        uint32_t of = TT;
        if (SPLIT) {
          if (of > 64u && ref.total < 128u * kSplitBits) of = 64u;
          if (ref.total < 64u * kSplitBits || (DENSE && 4u * ref.total >= 11u * db && 4u * ref.total < 13u * db)) of = 32u;
        }
        uint32_t per = max((ref.total + of - 1u) / of, kLeastPart);
        if (DENSE && ref.total < 3u * db) per = (per + 1u) & ~1u;
        const uint32_t lo = min(first + tt * per, end), hi = tt == TT - 1u ? end : min(lo + per, end);
        uint32_t start = lo;
        Marks<MARKS> m;
#pragma unroll
        for (uint32_t q = 0; q < MARKS; ++q) { m.pos[q] = lo; m.sum[q] = 0u; }
        const uint32_t readers = __ballot_sync(0xffffffffu, reads);
        if (reads) {
          if (tt == 0u) {
            Window in;
            in.open(words, first - 32u);
            scales[j] = __uint_as_float(in.peek());
          } else if (lo < end) {
            uint32_t skipped;
            start = walk<DENSE, WIDTH>(tab, words, lo - min(kWarmUp<DENSE>, lo - first), lo, end, &skipped);
          }
          read_part<DENSE, WIDTH, MARKS>(tab, words, start, lo, hi, end, false, readers, m);
        } else if (j < rows && tt == 0u) {
          scales[j] = 0.f;
        }
        uint32_t other = start;                           // dense code: where the other reading started (below)
        Marks<MARKS> o = m;
        uint32_t rounds = reads && ref.total < 3u * db ? 1u : 0u;           // until all lanes read again; 0: never
        for (;;) {
          if constexpr (!DENSE) {
            for (;;) {
              const uint32_t before = __shfl_up_sync(0xffffffffu, m.pos[MARKS - 1u], 1, (int)T);
              const bool again = t != 0u && before != start;
              const uint32_t who = __ballot_sync(0xffffffffu, again);
              if (who == 0u) break;
              if (again) {
                start = before;
                read_part<DENSE, WIDTH, MARKS>(tab, words, start, lo, hi, end, true, who, m);
              }
            }
          } else {
            // Short symbols again: one of an odd length, where they are rare, puts all lanes behind it out of step, each of
            // which would find out a round after the one in front of it. So where a lane that had to start elsewhere ended
            // elsewhere too, all lanes of the string read their parts from a bit further on, and keep both readings (K = 4,
            // n = 67 M, a mixture, s = 15: 1258 -> 583 us at d = 4096, 922 -> 651 at d = 2048).
            for (;;) {
              uint32_t before;
              bool again;
              for (;;) {
                before = __shfl_up_sync(0xffffffffu, m.pos[MARKS - 1u], 1, (int)T);
                again = t != 0u && before != start;
                const bool had = again && before == other;
                if (!__any_sync(0xffffffffu, had)) break;
                if (had) {
                  const Marks<MARKS> q = m;
                  m = o; o = q;
                  other = start; start = before;
                }
              }
              const uint32_t wrong = __ballot_sync(0xffffffffu, again);
              if (wrong == 0u) break;
              const bool astray = rounds != 0u && (wrong & (0xFFFFFFFFu >> (32u - T) << (lane & ~(T - 1u)))) != 0u;
              const bool now = astray && rounds == 2u;
              if (astray) rounds = now ? 0u : 2u;
              const bool further = now && t != 0u && start < hi && other == start;
              const uint32_t who = __ballot_sync(0xffffffffu, further);
              if (further) {
                other = start + 1u;
                read_part<DENSE, WIDTH, MARKS>(tab, words, other, lo, hi, end, true, who, o);
              }
              if (__any_sync(0xffffffffu, now)) continue;
              if (again) {
                o = m; other = start;
                start = before;
                read_part<DENSE, WIDTH, MARKS>(tab, words, start, lo, hi, end, true, wrong, m);
              }
            }
          }
          if constexpr (!SPLIT) break;
          // the warps of a string: the first lane of each begins where the warp in front of it ended
          if (lane == 31u) warp_end[SPLIT ? warp : 0u] = m.pos[MARKS - 1u];
          __syncthreads();
          const uint32_t before = SPLIT && part != 0u ? warp_end[SPLIT ? warp - most : 0u] : start;
          const bool wrong = reads && t == 0u && before != start;
          if (!__syncthreads_or(wrong ? 1 : 0)) break;
          if (wrong) {
            o = m; other = start;
            start = before;
            read_part<DENSE, WIDTH, MARKS>(tab, words, start, lo, hi, end, true, 1u, m);     // (lane 0)
          }
        }
        const uint32_t sum = m.sum[MARKS - 1u], stop = m.pos[MARKS - 1u];
        uint32_t upto = sum;                              // positions passed by the lanes up to this one
        for (uint32_t o = 1; o < T; o <<= 1) {
          const uint32_t q = __shfl_up_sync(0xffffffffu, upto, o, (int)T);
          if (t >= o) upto += q;
        }
        if constexpr (SPLIT) {
          if (lane == 31u) warp_sum[warp] = upto;
          __syncthreads();
          for (uint32_t w = team; w < warp; w += most) upto += warp_sum[w];
        }
        uint32_t err = ref.err;
        if (reads) {
          uint8_t* row = tsm + (size_t)j * p.row_bytes;
          if constexpr (DENSE) err |= emit_dense<WIDTH>(tab, words, start, hi, end, upto - sum, db, p.s, ref.total > kFewBits * db, row);
          else err |= emit<WIDTH>(tab, words, start, hi, end, upto - sum - 1u, db, p.s, row);
          // a string must end exactly where the table says and, in the dense code, hold every coordinate
          if (tt == TT - 1u && (stop != end || (DENSE && upto != db))) err |= QSGD_DEV_OVERRUN;
        }
        if (err) atomicOr(p.status, err);
      }
      __syncthreads();

      // ---- ascending-k sum; a thread takes 8 coordinates per pass ------------------------------------
      const uint32_t slots_per_bucket = p.d >> 3, slots = nb * slots_per_bucket;
      for (uint32_t s0 = 0; s0 < slots; s0 += threads) {
        const uint32_t slot = s0 + tid;
        const uint32_t g = slot / slots_per_bucket, c = (slot - g * slots_per_bucket) << 3;
        const uint64_t b = b0 + g;
        const bool live = slot < slots && b * p.d + c < p.n;
        if (!__any_sync(0xffffffffu, live)) continue;
        const uint32_t gg = live ? g : 0u, cc = live ? c : 0u;
        const uint8_t* codes = tsm + (size_t)gg * kc * p.row_bytes + place<DENSE, WIDTH>(cc);
        const float* sc = scales + gg * kc;
        float4* carry = reinterpret_cast<float4*>(sums + gg * p.d + cc);
        float2p sum[4] = {0ull, 0ull, 0ull, 0ull};
        if (k0) {                                         // the peers of the passes before, added by this thread
          const float4 u = carry[0], v = carry[1];
          sum[0] = pair2(u.x, u.y); sum[1] = pair2(u.z, u.w); sum[2] = pair2(v.x, v.y); sum[3] = pair2(v.z, v.w);
        }
        if (WIDTH == kWide) {
          for (uint32_t k = 0; k < kc; ++k) {
            const uint4 q = *reinterpret_cast<const uint4*>(codes + k * p.row_bytes);
            const uint32_t w[4] = {q.x, q.y, q.z, q.w};
            const float Ak = sc[k];
#pragma unroll
            for (int h = 0; h < 4; ++h) sum[h] = add_product2(sum[h], Ak, xi[w[h] & 0xFFFFu], xi[w[h] >> 16], p.minus_zero);
          }
        } else {
          const float lut = WIDTH == kNibble ? xi[lane] : 0.f;
#pragma unroll 2
          for (uint32_t k = 0; k < kc; ++k) {
            const uint2 q = *reinterpret_cast<const uint2*>(codes + k * p.row_bytes);
            const float Ak = sc[k];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              const uint32_t two = (e < 2 ? q.x : q.y) >> (16 * (e & 1));
              const float v0 = WIDTH == kNibble ? shfl_f(lut, two) : xi[two & 0xFFu];
              const float v1 = WIDTH == kNibble ? shfl_f(lut, two >> 8) : xi[(two >> 8) & 0xFFu];
              sum[e] = add_product2(sum[e], Ak, v0, v1, p.minus_zero);
            }
          }
        }
        float acc[8];
#pragma unroll
        for (int e = 0; e < 4; ++e) { const float2 u = unpair2(sum[e]); acc[2 * e] = u.x; acc[2 * e + 1] = u.y; }
        if (!live) continue;
        if (k0 + kc < p.K) {
          carry[0] = make_float4(acc[0], acc[1], acc[2], acc[3]);
          carry[1] = make_float4(acc[4], acc[5], acc[6], acc[7]);
        } else {
          store_span8<FUSED>(out_span(p.out, p.map, b, c, p.d, p.n, 8u), acc, p.c);
        }
      }
      __syncthreads();                                    // the rows are free again
    }
  }
}

template <bool DENSE, int WIDTH, uint32_t MARKS>
int launch_width(TeamParams& p, bool fused, size_t smem, cudaStream_t stream) {
  static KernelSite site[4];
  void (*kern)(TeamParams);
  const bool split = p.split > 1u;
  if (split) kern = fused ? decode_elias_teams_kernel<DENSE, WIDTH, true, true, DENSE ? 1 : MARKS>
                          : decode_elias_teams_kernel<DENSE, WIDTH, false, true, DENSE ? 1 : MARKS>;
  else kern = fused ? decode_elias_teams_kernel<DENSE, WIDTH, true, false, MARKS> : decode_elias_teams_kernel<DENSE, WIDTH, false, false, MARKS>;
  const uint32_t parts = p.buckets * p.Kc * p.split * 32u, threads = split && parts > kThreads ? parts : kThreads;
  int sms = 0, occ = 0;
  const int st = site[(split ? 2 : 0) + (fused ? 1 : 0)].lookup_dynamic(kern, (int)threads, smem, &sms, &occ);
  if (st) return st;
  const uint64_t groups = (p.B + p.buckets - 1) / p.buckets, cap = (uint64_t)sms * occ;
  ScopedKernel sk(kKernDecodeEliasTeams, stream);
  return (int)launch_chained(kern, (uint32_t)(groups < cap ? groups : cap), threads, smem, stream, p);
}

}  // namespace

int launch_elias_teams(const FieldParams& f, bool dense, uint32_t mean, bool fused, cudaStream_t stream) {
  TeamParams p;
  p.peers = f.peers; p.K = f.K; p.n = f.n; p.d = f.d; p.s = f.s; p.B = f.B; p.out = f.out; p.c = f.c;
  p.status = f.status; p.map = f.map; p.when = f.when; p.minus_zero = f.minus_zero;
  const int width = f.s <= 15u ? kNibble : f.s <= 127u ? kByte : kWide;
  p.row_bytes = ((p.d * (width == kWide ? 2u : 1u) + 127u) & ~127u) + kRowPad;
  auto bytes = [&](uint32_t buckets, uint32_t peers) {
    return (size_t)peers * (buckets * (p.row_bytes + 4ull)) + (peers < p.K ? buckets * p.d * 4ull : 0ull);
  };
  // all peers at once, or (long buckets and many peers) in as few passes as shared memory allows
  uint32_t passes = 1;
  while (bytes(1, (p.K + passes - 1) / passes) > kMostBytes) ++passes;
  p.Kc = (p.K + passes - 1) / passes;
  int sms = 0;
  const int st = device_sms(&sms);
  if (st) return st;
  const uint64_t strings = p.B * p.K, lanes = (uint64_t)sms * kLanesPerSm;
  // Lanes per string: as many as fill the GPU, but not more than the strings are likely to have work for
  // (96 bits a lane at 3, 5 or 9 bits per coordinate). Then as many buckets to a CTA as occupy its threads,
  // within 64 KB, and if that does not occupy them more lanes per string after all.
  p.T = 32;
  while (p.T > 1u && p.T * 96u > p.d * (width == kNibble ? 3u : width == kByte ? 5u : 9u)) p.T >>= 1;
  while (p.T > 1u && strings * p.T > lanes) p.T >>= 1;
  p.buckets = 1;
  while (p.buckets * 2u * p.Kc * p.T <= kThreads && p.buckets * 2u <= p.B && bytes(p.buckets * 2u, p.Kc) <= (64u << 10)) p.buckets *= 2u;
  while (p.T < 32u && p.buckets * p.Kc * p.T * 2u <= kThreads) p.T <<= 1;
  // Many peers: fewer lanes per string and one pass over the strings, not several with each its own latency, unless the
  // strings are long enough for the lanes' work to count (K = 17 to 48, s > 3, d >= 1024: up to a quarter slower). Small
  // problems of Code_s, s = 1, several passes against one (us): n = 57 K, d = 1024, K = 17 31.5 / 9.1, n = 118 K, d = 1024, K = 32
  // 45.0 / 10.2.
  if (p.d < 1024u || p.K <= 16u || p.s <= 3u)
    while (p.T > 4u && p.buckets * p.Kc * p.T > kThreads) p.T >>= 1;
  // So few strings that every CTA has an SM to itself: two warps to a string, where each lane then still has 96 bits or so, or
  // four with twice as many (less is lost to the bits ahead of a part). One against two, and four (us): n = 40 K, d = 4096,
  // s = 64, K = 8, dense code 30 / 26, 32; 131 K, d = 2048, s = 15, K = 4 32 / 28, 28; 64 K, d = 4096, s = 255, K = 2 73 / 48, 36.
  // By the strings' mean length where it is known, else by what is usual. Strings that are short all the same (gradients of
  // mostly small values) then cost up to 1 us of 10: so one level in Code_s, whose strings always are, stays with one warp.
  p.split = 1;
  if (p.T == 32u && p.Kc == p.K && (p.B + p.buckets - 1) / p.buckets <= (uint64_t)sms) {
    const uint32_t strings_of_cta = p.buckets * p.Kc;
    uint32_t likely = p.d * (width == kNibble ? 3u : width == kByte ? 4u : 9u), two = 64u * 96u, four = 128u * 192u;
    if (mean != kNoBound) { likely = mean; two = 64u * kSplitBits; four = 128u * kSplitBits; }
    else if (!dense && (p.s == 1u || p.d < (p.s <= 3u ? 3072u : 1536u))) likely = 0u;
    if (strings_of_cta * 64u <= kMostThreads && likely >= two) p.split = 2;
    if (strings_of_cta * 128u <= kMostThreads && likely >= four) p.split = 4;
  }
  const size_t smem = align16(bytes(p.buckets, p.Kc));
  // Marks of a dense string's parts: one is 2 to 4 % less work, two save half of a second reading, which is what long symbols and
  // many peers (few lanes to a string, long parts) lead to. Two against one (us): s = 3, d = 2048, K = 48 74 / 81; s = 127, d = 2048,
  // K = 32, max-norm 311 / 345; s = 15, d = 4096, K = 16 37.6 / 36.4.
  const bool two = dense && (p.K > 16u || (p.s > 15u && p.d >= 256u));
#define QSGD_RUN(D, W, M) launch_width<D, W, M>(p, fused, smem, stream)
#define QSGD_WIDTHS(D, M) (width == kNibble ? QSGD_RUN(D, kNibble, M) : width == kByte ? QSGD_RUN(D, kByte, M) : QSGD_RUN(D, kWide, M))
  return !dense ? QSGD_WIDTHS(false, 4) : two ? QSGD_WIDTHS(true, 2) : QSGD_WIDTHS(true, 1);
#undef QSGD_WIDTHS
#undef QSGD_RUN
}

}  // namespace qsgd
