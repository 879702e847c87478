// Decode-and-aggregate, Elias path (Code_s, s <= 15, at most 32 peers), where strings are many: a lane per
// (run of consecutive buckets, peer). (Section 3.1, end of "Efficient Coding of Gradients", for the string;
// Appendix A.2 for the integer code; Algorithm 1 for the sum and the step.)
//
// A peer's strings of consecutive buckets are one stretch of its payload, so a lane reads one stream from
// end to end, by background copies of 16 bytes into its own 128 bytes of shared memory: a load into a register
// that a later instruction moves or shifts holds up the whole warp, whichever lane it was for (that, not the
// instructions, was the time of reading: 300 of 360 us at n = 2^25). It writes one byte per nonzero -- level |
// negative << 4, the lane index of +-(level / s) in a shuffle table -- into its ring of 256 positions in
// shared memory. When all lanes of a warp have passed the next `step` positions, the warp adds them up
// (ascending k), writes the sums out, puts zeros back, and goes on; a lane whose string is short there
// meanwhile reads ahead, up to the ring's end, so lanes seldom wait for one another.
//
// The stream is read by table: the next kBits bits index an entry that says how far to go (up to two whole
// entries of the string, or one and the next gap, or a gap alone), which two bytes to store and where. A bit of
// state tells whether a gap or, after a gap alone, its sign and level come next. Nothing in the loop depends
// on what was read but data: lanes with different codes stay together. A gap
// that no table entry covers (64 or more) is decoded by all lanes that have come to one together, whatever else there is
// (a malformed code) by the definition's decoder with every check (slow_entry).
//
// What bounds it (n = 34 M, d = 512, s = 15, K = 16, a mixture of two scales): shared memory and the shuffles' data path, 70 % of
// its wavefronts (416 per step of a warp: 128 shuffles, about 96 byte stores and 48 lookups that meet in banks, 48 rows and
// scales, 36 copies, 34 zeros, 41 sums written), beside 67 % of the issue slots, with the 15 warps that fit. Sums in pairs: 469
// -> 461 us at n = 60 M. Without any sum it takes 359. A burst of 53 instead of 64 instructions, 18 warps with half of the
// stream's bytes in shared memory: no faster (472 and 457; 3265 and 3472 against 3284 at n = 268 M, N(0, 1)).
#include "elias_stream.cuh"

namespace qsgd {

namespace {

constexpr uint32_t kBits = 12;                         // stream bits per lookup
constexpr uint32_t kTabWords = 1u << kBits;            // entries per state
constexpr uint32_t kStateBit = 4u << kBits;            // byte offset of the second state's table: also its bit in an entry
constexpr uint32_t kRing = 256;                        // positions (bytes) per lane
constexpr uint32_t kStep = 128;                        // positions added up at a time
constexpr uint32_t kMostAdvance = 63;                  // positions per entry of the table
constexpr uint32_t kChunks = 8;                        // 16-byte pieces of the stream that a lane has in shared memory
constexpr uint32_t kStage = 16u * kChunks;             // bytes of them
constexpr int32_t kAhead = 128;                        // bits (one piece) that have to be there for a round of the burst
constexpr uint32_t kMaxWarps = 20;

// Table entry: bits 0-3 stream bits used (0: nothing here for the table), 4-8 first byte, 9-13 second byte (what
// stands above either is ignored by the shuffles), kStateBit next state, 15 and 24 whether there is a first and
// a second byte, byte 2 place of the first byte, 26-31 place of the second = how far the entry goes, both from
// the last position passed.
constexpr uint32_t kFirst = 1u << 15, kSecond = 1u << 24;

// Sign and level at the top of w, `room` bits of which are there: level | negative << 4, and its length (0: none).
__device__ __forceinline__ uint32_t tail_at(uint32_t w, uint32_t room, uint32_t s, uint32_t* len) {
  uint32_t level, ll;
  const bool ok = elias_from_window(w << 1, level, ll) && 1u + ll <= room && level <= s;
  *len = ok ? 1u + ll : 0u;
  return (level & 15u) | (w >> 31) << 4;
}

__device__ __forceinline__ uint32_t ring_entry(uint32_t i, bool tail_first, uint32_t s) {
  uint32_t w = i << (32u - kBits), room = kBits, used = 0;
  const uint32_t stuck = tail_first ? kStateBit : 0u;
  uint32_t gap = 1, len;
  if (!tail_first) {
    if (!elias_from_window(w, gap, len) || len > room || gap > kMostAdvance) return stuck;
    w <<= len; room -= len; used = len;
  }
  const uint32_t c1 = tail_at(w, room, s, &len);
  if (len == 0u)                                       // a gap alone: stop in front of its position
    return tail_first || gap == 1u ? stuck : used | kStateBit | (gap - 1u) << 26;
  w <<= len; room -= len; used += len;
  const uint32_t first = c1 << 4 | kFirst | gap << 16;
  uint32_t gap2;
  if (!elias_from_window(w, gap2, len) || len > room || gap + gap2 > kMostAdvance) return used | first | gap << 26;
  w <<= len; room -= len; used += len;
  const uint32_t c2 = tail_at(w, room, s, &len);
  if (len == 0u) return used | first | kStateBit | (gap + gap2 - 1u) << 26;       // the second gap alone
  return (used + len) | first | c2 << 9 | kSecond | (gap + gap2) << 26;
}

__device__ __forceinline__ uint32_t table_entry(const uint32_t* tab, uint32_t w, uint32_t state) {
  const uint32_t at = ((w >> (30u - kBits)) & (kStateBit - 4u)) | state;
  return *reinterpret_cast<const uint32_t*>(reinterpret_cast<const uint8_t*>(tab) + at);
}

struct RingParams {
  PeerSet peers;
  uint32_t K;
  uint32_t Kpad;          // lanes per run: K rounded up to a power of two
  uint64_t n;
  uint32_t d;
  uint32_t s;
  uint64_t B;
  float* out;             // acc (overwritten) or x (updated in place)
  float c;                // eta / K
  float minus_zero;       // add_product2
  uint32_t* status;
  uint32_t run;           // buckets per run
  uint32_t slots;         // scales kept per lane, a power of two: the buckets that a ring can touch
  uint32_t warp_bytes;
  Regime when;
  BucketMap map;
};

// One entry (or the rest of one) by the definition's decoder, with every check: the QSGD_DEV_* faults, or the
// next state, last position passed and bits used. The caller stores a rest's byte.
struct SlowStep {
  uint32_t err, at, used, state;
  uint32_t code;
};
__device__ __noinline__ SlowStep slow_entry(uint32_t w, uint32_t left, uint32_t at, uint32_t stop, uint32_t s, bool tail) {
  SlowStep r;
  r.err = 0; r.at = at; r.used = 0; r.state = 0; r.code = 0;
  uint32_t v, len;
  if (!tail) {
    const bool ok = elias_from_window(w, v, len);
    if (!ok || len > left) { r.err = QSGD_DEV_OVERRUN; return r; }
    if (v > stop - 1u - at) { r.err = QSGD_DEV_POSITION; return r; }
    r.at = at + v - 1u; r.used = len; r.state = 1u;
  } else {
    const bool ok = elias_from_window(w << 1, v, len);
    if (!ok || len + 1u > left) { r.err = QSGD_DEV_OVERRUN; return r; }
    if (v > s) { r.err = QSGD_DEV_LEVEL; return r; }
    r.at = at + 1u; r.used = len + 1u; r.code = v | (w >> 31) << 4;
  }
  return r;
}

// V: coordinates a lane adds up at a time: 8, or 4 where a warp has only one run.
template <bool FUSED, uint32_t V>
__global__ void __launch_bounds__(kMaxWarps * 32, 1) decode_elias_ring_kernel(const __grid_constant__ RingParams p) {
  extern __shared__ __align__(16) uint8_t ring_shared[];
  __shared__ uint32_t tab[2u * kTabWords];
  const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = blockDim.x >> 5;
  if (p.when.lo) {                                // standing down should cost little: before the table is made
    chain_wait();
    if (mean_below(p.when.lo, p.peers, p.K, p.B)) return;
  }
  for (uint32_t i = tid; i < 2u * kTabWords; i += blockDim.x) tab[i] = ring_entry(i & (kTabWords - 1u), i >= kTabWords, p.s);
  const uint32_t G = 32u / p.Kpad, g = lane / p.Kpad, k = lane % p.Kpad, rows = G * p.K;
  float lut0;
  {
    const float q = __fdiv_rn((float)(lane & 15u), (float)p.s);
    lut0 = lane & 16u ? -q : q;
  }
  // per warp: rows of kRing bytes | 32 lanes' pieces of their streams | slots x 32 scales. Position q of lane l's
  // row is byte q ^ 8 l of the row, so that lanes at the same position are in different banks.
  uint8_t* mine = ring_shared + ((256u - (shared_address(ring_shared) & 255u)) & 255u) + (size_t)warp * p.warp_bytes;
  for (uint32_t i = lane; i < p.warp_bytes / 16u; i += 32) reinterpret_cast<uint4*>(mine)[i] = make_uint4(0u, 0u, 0u, 0u);
  const uint32_t shared_mine = shared_address(mine);
  const uint32_t stage = shared_mine + rows * kRing + lane * kStage;
  float* scales = reinterpret_cast<float*>(mine + rows * kRing + 32u * kStage);
  const bool walker = k < p.K;
  const uint32_t ring = shared_mine + (walker ? g * p.K + k : 0u) * kRing;          // 256-aligned
  const uint32_t cell = ring | lane * 8u;                                            // address of q: (q & 255) ^ cell
  chain_wait();                                   // the messages come from the kernels ahead
  __syncthreads();

  const uint64_t first_of_warp = ((uint64_t)blockIdx.x * nwarps + warp) * G * p.run;
  const uint64_t first = first_of_warp + (uint64_t)g * p.run;             // the run's first bucket
  const uint32_t nb = first < p.B ? (uint32_t)min((uint64_t)p.run, p.B - first) : 0u;
  const uint32_t most = __reduce_max_sync(0xffffffffu, nb * p.d);         // positions of the warp's longest run

  // ---- the peer's table; the end of the string after the current one is always on its way -----------
  const uint64_t* table = nullptr;
  uint64_t all = 0, hi = 0, ahead = 0;
  uint32_t err = 0;
  uint32_t b = nb;                                // buckets opened so far
  if (walker && nb) {
    PeerTable pt;
    if (peer_table(p.peers, k, p.B, &pt)) {
      b = 0;
      table = pt.table + first;
      all = __ldg(pt.table + p.B);
      hi = __ldg(table);
      ahead = __ldg(table + 1);
      if (all > pt.cap_bits) all = 0;             // a payload that ends past its bound: no string passes
    } else {
      err = QSGD_DEV_TABLE;                       // nothing of this message is read
    }
  }
  // The stream: bits are counted from the 16-byte piece that it was entered in. Pieces [0, pieces) of it have been
  // asked for, of pieces_all that the payload has; bits up to `ready` are there. The window: w0 holds bit bp, edge is
  // the first bit of w1.
  const uint4* stream = nullptr;
  uint32_t pieces = 0, pieces_all = 0, ready = 0;
  uint32_t w0 = 0, w1 = 0, w2 = 0, bp = 0, edge = 32, end = 0;
  uint32_t at = 0xFFFFFFFFu;                      // last position passed
  uint32_t stop = 0;                              // first position behind the bucket
  uint32_t state = 0;                             // 0 or kStateBit
  bool live = false;                              // inside a string
  enum { kAway, kAsked, kThere } where = kAway;   // the window: not at the next string; its bits asked for; at it
  auto drop = [&](uint32_t bits) {                // at most 32
    bp += bits;
    const bool cross = bp >= edge;
    w0 = cross ? w1 : w0;
    w1 = cross ? w2 : w1;
    load_word_if(cross, w2, stage + (((edge >> 3) + 8u) & (kStage - 1u)));        // the word behind w2
    edge += cross ? 32u : 0u;
  };
  auto ask = [&]() {                              // for the pieces that there is room for
    if (where != kAway)
      while (pieces < pieces_all && pieces < (bp >> 7) + kChunks) {
        copy16(stage + ((pieces * 16u) & (kStage - 1u)), stream + pieces);
        ++pieces;
      }
  };

  // ---- this lane's part in adding up: V positions of a run, from `off_sum` on in every step ----------
  constexpr uint32_t kParts = kStep / V;          // lanes per run
  const uint32_t off_sum = (lane & (kParts - 1u)) * V;
  uint32_t bucket_sum = 0, in_bucket = 0;         // bucket of the run, and place in it, of position `consumed`

  for (uint32_t consumed = 0; consumed < most; consumed += kStep) {
    const uint32_t goal = consumed + kStep;
    // ---- every lane reads on until it has passed `goal` ---------------------------------------------
    bool stuck = false;
    for (;;) {
      copies_done();
      ready = pieces == pieces_all ? 0x7FFFFFFFu : pieces * 128u;
      // a lane short of the goal is at the end of a string or at something the table does not cover, or its bits
      // have not been there
      const bool is_short = (live || b < nb) && (int32_t)at < (int32_t)goal - 1;
      const bool over = live && (int32_t)(at + (state ? 1u : 0u) - stop) >= 0;
      if (__any_sync(0xffffffffu, over || (is_short && (!live || bp >= end || stuck)))) {
        if (over) {                               // went past the bucket: take it back
          for (uint32_t q = stop; q != at + 1u; ++q) store_byte((q & (kRing - 1u)) ^ cell, 0u);
          err |= QSGD_DEV_POSITION;
          live = false;
          where = kAway;
        } else if (live && stuck && bp < end && (int32_t)(at + 1u - consumed) < (int32_t)kRing &&
                   (int32_t)(ready - bp) >= kAhead) {
          const SlowStep sl = slow_entry(__funnelshift_l(w1, w0, bp), end - bp, at, stop, p.s, state != 0u);
          if (sl.err) {
            err |= sl.err;
            live = false;
            where = kAway;
          } else {
            if (state) store_byte((sl.at & (kRing - 1u)) ^ cell, sl.code);
            at = sl.at;
            state = sl.state ? kStateBit : 0u;
            drop(sl.used);
          }
        }
        if (live && bp >= end) {                  // through: it must end exactly where the table says
          if (bp != end || state) { err |= QSGD_DEV_OVERRUN; where = kAway; }
          live = false;
        }
        if (!live) { end = bp; at = b * p.d - 1u; }
        if (!live && b < nb && (int32_t)(b * p.d - consumed) < (int32_t)kRing) {      // the next one
          const uint64_t lo = hi;
          const uint32_t db = (uint32_t)min((uint64_t)p.d, p.n - (first + b) * p.d);
          uint32_t fault = 0;
          if (ahead < lo || ahead - lo < 32ull || ahead > all) fault = QSGD_DEV_TABLE;
          else if (ahead - lo > 32ull + 40ull * db) fault = QSGD_DEV_OVERRUN;
          if (!fault && where == kAway) {         // enter the stream there
            stream = reinterpret_cast<const uint4*>(p.peers.payload[k]) + (lo >> 7);
            pieces_all = (uint32_t)(((all + 127ull) >> 7) - (lo >> 7));
            pieces = 0;
            bp = end = (uint32_t)(lo & 127u);
            ready = 0;
            where = kAsked;
          }
          if (fault || (int32_t)(ready - bp) >= kAhead + 32) {
            float A = 0.f;
            if (fault) {                          // nothing of this string is read
              err |= fault;
              where = kAway;
              at = (b + 1u) * p.d - 1u;
            } else {
              if (where == kAsked) {
                const uint32_t word = (bp >> 5) * 4u;
                w0 = load_word(stage + (word & (kStage - 1u)));
                w1 = load_word(stage + ((word + 4u) & (kStage - 1u)));
                w2 = load_word(stage + ((word + 8u) & (kStage - 1u)));
                edge = (bp & ~31u) + 32u;
                where = kThere;
              }
              end = bp + (uint32_t)(ahead - lo);
              A = __uint_as_float(__funnelshift_l(w1, w0, bp));
              drop(32u);
              stop = b * p.d + db;
              state = 0u;
              live = true;
            }
            scales[(b & (p.slots - 1u)) * 32u + lane] = A;
            hi = ahead;
            ++b;
            if (b < nb) ahead = __ldg(table + b + 1);
          }
        }
      }
      ask();
      // the burst: all lanes together, until none that can go on is short of the goal
      const int32_t room = (int32_t)(consumed + kRing - kMostAdvance);      // of `at`: room for an entry
      int32_t until = room;
      const uint32_t last = ready ? min(end, ready - (uint32_t)kAhead + 1u) : 0u;        // first bit to stop at
      bool hard = false, done;
      for (;;) {
        for (;;) {
          const bool go = (int32_t)at < until && (int32_t)(last - bp) > 0;
          if (!__any_sync(0xffffffffu, go && (int32_t)at < (int32_t)goal - 1)) break;
          // (a lane that does not go on finds an entry for nothing)
          // bits behind the string's end read as ones: no code is complete with them
          const uint32_t w = __funnelshift_l(w1, w0, bp) | __funnelshift_rc(0xFFFFFFFFu, 0u, end - bp);
          uint32_t e = table_entry(tab, w, state);
          e = go ? e : state;
          store_byte_if(e & kFirst, (__dp4a(e, 0x00010000u, at) & (kRing - 1u)) ^ cell, e >> 4);
          at += e >> 26;
          store_byte_if(e & kSecond, (at & (kRing - 1u)) ^ cell, e >> 9);
          state = e & kStateBit;
          uint32_t f = table_entry(tab, w << (e & 15u), state);
          f = go && (int32_t)at < until ? f : state;
          store_byte_if(f & kFirst, (__dp4a(f, 0x00010000u, at) & (kRing - 1u)) ^ cell, f >> 4);
          at += f >> 26;
          store_byte_if(f & kSecond, (at & (kRing - 1u)) ^ cell, f >> 9);
          until = f & 15u ? until : INT32_MIN;      // nothing for the table here, or far enough
          state = f & kStateBit;
          drop((e & 15u) + (f & 15u));
        }
        done = !__any_sync(0xffffffffu, ((live || b < nb) && (int32_t)at < (int32_t)goal - 1) ||
                                            (live && (int32_t)(at + (state ? 1u : 0u) - stop) >= 0));
        if (done) break;
        // a gap that is too long for the table, in all lanes that have come to one (478 -> 467 us against leaving it to
        // slow_entry at n = 60 M, d = 512, s = 15, K = 16, a mixture of two scales; 161 -> 155 at s = 3, d = 256)
        const bool gap = until == INT32_MIN && !hard && state == 0u && (int32_t)at < room && (int32_t)(last - bp) > 0;
        if (!__any_sync(0xffffffffu, gap && (int32_t)at < (int32_t)goal - 1)) break;
        if (gap) {
          uint32_t v, len;
          hard = !elias_from_window(__funnelshift_l(w1, w0, bp), v, len) || len > end - bp || v > stop - 1u - at;
          if (!hard) {
            at += v - 1u;
            state = kStateBit;
            until = room;
            drop(len);
          }
        }
      }
      if (done) break;
      stuck = until == INT32_MIN;
    }
    ask();                                        // they come while the warp adds up
    __syncwarp();

    // ---- ascending-k sums of positions [consumed, goal) of each run ------------------------------------
    uint32_t bq = bucket_sum, c = in_bucket + off_sum;
    while (c >= p.d) { c -= p.d; ++bq; }
    const uint32_t q = consumed + off_sum;
    for (uint32_t gq = lane / kParts; gq < G; gq += 32u / kParts) {        // all lanes alike: 32 / kParts divides G
      const uint64_t run_first = first_of_warp + (uint64_t)gq * p.run;
      OutSpan sp;
      sp.ptr = p.out; sp.valid = 0u;
      if (bq < p.run) {
        if (p.map.src) {
          if (run_first + bq < p.B) sp = out_span(p.out, p.map, run_first + bq, c, p.d, p.n, V);
        } else {                                  // buckets follow one another: position q of the run is simply there
          const uint64_t i = run_first * p.d + q;
          sp.ptr = p.out + i;
          sp.valid = i < p.n ? (uint32_t)min((uint64_t)V, p.n - i) : 0u;
        }
      }
      const bool whole = sp.valid == V && (reinterpret_cast<uintptr_t>(sp.ptr) & 15u) == 0;
      float4 x[V / 4];
      if (FUSED && whole)
#pragma unroll
        for (uint32_t h = 0; h < V / 4; ++h) x[h] = reinterpret_cast<const float4*>(sp.ptr)[h];
      const uint32_t row0 = shared_mine + gq * p.K * kRing, pos = (q & (kRing - 1u)) ^ (gq * p.Kpad * 8u);
      const float* sc = scales + (bq & (p.slots - 1u)) * 32u + gq * p.Kpad;
      float2p sum[V / 2];
#pragma unroll
      for (uint32_t e = 0; e < V / 2; ++e) sum[e] = 0ull;
#pragma unroll 4
      for (uint32_t kk = 0; kk < p.K; ++kk) {
        uint32_t w[V / 4];
        const uint32_t addr = row0 + kk * kRing + (pos ^ (kk * 8u));
        if (V == 8) load_words(addr, w[0], w[V / 4 - 1]);
        else w[0] = load_word(addr);
        const float A = sc[kk];
#pragma unroll
        for (uint32_t e = 0; e < V; e += 2)
          sum[e / 2] = add_product2(sum[e / 2], A, shfl_f(lut0, w[e >> 2] >> (8u * (e & 3u))), shfl_f(lut0, w[e >> 2] >> (8u * (e & 3u) + 8u)),
                                    p.minus_zero);
      }
      float acc[V];
#pragma unroll
      for (uint32_t e = 0; e < V / 2; ++e) { const float2 u = unpair2(sum[e]); acc[2 * e] = u.x; acc[2 * e + 1] = u.y; }
      if (whole) {
#pragma unroll
        for (uint32_t h = 0; h < V / 4; ++h) {
          float4 o = make_float4(acc[4 * h], acc[4 * h + 1], acc[4 * h + 2], acc[4 * h + 3]);
          if (FUSED) {
            o.x = __fsub_rn(x[h].x, __fmul_rn(p.c, o.x)); o.y = __fsub_rn(x[h].y, __fmul_rn(p.c, o.y));
            o.z = __fsub_rn(x[h].z, __fmul_rn(p.c, o.z)); o.w = __fsub_rn(x[h].w, __fmul_rn(p.c, o.w));
          }
          reinterpret_cast<float4*>(sp.ptr)[h] = o;
        }
      } else if (sp.valid) {
#pragma unroll
        for (uint32_t e = 0; e < V; ++e)
          if (e < sp.valid) sp.ptr[e] = FUSED ? __fsub_rn(sp.ptr[e], __fmul_rn(p.c, acc[e])) : acc[e];
      }
    }
    in_bucket += kStep;
    while (in_bucket >= p.d) { in_bucket -= p.d; ++bucket_sum; }
    __syncwarp();
    // ---- zeros back: each lane its own row, 16 bytes at a time, starting at different banks ------------
    if (walker) {
      const uint32_t from = ((consumed & (kRing - 1u)) ^ cell) & ~(kStep - 1u);
#pragma unroll
      for (uint32_t i = 0; i < kStep / 16u; ++i) zero_quad(from | (((i + lane) & (kStep / 16u - 1u)) << 4));
    }
    __syncwarp();
  }
  copies_done();
  if (live && (bp != end || state)) err |= QSGD_DEV_OVERRUN;      // a string must end exactly where the table says
  if (err) atomicOr(p.status, err);
}

}  // namespace

int launch_elias_ring(const FieldParams& f, bool fused, cudaStream_t stream) {
  static KernelSite site[4];
  RingParams p;
  p.peers = f.peers; p.K = f.K; p.n = f.n; p.d = f.d; p.s = f.s; p.B = f.B; p.out = f.out; p.c = f.c;
  p.status = f.status; p.map = f.map; p.when = f.when; p.minus_zero = f.minus_zero;
  p.Kpad = 1;
  while (p.Kpad < p.K) p.Kpad <<= 1;
  const uint32_t G = 32u / p.Kpad;
  p.slots = 2;
  while (p.slots < kRing / p.d + 2u) p.slots <<= 1;
  p.warp_bytes = G * p.K * kRing + 32u * kStage + p.slots * 128u;
  p.warp_bytes = (p.warp_bytes + 255u) & ~255u;
  int sms = 0, most_shared = 0, occ = 0;
  int st = device_sms(&sms);
  if (!st) st = device_shared_memory(&most_shared);
  if (st) return st;
  uint32_t warps = ((uint32_t)most_shared - 2u * kStateBit - 2048u) / p.warp_bytes;
  if (warps > kMaxWarps) warps = kMaxWarps;
  // one run of consecutive buckets per lane group, all of the same length, in one wave
  const uint64_t groups = (uint64_t)sms * warps * G;
  p.run = (uint32_t)((p.B + groups - 1) / groups);
  const uint64_t need = (p.B + (uint64_t)p.run * G - 1) / ((uint64_t)p.run * G);      // warps with work
  const uint32_t per_sm = (uint32_t)((need + sms - 1) / sms);
  if (per_sm < warps) warps = per_sm < 8u ? 8u : per_sm;
  const size_t smem = (size_t)warps * p.warp_bytes + 1024u;
  void (*kern)(RingParams);
  if (G == 1u) kern = fused ? decode_elias_ring_kernel<true, 4> : decode_elias_ring_kernel<false, 4>;
  else kern = fused ? decode_elias_ring_kernel<true, 8> : decode_elias_ring_kernel<false, 8>;
  st = site[(G == 1u ? 2 : 0) + (fused ? 1 : 0)].lookup_dynamic(kern, (int)warps * 32, smem, &sms, &occ);
  if (st) return st;
  ScopedKernel sk(kKernDecodeElias, stream);
  return (int)launch_chained(kern, (uint32_t)((need + warps - 1) / warps), warps * 32u, smem, stream, p);
}

}  // namespace qsgd
