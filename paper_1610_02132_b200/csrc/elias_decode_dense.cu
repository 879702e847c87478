// Decode-and-aggregate, dense code (Code'_s, s <= 127, at most 32 peers), where strings are many and levels are not: a lane per (run of
// consecutive buckets, peer). (Appendix A.3 for the code, Appendix A.2 for its integers; Algorithm 1 for the sum and the step.)
//
// A symbol for every coordinate: lanes that read at the same rate stay at the same positions, so a lane reads its stream from
// end to end, once, without looking for the place of its part first as the teams have to (elias_decode_teams.cu, which read a
// string two to four times). The stream comes by background copies into the lane's 128 bytes of shared memory, two table
// entries of up to four symbols are taken from a window of 32 bits, and the codes -- 2 level + negative, a byte each -- are
// gathered in a word and stored whole into the lane's ring of 256 positions. Every 128 positions the warp adds the peers'
// codes up in ascending k, as the stream reader of Code_s does (elias_decode_ring.cu).
//
// What bounds it: the latency of a lane's chain of lookups, with seven warps on an SM at n = 17 M, d = 4096, K = 8, s = 64 (0.4
// of the issue slots used): 182 us against 279 by teams; at 67 M, d = 4096, K = 4, s = 15, a mixture 248 against 541, at 17 M,
// d = 256, K = 4, s = 15, max-norm 143 against 426. 12 bits and up to four symbols a lookup instead of 10 and three: 208 -> 190;
// codes gathered during the next window's lookups: 190 -> 182. Twice the ring, the step and the stream in shared memory: 174
// there, but 373 instead of 248 at 67 M, where it leaves eight warps.
#include "elias_stream.cuh"

namespace qsgd {

namespace {

constexpr uint32_t kBits = 12;                         // stream bits per lookup
constexpr uint32_t kRing = 256;                        // positions (bytes) per lane
constexpr uint32_t kStep = 128;                        // positions added up at a time
constexpr uint32_t kChunks = 8;                        // 16-byte pieces of the stream that a lane has in shared memory
constexpr uint32_t kStage = 16u * kChunks;             // bytes of them
constexpr int32_t kAhead = 160;                        // bits that have to be there for a window: two entries or one and a symbol
                                                       // (35 bits), and the words that follow
// Places in the window of shared memory: of the table, a multiple of its length, so that an index and the place need no
// addition, of the entry for lanes that stand still, and of the values by code.
constexpr uint32_t kTableAt = 8u << kBits, kNothingAt = 2u * kTableAt, kValuesAt = kNothingAt + 1024u, kTableEnd = kValuesAt + 1024u;
constexpr uint32_t kMaxWarps = 16;

struct DenseParams {
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
  uint32_t in_front;      // warps whose shared memory lies in front of the tables
  uint32_t work;          // warps of a CTA that have runs; the others help to make the tables
  BucketMap map;
};

// What the next 12 bits hold, up to four symbols of levels <= min(s, 127): x: their codes; y: their length in bits 0-4, 8 x
// their number from bit 8 on; 0 when they hold none.
__device__ __forceinline__ uint2 symbols_entry(uint32_t i, uint32_t s) {
  const uint32_t w = i << (32u - kBits);
  uint32_t used = 0, held = 0, codes = 0;
  while (held < 4u) {
    const uint32_t x = w << used;
    uint32_t v, len;
    if (!elias_from_window(x << 1, v, len) || used + 1u + len > kBits || v - 1u > min(s, 127u)) break;
    codes |= (2u * (v - 1u) | (v > 1u ? x >> 31 : 0u)) << (8u * held);
    used += 1u + len;
    ++held;
  }
  return make_uint2(codes, held ? used | held << 11 : 0u);
}

__device__ __forceinline__ uint2 load_entry(uint32_t addr) {
  uint2 e;
  asm("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(e.x), "=r"(e.y) : "r"(addr));
  return e;
}
__device__ __forceinline__ uint32_t entry_at(uint32_t w) { return ((w >> (29u - kBits)) & (kTableAt - 8u)) | kTableAt; }
// Value of the code in byte j of w.
__device__ __forceinline__ float value_at(uint32_t w, uint32_t j) {
  float v;
  asm("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(((j ? w >> (8u * j - 2u) : w << 2) & 0x3FCu) | kValuesAt));
  return v;
}

// BYTE: codes of more than 5 bits (s > 15), looked up in shared memory instead of across the lanes. V: coordinates that a
// lane adds up at a time: 8, or 4 where a warp has only one run.
template <bool FUSED, bool BYTE, uint32_t V>
__global__ void __launch_bounds__(kMaxWarps * 32, 1) decode_elias_dense_kernel(const __grid_constant__ DenseParams p) {
  extern __shared__ __align__(16) uint8_t dense_shared[];
  __shared__ uint2 code[kCodeEntries];
  const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (uint32_t i = tid; i <= (1u << kBits); i += blockDim.x) {
    const uint2 e = i == 1u << kBits ? make_uint2(0u, 0u) : symbols_entry(i, p.s);
    asm volatile("st.shared.v2.u32 [%0], {%1, %2};" ::"r"(kTableAt + 8u * i), "r"(e.x), "r"(e.y) : "memory");
  }
  for (uint32_t i = tid; i < kCodeEntries; i += blockDim.x) code[i] = code_entry(i);
  const float sf = (float)p.s;
  if (BYTE)                                             // +-(level / s) by code
    for (uint32_t i = tid; i < 256u; i += blockDim.x) {
      const float q = __fdiv_rn((float)(i >> 1), sf);
      asm volatile("st.shared.f32 [%0], %1;" ::"r"(kValuesAt + 4u * i), "f"(i & 1u ? -q : q) : "memory");
    }
  const float q0 = __fdiv_rn((float)(lane >> 1), sf), lut0 = lane & 1u ? -q0 : q0;
  const uint32_t G = 32u / p.Kpad, g = lane / p.Kpad, k = lane % p.Kpad, rows = G * p.K;
  // per warp: rows of kRing bytes | 32 lanes' pieces of their streams | slots x 32 scales. Position q of lane l's
  // row is byte q ^ 8 l of the row, so that lanes at the same position are in different banks.
  // Warps lie in front of the table and behind it.
  const uint32_t front = (shared_address(dense_shared) + 255u) & ~255u;
  const uint32_t shared_mine = warp < p.in_front ? front + warp * p.warp_bytes : kTableEnd + (warp - p.in_front) * p.warp_bytes;
  if (warp < p.work)
    for (uint32_t i = lane; i < p.warp_bytes / 16u; i += 32) zero_quad(shared_mine + 16u * i);
  const uint32_t stage = shared_mine + rows * kRing + lane * kStage;
  float* scales = reinterpret_cast<float*>(dense_shared + (shared_mine - shared_address(dense_shared)) + rows * kRing + 32u * kStage);
  const bool walker = k < p.K;
  const uint32_t ring = shared_mine + (walker ? g * p.K + k : 0u) * kRing;          // 256-aligned
  const uint32_t cell = ring | lane * 8u;                                            // address of q: (q & 255) ^ cell
  __syncthreads();
  chain_wait();                                   // the messages come from the kernels ahead
  if (warp >= p.work) return;

  const uint64_t first_of_warp = ((uint64_t)blockIdx.x * p.work + warp) * G * p.run;
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
  // asked for, of pieces_all that the payload has. The window: w0 holds bit bp, edge is the first bit of w1, fetch the place
  // in the stream, in bytes, of the word behind w2.
  const uint4* stream = nullptr;
  uint32_t pieces = 0, pieces_all = 0;
  uint32_t w0 = 0, w1 = 0, w2 = 0, bp = 0, edge = 32, fetch = 0, end = 0;
  uint32_t q = 0;                                 // 8 x the next position
  uint32_t stop = 0;                              // 8 x the first position behind the bucket
  uint32_t codes = 0;                             // of the word that q lies in
  bool live = false;                              // inside a string
  enum { kAway, kAsked, kThere } where = kAway;   // the window: not at the next string; its bits asked for; at it
  auto drop = [&](uint32_t bits) {                // at most 32
    bp += bits;
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ge.u32 p, %5, %4;\n\t@p mov.b32 %0, %1;\n\t@p mov.b32 %1, %2;\n\t@p ld.shared.u32 %2, [%6];\n\t"
                 "@p add.u32 %3, %3, 4;\n\t@p add.u32 %4, %4, 32;\n\t}"
                 : "+r"(w0), "+r"(w1), "+r"(w2), "+r"(fetch), "+r"(edge) : "r"(bp), "r"((fetch & (kStage - 1u)) | stage) : "memory");
  };
  auto ask = [&]() {                              // for the pieces that there is room for
    if (where != kAway)
      while (pieces < pieces_all && pieces < (bp >> 7) + kChunks) {
        copy16(stage + ((pieces * 16u) & (kStage - 1u)), stream + pieces);
        ++pieces;
      }
  };
  auto gather = [&](uint32_t more, uint32_t width) {       // codes, 8 bits each
    codes |= __funnelshift_l(0u, more, q);        // (the shift takes q mod 32)
    const uint32_t over = __funnelshift_l(more, 0u, q), next = q + width;
    asm volatile("{\n\t.reg .pred p;\n\t.reg .u32 x;\n\txor.b32 x, %2, %3;\n\tand.b32 x, x, 32;\n\tsetp.ne.u32 p, x, 0;\n\t"
                 "@p st.shared.u32 [%1], %0;\n\t@p mov.u32 %0, %4;\n\t}"
                 : "+r"(codes) : "r"(((q >> 3) & (kRing - 4u)) ^ cell), "r"(q), "r"(next), "r"(over) : "memory");
    q = next;
  };
  auto give_up = [&](uint32_t fault) {            // the rest of the string counts nothing
    err |= fault;
    live = false;
    where = kAway;
    scales[((b - 1u) & (p.slots - 1u)) * 32u + lane] = 0.f;
  };
  auto single = [&]() {                           // one symbol by the general table, with every check
    const uint32_t x0 = __funnelshift_l(w1, w0, bp), x = x0 << 1;
    const uint2 c = code[x >> 25];
    const uint32_t body = code_body(c), level = code_value(x, c) - 1u;
    if (body + 2u > end - bp || ((x << body) >> 31)) { give_up(QSGD_DEV_OVERRUN); return; }
    if (level > p.s) { give_up(QSGD_DEV_LEVEL); return; }
    gather(2u * level | (level ? x0 >> 31 : 0u), 8u);
    drop(body + 2u);
  };

  // ---- this lane's part in adding up: V positions of a run, from `off_sum` on in every step ----------
  constexpr uint32_t kParts = kStep / V;          // lanes per run
  const uint32_t off_sum = (lane & (kParts - 1u)) * V;
  uint32_t bucket_sum = 0, in_bucket = 0;         // bucket of the run, and place in it, of position `consumed`

  for (uint32_t consumed = 0; consumed < most; consumed += kStep) {
    const uint32_t goal = 8u * (consumed + kStep), room = 8u * (consumed + kRing);
    // ---- every lane reads on until it has passed `goal` ---------------------------------------------
    while (__any_sync(0xffffffffu, (live || b < nb) && q < goal)) {
      copies_done();
      const uint32_t ready = pieces == pieces_all ? 0x7FFFFFFFu : pieces * 128u;    // bits up to here are there
      const bool ended = live && (q >= stop || bp >= end);
      if (__any_sync(0xffffffffu, ended || (!live && b < nb))) {
        if (ended) {                              // it must end exactly where the table says, with every coordinate
          if (q & 31u) asm volatile("st.shared.u32 [%0], %1;" ::"r"(((q >> 3) & (kRing - 4u)) ^ cell), "r"(codes) : "memory");
          if (q != stop || bp != end) give_up(QSGD_DEV_OVERRUN);
          live = false;
        }
        if (!live) { end = bp; q = 8u * b * p.d; codes = 0u; }
        if (!live && b < nb && q < room) {        // the next one
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
            where = kAsked;
          } else if (fault || (int32_t)(ready - bp) >= kAhead + 32) {
            float A = 0.f;
            if (fault) {                          // nothing of this string is read
              err |= fault;
              where = kAway;
              q = 8u * (b + 1u) * p.d;
            } else {
              if (where == kAsked) {
                const uint32_t word = (bp >> 5) * 4u;
                w0 = load_word(stage + (word & (kStage - 1u)));
                w1 = load_word(stage + ((word + 4u) & (kStage - 1u)));
                w2 = load_word(stage + ((word + 8u) & (kStage - 1u)));
                edge = (bp & ~31u) + 32u;
                fetch = word + 12u;
                where = kThere;
              }
              end = bp + (uint32_t)(ahead - lo);
              A = __uint_as_float(__funnelshift_l(w1, w0, bp));
              drop(32u);
              stop = 8u * (b * p.d + db);
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
      const uint32_t last = ready > (uint32_t)kAhead ? ready - (uint32_t)kAhead + 1u : 0u;      // first bit to stop at
      for (;;) {
        // Windows of two entries; the warp goes on while a lane that can is short of the goal. The codes of a window are
        // gathered while the entries of the next one are on their way.
        const int32_t most_q = (int32_t)min(stop, room) - 64, most_bp = (int32_t)min(end, last + 2u * kBits - 1u) - (int32_t)(2u * kBits);
        uint2 e0 = make_uint2(0u, 0u), f0 = e0;
        uint32_t passed = q;                      // q with the codes that are still to be gathered
        for (;;) {
          const bool go = live && (int32_t)passed <= most_q && (int32_t)bp <= most_bp;
          if (!__any_sync(0xffffffffu, go && passed < goal)) break;
          const uint32_t w = __funnelshift_l(w1, w0, bp), at0 = entry_at(w);
          const uint2 e = load_entry(go ? at0 : kNothingAt);
          gather(e0.x, e0.y >> 8);
          const uint32_t at1 = entry_at(__funnelshift_l(0u, w, e.y));
          const uint2 f = load_entry(go ? at1 : kNothingAt);
          gather(f0.x, f0.y >> 8);
          const uint32_t both = e.y + f.y;
          passed += both >> 8;
          drop(both & 31u);
          e0 = e; f0 = f;
          const bool hard = go && f.y == 0u;      // a symbol that the table does not hold (its bits are there: kAhead)
          if (__any_sync(0xffffffffu, hard)) {
            gather(e0.x, e0.y >> 8);
            gather(f0.x, f0.y >> 8);
            e0 = f0 = make_uint2(0u, 0u);
            if (hard) single();
            passed = q;
          }
        }
        gather(e0.x, e0.y >> 8);
        gather(f0.x, f0.y >> 8);
        // at a string's end, or that of the ring: an entry at a time
        const bool can = live && q < min(stop, room) && bp < min(end, last);
        if (!__any_sync(0xffffffffu, can && q < goal)) break;
        if (can) {
          const uint2 e = load_entry(entry_at(__funnelshift_l(w1, w0, bp)));
          const uint32_t width = e.y >> 8;
          if (e.y != 0u && (e.y & 31u) <= end - bp && q + width <= min(stop, room)) {
            gather(e.x, width);
            drop(e.y & 31u);
          } else {
            single();
          }
        }
      }
    }
    ask();                                        // they come while the warp adds up
    __syncwarp();

    // ---- ascending-k sums of positions [consumed, consumed + kStep) of each run --------------------------
    uint32_t bq = bucket_sum, c = in_bucket + off_sum;
    while (c >= p.d) { c -= p.d; ++bq; }
    const uint32_t at = consumed + off_sum;
    for (uint32_t gq = lane / kParts; gq < G; gq += 32u / kParts) {        // all lanes alike: 32 / kParts divides G
      const uint64_t run_first = first_of_warp + (uint64_t)gq * p.run;
      OutSpan sp;
      sp.ptr = p.out; sp.valid = 0u;
      if (bq < p.run) {
        if (p.map.src) {
          if (run_first + bq < p.B) sp = out_span(p.out, p.map, run_first + bq, c, p.d, p.n, V);
        } else {                                  // buckets follow one another: position q of the run is simply there
          const uint64_t i = run_first * p.d + at;
          sp.ptr = p.out + i;
          sp.valid = i < p.n ? (uint32_t)min((uint64_t)V, p.n - i) : 0u;
        }
      }
      const bool whole = sp.valid == V && (reinterpret_cast<uintptr_t>(sp.ptr) & 15u) == 0;
      float4 x[V / 4];
      if (FUSED && whole)
#pragma unroll
        for (uint32_t h = 0; h < V / 4; ++h) x[h] = reinterpret_cast<const float4*>(sp.ptr)[h];
      const uint32_t row0 = shared_mine + gq * p.K * kRing, pos = (at & (kRing - 1u)) ^ (gq * p.Kpad * 8u);
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
        for (uint32_t e = 0; e < V; e += 2) {
          const uint32_t two = w[e >> 2] >> (8u * (e & 3u));
          const float v0 = BYTE ? value_at(w[e >> 2], e & 3u) : shfl_f(lut0, two);
          const float v1 = BYTE ? value_at(w[e >> 2], (e & 3u) + 1u) : shfl_f(lut0, two >> 8);
          sum[e / 2] = add_product2(sum[e / 2], A, v0, v1, p.minus_zero);
        }
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
  }
  copies_done();
  if (live && (q != stop || bp != end)) err |= QSGD_DEV_OVERRUN;      // a string must end exactly where the table says
  if (err) atomicOr(p.status, err);
}

}  // namespace

int launch_elias_dense(const FieldParams& f, bool fused, cudaStream_t stream) {
  static KernelSite site[8];
  DenseParams p;
  p.peers = f.peers; p.K = f.K; p.n = f.n; p.d = f.d; p.s = f.s; p.B = f.B; p.out = f.out; p.c = f.c;
  p.status = f.status; p.map = f.map; p.minus_zero = f.minus_zero;
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
  constexpr uint32_t kOwn = 3072u;                 // static shared memory, what CUDA reserves, alignment
  const uint32_t in_front = (kTableAt - kOwn) / p.warp_bytes;
  p.in_front = in_front;
  uint32_t warps = in_front + ((uint32_t)most_shared - kOwn - kTableEnd) / p.warp_bytes;
  if (warps > kMaxWarps) warps = kMaxWarps;
  // one run of consecutive buckets per lane group, all of the same length, in one wave
  const uint64_t groups = (uint64_t)sms * warps * G;
  p.run = (uint32_t)((p.B + groups - 1) / groups);
  const uint64_t need = (p.B + (uint64_t)p.run * G - 1) / ((uint64_t)p.run * G);      // warps with work
  const uint32_t per_sm = (uint32_t)((need + sms - 1) / sms);
  if (per_sm < warps) warps = per_sm;
  p.work = warps;
  const size_t smem = kTableEnd + (size_t)(warps > in_front ? warps - in_front : 0u) * p.warp_bytes;
  const bool byte = p.s > 15u, one = G == 1u;
  void (*kern)(DenseParams);
  if (one) {
    if (byte) kern = fused ? decode_elias_dense_kernel<true, true, 4> : decode_elias_dense_kernel<false, true, 4>;
    else kern = fused ? decode_elias_dense_kernel<true, false, 4> : decode_elias_dense_kernel<false, false, 4>;
  } else {
    if (byte) kern = fused ? decode_elias_dense_kernel<true, true, 8> : decode_elias_dense_kernel<false, true, 8>;
    else kern = fused ? decode_elias_dense_kernel<true, false, 8> : decode_elias_dense_kernel<false, false, 8>;
  }
  KernelSite& here = site[(one ? 4 : 0) + (byte ? 2 : 0) + (fused ? 1 : 0)];
  st = here.dynamic_begins_within(kern, kOwn - 256u);            // (and up to 256 bytes to the next multiple)
  if (!st) st = here.lookup_dynamic(kern, (int)kMaxWarps * 32, smem, &sms, &occ);
  if (st) return st;
  ScopedKernel sk(kKernDecodeEliasDense, stream);
  return (int)launch_chained(kern, (uint32_t)((need + warps - 1) / warps), kMaxWarps * 32u, smem, stream, p);
}

}  // namespace qsgd
