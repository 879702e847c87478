// Decode-and-aggregate, Elias path (Code_s, s <= 15, at most 32 peers), where strings are many: a lane per
// (run of consecutive buckets, peer). (Section 3.1, end of "Efficient Coding of Gradients", for the string;
// Appendix A.2 for the integer code; Algorithm 1 for the sum and the step.)
//
// A peer's strings of consecutive buckets are one stretch of its payload, so a lane reads one stream from
// end to end, by background copies of 16 bytes into its own 64 bytes of shared memory: a load into a register
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
// on what was read but data: lanes with different codes stay together. What no table entry covers -- a gap
// of 64 or more, a malformed code -- is read by the definition's decoder (slow_entry).
#include "elias_decode.cuh"

namespace qsgd {

namespace {

constexpr uint32_t kBits = 12;                         // stream bits per lookup
constexpr uint32_t kTabWords = 1u << kBits;            // entries per state
constexpr uint32_t kStateBit = 4u << kBits;            // byte offset of the second state's table: also its bit in an entry
constexpr uint32_t kRing = 256;                        // positions (bytes) per lane
constexpr uint32_t kMostAdvance = 63;                  // positions per entry of the table
constexpr uint32_t kChunks = 4;                        // 16-byte pieces of the stream that a lane has in shared memory
constexpr uint32_t kStage = 16u * kChunks;             // bytes of them
constexpr int32_t kAhead = 128;                        // bits (one piece) that have to be there for a round of the burst
constexpr uint32_t kMaxWarps = 20;

// Table entry: bits 0-3 stream bits used (0: nothing here for the table), 4-8 first byte, 9-13 second byte (what
// stands above either is ignored by the shuffles), kStateBit next state, byte 2 place of the first byte, 26-31
// place of the second = how far the entry goes, both from the last position passed. Where there is no second
// byte its place is the first one's again, with the same value, or one that is still zero, with 0: both stores
// are always made. An entry for nothing puts its first byte, 0, in front of everything.
struct EntryBits {
  uint32_t used, c1, c2, next, p1, p2;
  __device__ __forceinline__ uint32_t pack() const {
    return used | c1 << 4 | c2 << 9 | (next ? kStateBit : 0u) | p1 << 16 | p2 << 26;
  }
};

// Sign and level at the top of w, `room` bits of which are there: level | negative << 4, and its length (0: none).
__device__ __forceinline__ uint32_t tail_at(uint32_t w, uint32_t room, uint32_t s, uint32_t* len) {
  uint32_t level, ll;
  const bool ok = elias_from_window(w << 1, level, ll) && 1u + ll <= room && level <= s;
  *len = ok ? 1u + ll : 0u;
  return (level & 15u) | (w >> 31) << 4;
}

__device__ __forceinline__ uint32_t ring_entry(uint32_t i, bool tail_first, uint32_t s) {
  uint32_t w = i << (32u - kBits), room = kBits;
  EntryBits e{0u, 0u, 0u, tail_first ? 1u : 0u, 0u, 0u};
  const uint32_t stuck = (tail_first ? kStateBit : 0u) | 1u << 16;
  uint32_t gap = 1, len;
  if (!tail_first) {
    if (!elias_from_window(w, gap, len) || len > room || gap > kMostAdvance) return stuck;
    w <<= len; room -= len; e.used = len;
    uint32_t tl;
    tail_at(w, room, s, &tl);
    if (tl == 0u) {                                    // a gap alone: stop in front of its position
      if (gap == 1u) return stuck;
      e.next = 1u; e.p1 = gap; e.p2 = gap - 1u;
      return e.pack();
    }
  }
  e.c1 = tail_at(w, room, s, &len);
  if (len == 0u) return stuck;
  w <<= len; room -= len; e.used += len;
  e.next = 0u; e.p1 = gap; e.p2 = gap; e.c2 = e.c1;
  uint32_t gap2;
  if (!elias_from_window(w, gap2, len) || len > room || gap + gap2 > kMostAdvance) return e.pack();
  w <<= len; room -= len;
  uint32_t tl;
  const uint32_t c2 = tail_at(w, room, s, &tl);
  e.used += len;
  if (tl) {
    e.used += tl; e.c2 = c2; e.p2 = gap + gap2;
  } else {                                             // the second gap alone
    e.next = 1u; e.p2 = gap + gap2 - 1u;
    if (gap2 > 1u) e.c2 = 0u;
  }
  return e.pack();
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
  float minus_zero;       // -0
  uint32_t* status;
  uint32_t run;           // buckets per run
  uint32_t step;          // positions added up at a time: 64 or 128
  uint32_t slots;         // scales kept per lane, a power of two: the buckets that a ring can touch
  uint32_t warp_bytes;
  uint32_t defer_sparse;  // a sparse-regime kernel was launched beside this one
  BucketMap map;
};

__device__ __forceinline__ uint32_t shared_address(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void store_byte(uint32_t addr, uint32_t v) {
  asm volatile("st.shared.u8 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}
__device__ __forceinline__ uint32_t load_word(uint32_t addr) {
  uint32_t v;
  asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
  return v;
}
// 16 bytes from global to shared memory, in the background; and the wait for all of this thread's.
__device__ __forceinline__ void copy16(uint32_t addr, const void* from) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(addr), "l"(from) : "memory");
}
__device__ __forceinline__ void copies_done() { asm volatile("cp.async.wait_all;" ::: "memory"); }
__device__ __forceinline__ void zero_quad(uint32_t addr) {
  asm volatile("st.shared.v4.u32 [%0], {%1, %1, %1, %1};" ::"r"(addr), "r"(0) : "memory");
}

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

__device__ __forceinline__ unsigned long long pack2(float a, float b) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
// Two products and two sums, each rounded to nearest. The product is an fma with -0 that the compiler cannot see
// (`m0`, from the kernel's parameters): a mul.rn.f32x2 in front of an add.rn.f32x2 was contracted.
__device__ __forceinline__ void add_mul2(unsigned long long& acc, unsigned long long a, unsigned long long b,
                                         unsigned long long m0) {
  unsigned long long t;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(t) : "l"(a), "l"(b), "l"(m0));
  asm("add.rn.f32x2 %0, %0, %1;" : "+l"(acc) : "l"(t));
}
