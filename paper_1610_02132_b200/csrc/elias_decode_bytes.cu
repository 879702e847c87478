// Decode-and-aggregate, Elias path (Code_s, s <= 15, at most 32 peers): a lane per string, the bucket walked in ranges
// of at most 256 positions. (Section 3.1 for the string, Appendix A.2 for the integer code, Algorithm 1 for the sum and
// the step.) It stands between the teams, whose strings are few, and the ring reader, whose tables and rings take long to
// set up and which finds little to read in a round where strings are short; the lines are in elias_decode.cu.
//
// The lanes of a warp read G = 32 / Kpad buckets, K strings each. A lane writes one byte per nonzero -- level |
// negative << 4, the lane index of +-(level / s) in a shuffle table -- into its row, which holds one range, and
// keeps its place in its string between ranges (bit window, position, one entry that lies past the range). Then the
// warp adds the rows up in ascending k, 8 coordinates a lane. The sum's shuffles and the rows are shared-memory
// traffic, which is what bounds it; the table of gaps is small so that many warps are resident (20 to 24 an SM).
#include "elias_decode.cuh"

namespace qsgd {

namespace {

constexpr uint32_t kRange = 256;                       // positions
constexpr uint32_t kPad = 16;                          // bytes between rows: lanes at similar positions use other banks
constexpr uint32_t kGapBits = 12;

struct Tables {
  uint16_t gap[1u << kGapBits];   // value | length << 8 of the code that the next 12 bits start with, 0: none is complete
  uint16_t tail[256];             // level | negative << 4 | length << 8 of the sign and level in the next 8 bits, or 0
};

__device__ __forceinline__ void fill_tables(Tables& tab, uint32_t s) {
  for (uint32_t i = threadIdx.x; i < (1u << kGapBits); i += blockDim.x) {
    uint32_t v, len;
    const bool ok = elias_from_window(i << (32u - kGapBits), v, len) && len <= kGapBits;
    tab.gap[i] = ok ? (uint16_t)(v | len << 8) : (uint16_t)0;
  }
  for (uint32_t i = threadIdx.x; i < 256u; i += blockDim.x) {
    uint32_t level, len;
    const bool ok = elias_from_window(i << 25, level, len) && len <= 7u && level <= s && level <= 15u;
    tab.tail[i] = ok ? (uint16_t)(level | (i >> 7) << 4 | (len + 1u) << 8) : (uint16_t)0;
  }
}

struct BytesParams {
  PeerSet peers;
  uint32_t K;
  uint32_t Kpad;          // lanes per bucket: K rounded up to a power of two
  uint32_t G;             // buckets per warp
  uint32_t R;             // positions per range
  uint32_t warp_bytes;    // G * K rows of R + kPad bytes, 32 scales
  uint64_t n;
  uint32_t d;
  uint32_t s;
  uint64_t B;
  float* out;             // acc (overwritten) or x (updated in place)
  float c;                // eta / K
  float minus_zero;       // add_product2
  uint32_t* status;
  Regime when;
  BucketMap map;
};

struct Lane {
  BitSrc src;
  uint32_t used, total, at, err;
  uint32_t pend;          // entry that the last range had no place for (position | code << 16), or kNoEntry
};

// Reads on in a lane's string, up to the first entry at or past `lim` <= db, which is kept.
__device__ __forceinline__ void read_range(const Tables& tab, Lane& st, uint32_t rbeg, uint32_t lim, uint32_t db, uint32_t s,
                                           uint8_t* row) {
  if (st.pend != kNoEntry) {
    if ((st.pend & 0xFFFFu) >= lim) return;
    row[(st.pend & 0xFFFFu) - rbeg] = (uint8_t)(st.pend >> 16);
    st.pend = kNoEntry;
  }
  while (st.used < st.total) {
    st.src.refill();                                   // >= 33 bits: gap, sign and level by table take at most 20
    uint32_t gap, l1, l2;
    const uint32_t e1 = tab.gap[st.src.hi >> (32u - kGapBits)];
    if (e1) {
      gap = e1 & 0xFFu;
      l1 = e1 >> 8;
    } else {
      const bool ok = elias_from_window(st.src.hi, gap, l1);
      st.src.drop(l1);
      st.used += l1;
      if (!ok) { st.err = QSGD_DEV_OVERRUN; return; }
      st.src.refill();
      l1 = 0;
    }
    const uint32_t w = __funnelshift_lc(st.src.lo, st.src.hi, l1);
    const uint32_t e2 = tab.tail[w >> 24];
    if (e2 == 0u) {                                    // no level <= min(s, 15)
      uint32_t level;
      st.err = elias_from_window(w << 1, level, l2) && level > s ? QSGD_DEV_LEVEL : QSGD_DEV_OVERRUN;
      return;
    }
    l2 = e2 >> 8;
    st.src.drop(l1 + l2);
    st.used += l1 + l2;
    st.at += gap;
    if (st.at >= lim) {                                // a later range's, or past the bucket
      if (st.at < db) st.pend = st.at | (e2 & 0x1Fu) << 16;
      else st.err = QSGD_DEV_POSITION;
      return;
    }
    row[st.at - rbeg] = (uint8_t)(e2 & 0x1Fu);
  }
}

// SINGLE: a pass of 32 lanes x 8 coordinates stays inside one bucket (d a multiple of 256): the shuffle table is scaled
// once per peer instead of every value.
template <bool FUSED, bool SINGLE>
__global__ void __launch_bounds__(512) decode_elias_bytes_kernel(const __grid_constant__ BytesParams p) {
  extern __shared__ __align__(16) uint8_t bsm[];
  __shared__ Tables tab;
  chain_wait();                                   // the messages come from the kernels ahead
  if (p.when.hi != kNoBound && !mean_below(p.when.hi, p.peers, p.K, p.B)) return;
  if (p.when.lo && mean_below(p.when.lo, p.peers, p.K, p.B)) return;
  const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  fill_tables(tab, p.s);
  __syncthreads();
  float lut0;
  {
    const float q = __fdiv_rn((float)(lane & 15u), (float)p.s);
    lut0 = lane & 16u ? -q : q;
  }
  uint8_t* mine = bsm + (size_t)warp * p.warp_bytes;
  const uint32_t K = p.K, G = p.G, Kpad = p.Kpad, row_bytes = p.R + kPad, rows_bytes = G * K * row_bytes;
  float* scales = reinterpret_cast<float*>(mine + rows_bytes);
  const uint32_t pg = lane / Kpad, pk = lane % Kpad;           // reads: bucket in group, peer
  uint8_t* row = mine + (pg * K + pk) * row_bytes;             // this lane's row (when it reads)
  const uint64_t groups = (p.B + G - 1) / G;

  for (uint64_t grp = (uint64_t)blockIdx.x * nwarps + warp; grp < groups; grp += (uint64_t)gridDim.x * nwarps) {
    const uint64_t b0 = grp * G;
    Lane st;
    st.used = st.total = st.err = 0u;
    st.at = 0xFFFFFFFFu;
    st.pend = kNoEntry;
    uint32_t db = 0;
    float A = 0.f;
    if (b0 + pg < p.B) db = (uint32_t)min((uint64_t)p.d, p.n - (b0 + pg) * p.d);
    const bool reads = db != 0u && pk < K;
    if (reads) {
      const StringRef ref = string_ref(p.peers, pk, b0 + pg, p.B, db);
      st.err = ref.err;
      if (!ref.err) {
        st.total = ref.total;
        st.src.open(ref.words, ref.lo);
        A = __uint_as_float(st.src.take(32));
      }
    }
    scales[lane] = A;

    for (uint32_t rbeg = 0; rbeg < p.d; rbeg += p.R) {
      const uint32_t rend = min(rbeg + p.R, p.d);
      for (uint32_t q = lane; q < (rows_bytes >> 4); q += 32) reinterpret_cast<uint4*>(mine)[q] = make_uint4(0u, 0u, 0u, 0u);
      __syncwarp();
      if (reads && st.err == 0u) read_range(tab, st, rbeg, min(rend, db), db, p.s, row);
      __syncwarp();
      // ---- ascending-k sums; a lane takes 8 coordinates per pass ------------------------------------
      const uint32_t slots_per_bucket = (rend - rbeg) >> 3, slots = G * slots_per_bucket;
      for (uint32_t s0 = 0; s0 < slots; s0 += 32) {
        const uint32_t slot = s0 + lane;
        const uint32_t g = slot / slots_per_bucket, cl = (slot - g * slots_per_bucket) << 3, c = rbeg + cl;
        const uint64_t b = b0 + g;
        const bool there = slot < slots;                       // a lane past the end still holds its share of the table
        const bool live = there && b < p.B && b * p.d + c < p.n;
        const uint32_t gg = there ? g : 0u;
        const uint8_t* rows = mine + gg * K * row_bytes + cl;
        const float* sc = scales + gg * Kpad;
        float2p sum[4] = {0ull, 0ull, 0ull, 0ull};
#pragma unroll 4
        for (uint32_t k = 0; k < K; ++k) {
          const uint2 cw = there ? *reinterpret_cast<const uint2*>(rows + k * row_bytes) : make_uint2(0u, 0u);
          const float Ak = sc[k];
          const float lutk = SINGLE ? __fmul_rn(Ak, lut0) : lut0;
#pragma unroll
          for (int e = 0; e < 8; e += 2) {
            const uint32_t w = (e < 4 ? cw.x : cw.y) >> (8 * (e & 3));
            sum[e / 2] = add_pair_lut<SINGLE>(sum[e / 2], w, w >> 8, lutk, Ak, p.minus_zero);
          }
        }
        float acc[8];
#pragma unroll
        for (int e = 0; e < 4; ++e) { const float2 u = unpair2(sum[e]); acc[2 * e] = u.x; acc[2 * e + 1] = u.y; }
        if (live) store_span8<FUSED>(out_span(p.out, p.map, b, c, p.d, p.n, 8u), acc, p.c);
      }
      __syncwarp();
    }
    if (reads && st.err == 0u && st.used != st.total) st.err = QSGD_DEV_OVERRUN;      // it must end exactly where the table says
    if (st.err) atomicOr(p.status, st.err);
    __syncwarp();
  }
}

}  // namespace

int launch_elias_bytes(const FieldParams& f, bool fused, cudaStream_t stream) {
  static KernelSite site[4];
  BytesParams p;
  p.peers = f.peers; p.K = f.K; p.n = f.n; p.d = f.d; p.s = f.s; p.B = f.B; p.out = f.out; p.c = f.c;
  p.status = f.status; p.when = f.when; p.map = f.map; p.minus_zero = f.minus_zero;
  p.Kpad = 1;
  while (p.Kpad < p.K) p.Kpad <<= 1;
  p.G = 32u / p.Kpad;
  p.R = p.d <= kRange ? p.d : kRange;
  p.warp_bytes = p.G * p.K * (p.R + kPad) + 128u;
  // Warps per CTA: the count that leaves the most warps resident on an SM (the tables are per CTA).
  const uint32_t per_cta = sizeof(Tables) + 1024u, per_sm = 227u << 10;
  uint32_t warps = 1, best = 0;
  for (uint32_t w = 1; w <= 16; ++w) {
    const uint32_t resident = per_sm / (w * p.warp_bytes + per_cta) * w;
    if (resident > best) { best = resident; warps = w; }
  }
  const bool single = (p.d & 255u) == 0u;
  void (*kern)(BytesParams);
  if (fused) kern = single ? decode_elias_bytes_kernel<true, true> : decode_elias_bytes_kernel<true, false>;
  else kern = single ? decode_elias_bytes_kernel<false, true> : decode_elias_bytes_kernel<false, false>;
  const size_t smem = (size_t)warps * p.warp_bytes;
  int sms = 0, occ = 0;
  const int st = site[(fused ? 1 : 0) + (single ? 2 : 0)].lookup_dynamic(kern, (int)warps * 32, smem, &sms, &occ);
  if (st) return st;
  const uint64_t groups = (p.B + p.G - 1) / p.G, want = (groups + warps - 1) / warps, cap = (uint64_t)sms * occ;
  ScopedKernel sk(kKernDecodeEliasBytes, stream);
  return (int)launch_chained(kern, (uint32_t)(want < cap ? want : cap), warps * 32u, smem, stream, p);
}

}  // namespace qsgd
