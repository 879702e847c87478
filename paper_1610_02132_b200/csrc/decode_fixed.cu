// Decode-and-aggregate, fixed-width path, optionally fused with the SGD step (Algorithm 1:
// g^l <- Decode(M^l); x <- x - (eta / K) * sum_l g^l).
//
// A warp owns chunks of 512 consecutive coordinates, a lane 16 of them, and walks the K
// messages in ascending k, so every coordinate's sum has the fixed order ((0 + g^0) + g^1) ...
// With K = 16 peers there are only a handful of issue slots per (peer, coordinate) at HBM
// speed, so reconstruction A * (level / s) * sign is a table lookup:
//   * s <= 15: the 2 * (s + 1) possible values +-A * (level / s) of one (peer, bucket) live one
//     per lane and are fetched with a warp shuffle indexed by "sign | level"; the sign bits are
//     spread next to the level nibbles with one multiply per four coordinates;
//   * s >= 16: +-(level / s) (correctly rounded) comes from a shared-memory table replicated per
//     lane (bank-conflict free), at an address that one byte permute makes of level and sign.
//
// What bounds it (n = 60 M, d = 512, K = 16): at s = 15 the L1 data path (one shuffle per coordinate and peer: 256 of 400
// wavefronts per chunk) and the latency of the loads, 221 us; at s = 255 HBM, 88 % of the copy rate. Sums in pairs, one scale
// read by all lanes instead of shuffled, places in 32 bits, `out` accessed in whole lines and the table with signs took 1489 to
// 1272 warp instructions per chunk (s = 15) and 1900 to 1488 (s = 255): 251 -> 221 and 340 -> 263 us. Four messages are read
// at a time (2: 252, 3: 236, 8 with 80 registers: 234 us at s = 15). More bytes in flight did not help: the next group read
// while this one is added 252 to 270 (spills, or fewer warps), fields copied to shared memory a group ahead 235 (their
// wavefronts), a ring of bulk copies per CTA 310 (warps that wait for the slowest), the next chunk prefetched to L2 240.
#include "decode_common.cuh"

namespace qsgd {

namespace {

constexpr int kThreads = 256;
constexpr int kChunk = 512;            // coordinates per warp iteration

struct DecodeParams {
  const uint8_t* msg[QSGD_MAX_PEERS];   // the K messages; all share one layout, so the three regions
  uint64_t off_sign, off_level;         // of every message sit at the same byte offsets
  uint32_t K;
  uint64_t n;
  uint32_t d;
  uint32_t s;
  uint32_t log2_chunks_per_bucket;   // SINGLE
  float* out;      // acc (overwritten) or x (updated in place)
  float c;         // eta / K (fused only)
  float minus_zero;   // -0 that the compiler cannot see (add_product2)
  uint32_t chunks;
  BucketMap map;
};

template <int LB> struct Shape {                     // 64 registers a thread
  static constexpr int kMostThreads = LB == 8 ? 1024 : 256, kCtas = LB == 8 ? 1 : 4;
};
// LB = 8: the table of level / s, and its place in the window of shared memory (a multiple of 64 KB: add_peer_tab)
constexpr uint32_t kTableBytes = 65536u, kTableAt = 65536u;
constexpr uint32_t kTurn = kChunk * 4u;              // bytes per warp to turn sums round
constexpr uint32_t kGroup = 4;                       // messages read at a time

// What a lane has of one message for its 16 coordinates.
template <int LB> struct Fields {
  static constexpr int kWords = LB == 8 ? 4 : LB == 4 ? 2 : 1;
  uint32_t w[kWords];
  uint32_t sb;
  float A;
};

template <int LB, bool FUSED, bool SINGLE>
__global__ void __launch_bounds__(Shape<LB>::kMostThreads, Shape<LB>::kCtas) decode_fixed_kernel(const __grid_constant__ DecodeParams p) {
  extern __shared__ __align__(128) uint8_t fixed_shared[];
  const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, warps = blockDim.x >> 5;
  const uint32_t turn = (LB == 8 ? kTableAt + kTableBytes : (uint32_t)__cvta_generic_to_shared(fixed_shared)) + warp * kTurn;
  float lut0 = 0.f;                                  // this lane's +-(level / s)
  const float sf = (float)p.s;
  if (LB == 8) {
    // every level's quotient by one lane, then handed round (by all lanes of all warps it was 0.3 us of a small decode)
    const uint32_t per = 256u / warps;               // 8, 16 or 32 levels a warp
    const float mine = __fdiv_rn((float)(warp * per + (lane & (per - 1u))), sf);
    for (uint32_t j = 0; j < per; ++j) {
      const float q = shfl_f(mine, j);
      const uint32_t at = kTableAt + (warp * per + j) * 256u + lane * 4u;
      asm volatile("st.shared.f32 [%0], %1;" ::"r"(at), "f"(q) : "memory");
      asm volatile("st.shared.f32 [%0], %1;" ::"r"(at + 128u), "f"(-q) : "memory");
    }
  } else {
    const uint32_t level = lane & ((1u << LB) - 1u), neg = (lane >> LB) & 1u;
    const float q = __fdiv_rn((float)level, sf);
    lut0 = neg ? -q : q;
  }
  if (LB == 8) __syncthreads();
  chain_wait();                                      // the messages come from the kernels ahead

  // Eight warps at a time take neighbouring chunks (they share sectors of the scales); CTAs with more take the next eight from
  // behind all CTAs' first, so that what is left for the last round lies on all SMs (n = 2.8 M, s = 100, K = 32 43 -> 34 us).
  const uint32_t stride = gridDim.x * warps, last_slot = (uint32_t)((p.n - 1) >> 4);
  for (uint32_t ch = ((warp >> 3) * gridDim.x + blockIdx.x) * 8u + (warp & 7u); ch < p.chunks; ch += stride) {
    // places of this lane's fields in any message (lanes past n read the last fields again)
    const uint32_t slot = min(ch * (kChunk / 16) + lane, last_slot);
    const uint32_t b = SINGLE ? ch >> p.log2_chunks_per_bucket : slot / (p.d >> 4);
    const uint32_t off_a = 4u * b, off_s = 2u * slot, off_l = (uint32_t)(2 * LB) * slot;       // n <= 2^32: below 2^32
    auto read = [&](Fields<LB>& to, uint32_t k) {
      const uint8_t* m = p.msg[k];
      to.A = __ldg(reinterpret_cast<const float*>(m + off_a));
      to.sb = __ldg(reinterpret_cast<const uint16_t*>(m + p.off_sign + off_s));
      const uint8_t* l = m + p.off_level + off_l;
      constexpr int W = Fields<LB>::kWords;
      if (LB == 8) {
        const uint4 t = __ldg(reinterpret_cast<const uint4*>(l));
        to.w[0] = t.x; to.w[1 % W] = t.y; to.w[2 % W] = t.z; to.w[3 % W] = t.w;
      } else if (LB == 4) {
        const uint2 t = __ldg(reinterpret_cast<const uint2*>(l));
        to.w[0] = t.x; to.w[1 % W] = t.y;
      } else if (LB == 2) {
        to.w[0] = __ldg(reinterpret_cast<const uint32_t*>(l));
      } else {
        to.w[0] = __ldg(reinterpret_cast<const uint16_t*>(l));
      }
    };
    float2p acc[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) acc[e] = 0ull;
    auto add = [&](const Fields<LB>& f) {
      if (LB == 8) add_peer_tab(acc, f.w, f.sb, lane, f.A, p.minus_zero);
      else add_peer_lut<LB, SINGLE>(acc, f.w, f.sb, SINGLE ? __fmul_rn(f.A, lut0) : lut0, f.A, p.minus_zero);
    };
    uint32_t k = 0;
    for (; k + kGroup <= p.K; k += kGroup) {
      Fields<LB> f[kGroup];
#pragma unroll
      for (uint32_t u = 0; u < kGroup; ++u) read(f[u], k + u);
#pragma unroll
      for (uint32_t u = 0; u < kGroup; ++u) add(f[u]);
    }
    if constexpr (LB <= 2 || (LB == 8 && !SINGLE)) {
      if (k < p.K) {                                 // the last one to three, side by side as well
        Fields<LB> f[kGroup - 1];
#pragma unroll
        for (uint32_t u = 0; u < kGroup - 1u; ++u)
          if (u == 0u || k + u < p.K) read(f[u], k + u);
#pragma unroll
        for (uint32_t u = 0; u < kGroup - 1u; ++u)
          if (u == 0u || k + u < p.K) add(f[u]);
      }
    } else {                                         // (side by side, these cost the loop above registers: 2 to 18 %)
      for (; k < p.K; ++k) {
        Fields<LB> f;
        read(f, k);
        add(f);
      }
    }
    store_chunk16<FUSED, SINGLE>(p.out, p.map, acc, turn, ch, p.log2_chunks_per_bucket, p.d, p.n, p.c, lane);
  }
}

__global__ void __launch_bounds__(kThreads) sgd_step_kernel(float* __restrict__ x,
                                                           const float* __restrict__ acc, float c,
                                                           uint64_t n) {
  const uint64_t i0 = ((uint64_t)blockIdx.x * kThreads + threadIdx.x) * 4;
  chain_wait();
  if (i0 + 4 <= n) {
    const float4 a = __ldcs(reinterpret_cast<const float4*>(acc + i0));
    float4 v = *reinterpret_cast<const float4*>(x + i0);
    v.x = __fsub_rn(v.x, __fmul_rn(c, a.x));
    v.y = __fsub_rn(v.y, __fmul_rn(c, a.y));
    v.z = __fsub_rn(v.z, __fmul_rn(c, a.z));
    v.w = __fsub_rn(v.w, __fmul_rn(c, a.w));
    *reinterpret_cast<float4*>(x + i0) = v;
  } else {
    for (uint64_t i = i0; i < n; ++i) x[i] = __fsub_rn(x[i], __fmul_rn(c, acc[i]));
  }
}

template <int LB, bool FUSED, bool SINGLE>
int launch_one(const DecodeParams& p, cudaStream_t stream) {
  static KernelSite site;
  auto kern = decode_fixed_kernel<LB, FUSED, SINGLE>;
  int sms = 0, occ = 0, st = 0;
  uint32_t warps = 8;
  size_t smem = warps * kTurn;
  if constexpr (LB == 8) {
    st = device_sms(&sms);
    if (!st) st = site.dynamic_begins_within(kern, kTableAt);
    if (st) return st;
    while (warps < Shape<LB>::kMostThreads / 32 && p.chunks > warps * (uint32_t)sms) warps *= 2;
    smem = kTableAt + kTableBytes + warps * kTurn;
    st = site.lookup_dynamic(kern, (int)warps * 32, smem, &sms, &occ);
  } else {
    st = site.lookup(kern, (int)warps * 32, smem, &sms, &occ);
  }
  if (st) return st;
  const uint32_t want = (p.chunks + warps - 1) / warps, cap = (uint32_t)(sms * occ);
  ScopedKernel sk(kKernDecodeFixed, stream);
  return (int)launch_chained(kern, want < cap ? want : cap, warps * 32u, smem, stream, p);
}

template <int LB>
int launch_lb(const DecodeParams& p, bool fused, bool single, cudaStream_t stream) {
  if (fused) return single ? launch_one<LB, true, true>(p, stream) : launch_one<LB, true, false>(p, stream);
  return single ? launch_one<LB, false, true>(p, stream) : launch_one<LB, false, false>(p, stream);
}

}  // namespace

int launch_decode_fixed(const PeerSet& peers, uint32_t K, uint64_t n, uint32_t d, uint32_t s,
                        float* acc_or_x, bool fused, float eta, const BucketMap& map, cudaStream_t stream) {
  DecodeParams p;
  const FixedLayout L = make_fixed_layout(n, d, s);
  for (uint32_t k = 0; k < K; ++k) p.msg[k] = reinterpret_cast<const uint8_t*>(peers.A[k]);   // the scales open a message
  p.off_sign = L.off_sign; p.off_level = L.off_level;
  p.K = K; p.n = n; p.d = d; p.s = s; p.out = acc_or_x; p.map = map;
  p.c = eta / (float)K;
  p.minus_zero = -0.f;
  p.chunks = (uint32_t)((n + kChunk - 1) / kChunk);
  // one scale per chunk when the bucket size is 512 * 2^j
  const bool single = d >= (uint32_t)kChunk && (d & (d - 1)) == 0;
  p.log2_chunks_per_bucket = 0;
  for (uint32_t t = d / kChunk; single && t > 1; t >>= 1) ++p.log2_chunks_per_bucket;
  switch (level_bits_for(s)) {
    case 1: return launch_lb<1>(p, fused, single, stream);
    case 2: return launch_lb<2>(p, fused, single, stream);
    case 4: return launch_lb<4>(p, fused, single, stream);
    default: return launch_lb<8>(p, fused, single, stream);
  }
}

int launch_sgd_step(float* x, const float* acc, float eta, uint32_t K, uint64_t n,
                    cudaStream_t stream) {
  const float c = eta / (float)K;
  const uint64_t quads = (n + 3) / 4;
  const uint32_t grid = (uint32_t)((quads + kThreads - 1) / kThreads);
  {
    ScopedKernel sk(kKernSgdStep, stream);
    const cudaError_t e = launch_chained(sgd_step_kernel, grid, kThreads, 0, stream, x, acc, c, n);
    if (e != cudaSuccess) return (int)e;
  }
  return (int)cudaGetLastError();
}

}  // namespace qsgd
