// Encode, Elias path (Section 3.1 "Efficient Coding of Gradients", string S; Appendix A.3 for
// the dense variant). Pipeline on one stream:
//   1. quantize into the fixed-width layout held in the workspace (quantize_fixed.cu);
//   2. string length L_b of every bucket, the sum of the lengths of each CTA's run of consecutive
//      buckets, and by atomic additions the sum of each group of kSumGroup CTAs (elias_length_kernel);
//   3. each CTA of the scatter kernel adds up the sums in front of its run (find_start), derives the
//      bit offsets of its own buckets, writes their
//      offset-table entries, assembles its run of strings in shared memory (lanes own
//      consecutive sub-ranges of a bucket; bits of neighbouring lanes and buckets meet inside
//      words and are merged with shared-memory atomics) and flushes whole words to the payload
//      with coalesced stores (flush_run).
// A bucket is handled by a team of d / 64 lanes (at most a warp, at least one lane), so that the
// sequential walk over a lane's nonzeros is long enough to amortise the team's scans. Levels above 15 go by tiles, a
// thread with 16 coordinates, in the dense code and in the longest buckets (use_tiles), and small problems are quantized and
// measured in one kernel (elias_encode_small.cu).
//
// What bounds them (n = 34 M, d = 512, s = 15, a mixture of two scales): both the integer pipe, 79 % (length, 16.5 us) and 65 %
// (scatter, 31 us, of which half is the walk over the nonzeros of the lane that has most). Without a scan by the CTA that draws
// the last ticket, for which every CTA waited at its end: length 20.7 -> 16.5. Code words from bit 31 down with their length
// beside them, sign included, level words where a lane can index them: scatter 361 -> 303 warp instructions per bucket,
// 34.3 -> 30.8; whole encode at 60 M 152 -> 137, at 17 M, d = 4096, s = 64, dense code, 85 -> 60.
#include <mutex>

#include "elias_encode.cuh"

namespace qsgd {

namespace {

using namespace elias;

// ---- 2. string length per bucket, sums per CTA and per group of CTAs ------------------------------------
template <int LB, bool DENSE>
__global__ void __launch_bounds__(kThreads) elias_length_kernel(const BucketParams p,
                                                                uint32_t* __restrict__ len,
                                                                uint32_t* __restrict__ lane_rec,
                                                                uint32_t* __restrict__ cta_sums, uint64_t* group_sums) {
  __shared__ uint32_t warp_sum[kWarps];
  __shared__ uint32_t tab[17];
  __shared__ SymbolLengths<DENSE ? LB : 1> lengths;
  fill_code_table(tab);
  if (DENSE) fill_symbol_lengths<DENSE ? LB : 1>(lengths);
  __syncthreads();
  chain_wait();                                    // the fields come from the kernel ahead
  const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t tl = lane & (p.lpb - 1), team = lane / p.lpb, bpw = 32 / p.lpb;
  const uint64_t b = (uint64_t)blockIdx.x * p.nbc + warp * bpw + team;
  const bool live = b < p.B;
  const uint64_t base = live ? b * p.d : 0;
  const uint32_t db = live ? (uint32_t)min((uint64_t)p.d, p.n - base) : 0;
  const uint32_t c_lo = min(tl * p.seg, db), c_hi = min(c_lo + p.seg, db);
  const uint32_t* lwb = p.level + ((base * LB) >> 5);            // the bucket's first level word
  int32_t prev;
  const uint32_t bits = lane_bits<LB, DENSE>(tab, lengths, lwb, p.lpb, c_lo, c_hi, tl, live, &prev);
  if (live) lane_rec[b * p.lpb + tl] = bits | ((uint32_t)(prev + 1) << 16);   // reused by the scatter
  const uint32_t L = team_sum(bits, p.lpb);
  if (live && tl == 0) len[b] = L;
  const uint32_t w = __reduce_add_sync(0xffffffffu, tl == 0 ? L : 0u);        // one contribution per bucket
  if (lane == 0) warp_sum[warp] = w;
  __syncthreads();
  if (threadIdx.x == 0) {
    uint32_t s = 0;
#pragma unroll
    for (int i = 0; i < kWarps; ++i) s += warp_sum[i];
    cta_sums[blockIdx.x] = s;
    add_to_groups(group_sums, s);
  }
}

// ---- 3. scatter ----------------------------------------------------------------------------------
struct ScatterArgs {
  BucketParams p;
  const uint32_t* len;
  const uint32_t* lane_rec;
  const uint32_t* cta_sums;
  const uint64_t* group_sums;
  uint8_t* out;
  size_t out_capacity;
  uint64_t* out_bits;
  uint32_t* status_dev;
};

template <int LB, bool DENSE>
__global__ void __launch_bounds__(kThreads) elias_scatter_kernel(const __grid_constant__ ScatterArgs a) {
  constexpr uint32_t kFields = 32u / LB, kMask = (1u << LB) - 1u, kWords = 2u * LB;      // of a block of 64 coordinates
  extern __shared__ uint32_t stage[];
  __shared__ uint32_t warp_sum[kWarps];
  __shared__ uint64_t start_s, total_s;
  __shared__ uint32_t tab[17];
  __shared__ CodeWords<LB, DENSE> words;
  __shared__ uint32_t column[DENSE || LB == 1 ? 1 : kWords * kThreads];       // a block's level words, for each thread its own
  const BucketParams& p = a.p;
  fill_code_table(tab);
  fill_code_words(words);
  chain_wait();                                    // lengths and sums come from the kernel ahead
  const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t tl = lane & (p.lpb - 1), team = lane / p.lpb, bpw = 32 / p.lpb;
  const uint64_t b = (uint64_t)blockIdx.x * p.nbc + warp * bpw + team;
  const bool live = b < p.B;
  const uint64_t base = live ? b * p.d : 0;
  const uint32_t db = live ? (uint32_t)min((uint64_t)p.d, p.n - base) : 0;
  const uint32_t c_lo = min(tl * p.seg, db), c_hi = min(c_lo + p.seg, db);

  const uint32_t span = __ldg(a.cta_sums + blockIdx.x);             // bits of this CTA's run
  if (warp == 0) find_start(a.cta_sums, a.group_sums, &start_s, &total_s);
  for (uint32_t j = threadIdx.x; j < (span + 62u) >> 5; j += kThreads) stage[j] = 0u;

  // bit offset of every bucket inside the CTA's run: scan of the bucket lengths
  const uint32_t L = (live && tl == 0) ? __ldg(a.len + b) : 0u;
  uint32_t inc = L;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t t = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= (uint32_t)o) inc += t;
  }
  if (lane == 31) warp_sum[warp] = inc;
  __syncthreads();                                                  // staging zeroed, sums and tables there
  const uint64_t start = start_s;
  const uint32_t lead = (uint32_t)(start & 31);                     // bits of the first word owned by the previous CTA
  uint64_t payload_bytes;
  if (!fix_geometry(total_s, p.B, a.out_capacity, a.out_bits, a.status_dev, blockIdx.x == 0, &payload_bytes)) return;
  uint32_t before = 0;
#pragma unroll
  for (int w = 0; w < kWarps; ++w) if ((uint32_t)w < warp) before += warp_sum[w];
  uint32_t bucket_off = before + inc - L;                           // valid in team lane 0
  bucket_off = __shfl_sync(0xffffffffu, bucket_off, (int)(lane - tl));
  if (live && tl == 0) {
    uint64_t* table = reinterpret_cast<uint64_t*>(a.out + payload_bytes);
    table[b] = start + bucket_off;
    if (b == p.B - 1) table[p.B] = start + bucket_off + L;
  }

  // this lane's first bit inside its bucket: scan of the lane lengths over the team
  const uint32_t* lwb = p.level + ((base * LB) >> 5);            // the bucket's first level word
  const uint32_t* swb = p.sign + (base >> 5);                    // ... and first sign word
  // this lane's share of the string and the nonzero before it were counted by the length kernel
  const uint32_t rec = live ? __ldg(a.lane_rec + b * p.lpb + tl) : 0u;
  const uint32_t bits = rec & 0xFFFFu;
  uint32_t linc = bits;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t t = __shfl_up_sync(0xffffffffu, linc, o);
    if ((uint32_t)o < p.lpb && tl >= (uint32_t)o) linc += t;
  }
  if (bits != 0) {
    StageWriter bw;
    bw.begin(stage, lead + bucket_off + (linc - bits));
    if (tl == 0) bw.put_word(__float_as_uint(__ldg(p.A + b)));
    uint32_t prev = (rec >> 16) - 1u;
    for (uint32_t c0 = c_lo; c0 < c_hi; c0 += 64u) {             // blocks of 64 coordinates
      const uint32_t* wp = lwb + ((c0 * LB) >> 5);
      uint32_t w[kWords];
#pragma unroll
      for (uint32_t j = 0; j < kWords; ++j) w[j] = c0 + j * kFields < c_hi ? __ldg(wp + j) : 0u;
      uint32_t s0 = __ldg(swb + (c0 >> 5)), s1 = (c0 + 32u < c_hi) ? __ldg(swb + (c0 >> 5) + 1) : 0u;
      if constexpr (DENSE) {
        const uint32_t left = c_hi - c0;
#pragma unroll
        for (uint32_t j = 0; j < kWords; ++j) {
          const uint32_t sg = (j * kFields) & 32u ? s1 : s0;
#pragma unroll
          for (uint32_t f = 0; f < kFields; ++f) {
            const uint32_t at = j * kFields + f;
            const uint32_t e = at < left ? words.level[((w[j] >> (f * LB)) & kMask) | ((sg >> (at & 31u)) & 1u) << LB] : 0u;
            bw.put_even(e & ~31u, e & 31u);
          }
        }
      } else {
        // the block's nonzero masks and signs sit in registers, its level words where they can be indexed
        uint32_t m0 = 0u, m1 = 0u;
#pragma unroll
        for (uint32_t j = 0; j < kWords; ++j) {
          const uint32_t m = nonzero_mask<LB>(w[j]);
          if (j * kFields < 32u) m0 |= m << (j * kFields & 31u);
          else m1 |= m << (j * kFields & 31u);
          if (LB != 1) column[j * kThreads + threadIdx.x] = w[j];
        }
        uint32_t half = c0;                                      // first coordinate of the half at hand
        const uint32_t* mine = column + threadIdx.x;
        while (m0 | m1) {
          if (m0 == 0u) {
            m0 = m1; m1 = 0u; s0 = s1;
            half = c0 + 32u;
            if (LB != 1) mine = column + threadIdx.x + LB * kThreads;
          }
          const uint32_t off = (uint32_t)__ffs((int)m0) - 1u, pos = half + off;
          m0 &= m0 - 1u;
          uint32_t idx = 1u;
          if (LB != 1) idx = __funnelshift_r(mine[off / kFields * kThreads], 0u, off * LB) & kMask;
          idx |= ((s0 >> off) & 1u) << LB;
          put_entry<LB>(bw, tab, words, pos - prev, idx);
          prev = pos;
        }
      }
    }
    bw.finish();
  }
  __syncthreads();
  const uint64_t next = (uint64_t)(blockIdx.x + 1u) * p.nbc;       // the next CTA's first bucket
  flush_run(reinterpret_cast<uint32_t*>(a.out) + (start >> 5), stage, lead, span, next >= p.B, p.A + next,
            (uint32_t)(payload_bytes / 4 - (start >> 5)));
}

// ---- 2. for tiles ----------------------------------------------------------------------------------
template <int LB, bool DENSE>
__global__ void __launch_bounds__(kThreads) elias_tile_length_kernel(const BucketParams p, uint32_t* tile_sums, uint64_t* group_sums) {
  __shared__ uint32_t slots[2][kWarps];
  __shared__ uint32_t tab[17];
  __shared__ SymbolLengths<DENSE ? LB : 1> lengths;
  fill_code_table(tab);
  if (DENSE) fill_symbol_lengths<DENSE ? LB : 1>(lengths);
  __syncthreads();
  chain_wait();                                    // the fields come from the kernel ahead
  const Piece<LB> q = load_piece<LB>(p);
  const uint32_t mask = DENSE ? 0u : piece_mask<LB>(q);
  const int32_t prev = DENSE ? -1 : nonzero_before<LB>(q, mask, slots[0]);
  const uint32_t mine = __reduce_add_sync(0xffffffffu, piece_bits<LB, DENSE>(tab, lengths, q, mask, prev));
  if ((threadIdx.x & 31) == 0) slots[1][threadIdx.x >> 5] = mine;
  __syncthreads();
  if (threadIdx.x == 0) {
    uint32_t s = 0;
#pragma unroll
    for (int i = 0; i < kWarps; ++i) s += slots[1][i];
    tile_sums[blockIdx.x] = s;
    add_to_groups(group_sums, s);
  }
}

template <int LB, bool DENSE>
int run_pipeline(BucketParams& bp, const EliasWs& w, uint32_t s, uint8_t* out, size_t out_capacity,
                 uint64_t* out_bits, uint32_t* status_dev, cudaStream_t stream) {
  if (use_tiles(bp.n, bp.d, s, DENSE)) {
    bp.lpb = 0; bp.seg = 16; bp.nbc = tile_buckets(bp.d);
    const uint32_t tiles = (uint32_t)((bp.B + bp.nbc - 1) / bp.nbc);
    {
      ScopedKernel sk(kKernEliasLength, stream);
      const cudaError_t e = launch_chained(elias_tile_length_kernel<LB, DENSE>, tiles, kThreads, 0, stream, bp, w.tile_sums, w.tile_groups);
      if (e != cudaSuccess) return (int)e;
    }
    return launch_tile_scatter(bp, w, s, DENSE, out, out_capacity, out_bits, status_dev, stream);
  }
  const Teams tm = make_teams(bp.d);
  bp.lpb = tm.lpb; bp.seg = tm.seg; bp.nbc = tm.nbc;
  const uint64_t ctas = (bp.B + tm.nbc - 1) / tm.nbc;
  {
    ScopedKernel sk(kKernEliasLength, stream);
    const cudaError_t e = launch_chained(elias_length_kernel<LB, DENSE>, (uint32_t)ctas, kThreads, 0, stream, bp, w.len,
                                         w.lane_rec, w.cta_sums, w.group_sums);
    if (e != cudaSuccess) return (int)e;
  }
  const size_t smem = stage_bytes<DENSE>(tm.nbc, bp.d, s);
  auto kern = elias_scatter_kernel<LB, DENSE>;
  static KernelSite site;                          // (the opt-in is raised only: threads with other s share it)
  int sms = 0, occ = 0;
  const int st = site.lookup_dynamic(kern, kThreads, smem, &sms, &occ);
  if (st) return st;
  ScatterArgs a;
  a.p = bp; a.len = w.len; a.lane_rec = w.lane_rec; a.cta_sums = w.cta_sums; a.group_sums = w.group_sums;
  a.out = out; a.out_capacity = out_capacity; a.out_bits = out_bits; a.status_dev = status_dev;
  ScopedKernel sk(kKernEliasScatter, stream);
  return (int)launch_chained(kern, (uint32_t)ctas, kThreads, smem, stream, a);
}

}  // namespace

size_t elias_workspace_bytes(uint64_t n, uint32_t d, uint32_t s) {
  return carve(nullptr, n, d, s).bytes;
}

int launch_elias_encode(const float* g, uint64_t n, uint32_t d, uint32_t s, int norm_kind,
                        bool dense, uint64_t seed, uint32_t step, uint32_t worker, uint8_t* out,
                        size_t out_capacity, uint64_t* out_bits, uint8_t* workspace,
                        uint32_t* status_dev, const BucketMap& map, cudaStream_t stream) {
  const EliasWs w = carve(workspace, n, d, s);
  if (use_small(n, d, map))
    return launch_elias_encode_small(g, n, d, s, norm_kind, dense, seed, step, worker, out, out_capacity, out_bits, w, status_dev, stream);
  const uint64_t per_cta = use_tiles(n, d, s, dense) ? tile_buckets(d) : make_teams(d).nbc, B = (n + d - 1) / d;
  const uint32_t words = sum_words((uint32_t)((B + per_cta - 1) / per_cta));
  int st = launch_quantize_fixed(g, n, d, s, norm_kind, seed, step, worker, w.fixed, status_dev, nullptr,
                                 ClearWords{use_tiles(n, d, s, dense) ? w.tile_groups : w.group_sums, words}, map, stream);
  if (st) return st;
  const FixedLayout L = make_fixed_layout(n, d, s);
  BucketParams bp;
  bp.A = reinterpret_cast<const float*>(w.fixed);
  bp.sign = reinterpret_cast<const uint32_t*>(w.fixed + L.off_sign);
  bp.level = reinterpret_cast<const uint32_t*>(w.fixed + L.off_level);
  bp.n = n; bp.d = d; bp.B = L.B;
#define QSGD_RUN(LBV)                                                                            \
  (dense ? run_pipeline<LBV, true>(bp, w, s, out, out_capacity, out_bits, status_dev, stream)       \
         : run_pipeline<LBV, false>(bp, w, s, out, out_capacity, out_bits, status_dev, stream))
  switch (L.lb) {
    case 1: return QSGD_RUN(1);
    case 2: return QSGD_RUN(2);
    case 4: return QSGD_RUN(4);
    default: return QSGD_RUN(8);
  }
#undef QSGD_RUN
}

}  // namespace qsgd

// ================================================================================================
// Elias encode with library-owned scratch (see qsgd_encode_elias_static in include/qsgd.h).
//
// The scratch lives in this translation unit as one file-scope device array, so the entry point
// never asks the driver (or anybody's allocator) for memory. In host code the name of a
// __device__ array is only a handle for the runtime: its device address has to be looked up with
// cudaGetSymbolAddress, once per device, with that device current. The looked-up pointer is what
// the kernels receive.
// ================================================================================================
namespace qsgd {
namespace {

constexpr size_t kStaticScratchBytes = (size_t)QSGD_STATIC_SCRATCH_BYTES;
static __device__ __align__(256) unsigned char g_static_scratch[kStaticScratchBytes];

constexpr int kMaxDevices = 64;
static std::mutex g_scratch_mu;
static uint8_t* g_scratch_ptr[kMaxDevices] = {};

// Device address of the scratch array on the current device; looked up on first use.
int static_scratch_pointer(uint8_t** out) {
  int dev = -1;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return (int)e;
  if (dev < 0 || dev >= kMaxDevices) return (int)cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lk(g_scratch_mu);
  if (!g_scratch_ptr[dev]) {
    void* p = nullptr;
    e = cudaGetSymbolAddress(&p, g_static_scratch);
    if (e != cudaSuccess) return (int)e;
    if (!p) return (int)cudaErrorInvalidSymbol;
    g_scratch_ptr[dev] = static_cast<uint8_t*>(p);
  }
  *out = g_scratch_ptr[dev];
  return 0;
}

}  // namespace
}  // namespace qsgd

extern "C" {

size_t qsgd_static_scratch_bytes(void) { return qsgd::kStaticScratchBytes; }

int qsgd_encode_elias_static(const float* g, uint64_t n, uint32_t bucket, uint32_t s, int norm_kind,
                             int code_kind, uint64_t seed, uint32_t step, uint32_t worker, void* out,
                             size_t out_capacity, uint64_t* out_bits, uint32_t* status_dev,
                             qsgd_stream_t stream) {
  using namespace qsgd;
  if (!g || !out || !out_bits || !status_dev) return QSGD_ERR_NULL;
  if (n == 0 || n > QSGD_MAX_COORDS) return QSGD_ERR_SIZE;
  if (bucket < 32 || bucket > QSGD_MAX_BUCKET || (bucket & 31u)) return QSGD_ERR_BUCKET;
  if (s < 1 || s > QSGD_MAX_LEVELS) return QSGD_ERR_LEVELS;
  if (code_kind != QSGD_CODE_ELIAS && code_kind != QSGD_CODE_ELIAS_DENSE) return QSGD_ERR_KIND;
  if (norm_kind != QSGD_NORM_L2 && norm_kind != QSGD_NORM_MAX) return QSGD_ERR_KIND;
  if ((reinterpret_cast<uintptr_t>(g) & 15u) || (reinterpret_cast<uintptr_t>(out) & 15u)) return QSGD_ERR_ALIGN;
  const uint64_t B = (n + bucket - 1) / bucket;
  if (out_capacity < align16(4 * B) + 8 * (B + 1)) return QSGD_ERR_CAPACITY;
  if (elias_workspace_bytes(n, bucket, s) > kStaticScratchBytes) return QSGD_ERR_SCRATCH;
  uint8_t* scratch = nullptr;
  const int st = static_scratch_pointer(&scratch);
  if (st) return st;
  return launch_elias_encode(g, n, bucket, s, norm_kind, code_kind == QSGD_CODE_ELIAS_DENSE, seed, step,
                             worker, static_cast<uint8_t*>(out), out_capacity, out_bits, scratch,
                             status_dev, no_map(), static_cast<cudaStream_t>(stream));
}

}  // extern "C"
