// Encode, Elias path (Section 3.1 "Efficient Coding of Gradients", string S; Appendix A.3 for
// the dense variant). Pipeline on one stream:
//   1. quantize into the fixed-width layout held in the workspace (quantize_fixed.cu);
//   2. string length L_b of every bucket, and the sum of the lengths of each CTA's run of
//      consecutive buckets (elias_length_kernel);
//   3. the CTA of the length kernel that publishes its sum last (an arrival counter, no waiting)
//      scans the per-CTA sums, fixes the message geometry and checks the capacity;
//   4. each CTA of the scatter kernel derives the bit offsets of its own buckets, writes their
//      offset-table entries, assembles its run of strings in shared memory (lanes own
//      consecutive sub-ranges of a bucket; bits of neighbouring lanes and buckets meet inside
//      words and are merged with shared-memory atomics) and flushes whole words to the payload
//      with coalesced stores (flush_run).
// A bucket is handled by a team of d / 64 lanes (at most a warp, at least one lane), so that the
// sequential walk over a lane's nonzeros is long enough to amortise the team's scans. Small problems go
// by tiles instead (use_tiles), and the smaller ones of those are quantized and measured in one kernel
// (elias_encode_small.cu).
#include <mutex>

#include "elias_encode.cuh"

namespace qsgd {

namespace {

using namespace elias;

// ---- 2. string length per bucket, sum per CTA ------------------------------------------------------
template <int LB, bool DENSE>
__global__ void __launch_bounds__(kThreads) elias_length_kernel(const BucketParams p,
                                                                uint32_t* __restrict__ len,
                                                                uint32_t* __restrict__ lane_rec,
                                                                uint64_t* cta_sums, const ScanArgs sa) {
  __shared__ uint32_t warp_sum[kWarps];
  __shared__ uint32_t is_last;
  __shared__ uint32_t tab[17];
  fill_code_table(tab);
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
  const uint32_t bits = lane_bits<LB, DENSE>(tab, lwb, p.lpb, c_lo, c_hi, tl, live, &prev);
  if (live) lane_rec[b * p.lpb + tl] = bits | ((uint32_t)(prev + 1) << 16);   // reused by the scatter
  const uint32_t L = team_sum(bits, p.lpb);
  if (live && tl == 0) len[b] = L;
  uint32_t w = (tl == 0) ? L : 0u;                 // one contribution per bucket
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) w += __shfl_xor_sync(0xffffffffu, w, o);
  if (lane == 0) warp_sum[warp] = w;
  __syncthreads();
  if (threadIdx.x == 0) {
    uint64_t s = 0;
#pragma unroll
    for (int i = 0; i < kWarps; ++i) s += warp_sum[i];
    cta_sums[blockIdx.x] = s;
    // publish, then take a ticket: whoever draws the last one sees every CTA's sum
    __threadfence();
    is_last = atomicAdd(&sa.ctrl->arrived, 1u) == gridDim.x - 1u ? 1u : 0u;
  }
  __syncthreads();
  if (is_last) {
    __threadfence();
    scan_cta_sums(cta_sums, sa.ctas, p.B, sa.out_capacity, sa.ctrl, sa.out_bits, sa.status_dev);
  }
}

// ---- 4. scatter ----------------------------------------------------------------------------------
template <int LB, bool DENSE>
__global__ void __launch_bounds__(kThreads) elias_scatter_kernel(const BucketParams p,
                                                                 const uint32_t* __restrict__ len,
                                                                 const uint32_t* __restrict__ lane_rec,
                                                                 const uint64_t* __restrict__ cta_start,
                                                                 const Ctrl* __restrict__ ctrl,
                                                                 uint8_t* __restrict__ out) {
  extern __shared__ uint32_t stage[];
  __shared__ uint32_t warp_sum[kWarps];
  __shared__ uint32_t tab[17];
  __shared__ CodeWords<LB> words;
  fill_code_table(tab);
  if (!DENSE) fill_code_words<LB>(words);
  chain_wait();                                    // ctrl, lengths and sums come from the kernel ahead
  if (!ctrl->ok) return;
  const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t tl = lane & (p.lpb - 1), team = lane / p.lpb, bpw = 32 / p.lpb;
  const uint64_t b = (uint64_t)blockIdx.x * p.nbc + warp * bpw + team;
  const bool live = b < p.B;
  const uint64_t base = live ? b * p.d : 0;
  const uint32_t db = live ? (uint32_t)min((uint64_t)p.d, p.n - base) : 0;
  const uint32_t c_lo = min(tl * p.seg, db), c_hi = min(c_lo + p.seg, db);

  const uint64_t start = __ldg(cta_start + blockIdx.x), stop = __ldg(cta_start + blockIdx.x + 1);
  const uint32_t lead = (uint32_t)(start & 31);                     // bits of the first word owned by the previous CTA
  const uint32_t span = (uint32_t)(stop - start);                   // bits of this CTA's run
  const uint32_t nwords = (lead + span + 31) >> 5;
  for (uint32_t j = threadIdx.x; j < nwords; j += kThreads) stage[j] = 0u;

  // bit offset of every bucket inside the CTA's run: scan of the bucket lengths
  const uint32_t L = (live && tl == 0) ? __ldg(len + b) : 0u;
  uint32_t inc = L;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t t = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= (uint32_t)o) inc += t;
  }
  if (lane == 31) warp_sum[warp] = inc;
  __syncthreads();                                                  // staging zeroed, warp sums visible
  uint32_t before = 0;
#pragma unroll
  for (int w = 0; w < kWarps; ++w) if ((uint32_t)w < warp) before += warp_sum[w];
  uint32_t bucket_off = before + inc - L;                           // valid in team lane 0
  bucket_off = __shfl_sync(0xffffffffu, bucket_off, (int)(lane - tl));
  const uint32_t Lb = __shfl_sync(0xffffffffu, L, (int)(lane - tl));
  if (live && tl == 0) {
    uint64_t* table = reinterpret_cast<uint64_t*>(out + ctrl->payload_bytes);
    table[b] = start + bucket_off;
    if (b == p.B - 1) table[p.B] = start + bucket_off + Lb;
  }

  // this lane's first bit inside its bucket: scan of the lane lengths over the team
  int32_t prev;
  const uint32_t* lwb = p.level + ((base * LB) >> 5);            // the bucket's first level word
  const uint32_t* swb = p.sign + (base >> 5);                    // ... and first sign word
  // this lane's share of the string and the nonzero before it were counted by the length kernel
  const uint32_t rec = live ? __ldg(lane_rec + b * p.lpb + tl) : 0u;
  const uint32_t bits = rec & 0xFFFFu;
  prev = (int32_t)(rec >> 16) - 1;
  uint32_t linc = bits;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t t = __shfl_up_sync(0xffffffffu, linc, o);
    if ((uint32_t)o < p.lpb && tl >= (uint32_t)o) linc += t;
  }
  if (bits != 0) {
    StageWriter bw;
    bw.begin(stage, lead + bucket_off + (linc - bits));
    if (tl == 0) bw.put(__float_as_uint(__ldg(p.A + b)), 32);
    if (DENSE) {
      // ranges of whole 64-coordinate blocks: sign and level words are loaded once per block and word
      constexpr uint32_t kFields = 32u / LB, kMask = (1u << LB) - 1u;
      for (uint32_t c0 = c_lo; c0 < c_hi; c0 += 64u) {
        const uint32_t* wp = lwb + ((c0 * LB) >> 5);
        const uint32_t s0 = __ldg(swb + (c0 >> 5)), s1 = (c0 + 32u < c_hi) ? __ldg(swb + (c0 >> 5) + 1) : 0u;
        const unsigned long long signs = (unsigned long long)s0 | ((unsigned long long)s1 << 32);
#pragma unroll
        for (uint32_t j = 0; j < 2u * LB; ++j) {
          const uint32_t off = j * kFields;                   // first coordinate of this word in the block
          if (c0 + off >= c_hi) break;
          const uint32_t w = __ldg(wp + j);
          const uint32_t cnt = min(kFields, c_hi - (c0 + off));
          for (uint32_t f = 0; f < cnt; ++f) {
            uint32_t ln;
            const uint32_t code = tab_code(tab, ((w >> (f * LB)) & kMask) + 1u, &ln);
            bw.put((((uint32_t)(signs >> (off + f)) & 1u) << ln) | code, ln + 1);
          }
        }
      }
    } else {
      // ranges of whole 64-coordinate blocks: the block's nonzero mask
      // and sign bits sit in registers, code words come whole from the two tables.
      constexpr uint32_t kFields = 32u / LB, kMask = (1u << LB) - 1u;
      for (uint32_t c0 = c_lo; c0 < c_hi; c0 += 64u) {
        const uint32_t* wp = lwb + ((c0 * LB) >> 5);
        unsigned long long m = 0ull;
#pragma unroll
        for (uint32_t j = 0; j < 2u * LB; ++j) {
          const uint32_t w = (c0 + j * kFields < c_hi) ? __ldg(wp + j) : 0u;
          m |= (unsigned long long)nonzero_mask<LB>(w) << (j * kFields);
        }
        const uint32_t s0 = __ldg(swb + (c0 >> 5)), s1 = (c0 + 32u < c_hi) ? __ldg(swb + (c0 >> 5) + 1) : 0u;
        const unsigned long long signs = (unsigned long long)s0 | ((unsigned long long)s1 << 32);
        while (m) {
          const uint32_t off = (uint32_t)__ffsll((long long)m) - 1u;
          m &= m - 1ull;
          const uint32_t pos = c0 + off, bit = off * LB;
          const uint32_t level = (__ldg(wp + (bit >> 5)) >> (bit & 31u)) & kMask;
          const uint32_t gap = pos - (uint32_t)prev;
          uint32_t gcode, gl;
          if (gap < 64u) {
            const uint32_t e = words.gap[gap];
            gcode = e & 0xFFFFu;
            gl = e >> 16;
          } else {
            gcode = tab_code(tab, gap, &gl);
          }
          const uint32_t e = words.level[level];
          const uint32_t ll = e >> 16;
          const uint32_t lcode = (e & 0xFFFFu) | ((uint32_t)((signs >> off) & 1ull) << ll);
          if (gl + ll + 1u <= 32u) {                     // gap, sign and level in one piece (the rule)
            bw.put((gcode << (ll + 1u)) | lcode, gl + ll + 1u);
          } else {
            bw.put(gcode, gl);
            bw.put(lcode, ll + 1u);
          }
          prev = (int32_t)pos;
        }
      }
    }
    bw.finish();
  }
  __syncthreads();
  const uint64_t next = (uint64_t)(blockIdx.x + 1u) * p.nbc;       // the next CTA's first bucket
  flush_run(reinterpret_cast<uint32_t*>(out) + (start >> 5), stage, lead, span, next >= p.B, p.A + next,
            (uint32_t)(ctrl->payload_bytes / 4 - (start >> 5)));
}

// ---- 2. for tiles ----------------------------------------------------------------------------------
template <int LB, bool DENSE>
__global__ void __launch_bounds__(kThreads) elias_tile_length_kernel(const BucketParams p, uint64_t* cta_sums, const ScanArgs sa) {
  __shared__ uint32_t slots[2][kWarps];
  __shared__ uint32_t is_last;
  __shared__ uint32_t tab[17];
  fill_code_table(tab);
  __syncthreads();
  chain_wait();                                    // the fields come from the kernel ahead
  const Piece<LB> q = load_piece<LB>(p);
  const uint32_t mask = DENSE ? 0u : piece_mask<LB>(q);
  const int32_t prev = DENSE ? -1 : nonzero_before<LB>(q, mask, slots[0]);
  uint32_t total;
  cta_sum_before(piece_bits<LB, DENSE>(tab, q, mask, prev), slots[1], &total);
  if (threadIdx.x == 0) {
    cta_sums[blockIdx.x] = total;
    __threadfence();
    is_last = atomicAdd(&sa.ctrl->arrived, 1u) == gridDim.x - 1u ? 1u : 0u;
  }
  __syncthreads();
  if (is_last) {
    __threadfence();
    scan_cta_sums(cta_sums, sa.ctas, p.B, sa.out_capacity, sa.ctrl, sa.out_bits, sa.status_dev);
  }
}

template <int LB, bool DENSE>
int run_pipeline(BucketParams& bp, const EliasWs& w, uint32_t s, uint8_t* out, size_t out_capacity,
                 uint64_t* out_bits, uint32_t* status_dev, cudaStream_t stream) {
  if (use_tiles(bp.n, bp.d, s, DENSE)) {
    bp.lpb = 0; bp.seg = 16; bp.nbc = tile_buckets(bp.d);
    const uint64_t ctas = (bp.B + bp.nbc - 1) / bp.nbc;
    ScanArgs sa;
    sa.ctas = ctas; sa.out_capacity = out_capacity; sa.ctrl = w.ctrl; sa.out_bits = out_bits;
    sa.status_dev = status_dev;
    {
      ScopedKernel sk(kKernEliasLength, stream);
      const cudaError_t e = launch_chained(elias_tile_length_kernel<LB, DENSE>, (uint32_t)ctas, kThreads, 0, stream, bp,
                                           w.tile_sums, sa);
      if (e != cudaSuccess) return (int)e;
    }
    return launch_tile_scatter(bp, w, s, DENSE, out, stream);
  }
  const Teams tm = make_teams(bp.d);
  bp.lpb = tm.lpb; bp.seg = tm.seg; bp.nbc = tm.nbc;
  const uint64_t ctas = (bp.B + tm.nbc - 1) / tm.nbc;
  {
    ScanArgs sa;
    sa.ctas = ctas; sa.out_capacity = out_capacity; sa.ctrl = w.ctrl; sa.out_bits = out_bits;
    sa.status_dev = status_dev;
    ScopedKernel sk(kKernEliasLength, stream);
    const cudaError_t e = launch_chained(elias_length_kernel<LB, DENSE>, (uint32_t)ctas, kThreads, 0, stream, bp, w.len,
                                         w.lane_rec, w.cta_sums, sa);
    if (e != cudaSuccess) return (int)e;
  }
  {
    const size_t smem = stage_bytes<DENSE>(tm.nbc, bp.d, s);
    auto kern = elias_scatter_kernel<LB, DENSE>;
    if (smem > 48 * 1024) {                        // the opt-in is raised only: threads with other s share it
      static KernelSite site;
      int sms = 0, occ = 0;
      const int st = site.lookup_dynamic(kern, kThreads, smem, &sms, &occ);
      if (st) return st;
    }
    ScopedKernel sk(kKernEliasScatter, stream);
    return (int)launch_chained(kern, (uint32_t)ctas, kThreads, smem, stream, bp, w.len, w.lane_rec, w.cta_sums, w.ctrl, out);
  }
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
  int st = launch_quantize_fixed(g, n, d, s, norm_kind, seed, step, worker, w.fixed, status_dev, nullptr,
                                 &w.ctrl->arrived, map, stream);
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
