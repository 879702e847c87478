// Encode, Elias path, for small problems: quantizing and measuring the strings in one kernel, scanning and
// writing them in a second one; a single tile in one kernel altogether. Between two launches of a chain lie 3 to 4
// us, and three of them (quantize, length, scatter) were the time of an encode up to a million coordinates
// (n = 4096: 11.9 -> 4.5 us with one launch, n = 2^20: 11.9 -> 8.8 us with two, d = 512, s = 15).
//
// A CTA takes a tile of whole buckets (at most 4096 coordinates), a thread 16 consecutive coordinates. Complete
// tiles of power-of-two buckets are quantized in registers with the very operations and order of the
// streaming encoder (quantize_fixed.cu), so that the scales come out bit for bit the same; others by the tile
// code that both share. The scatter kernel's CTAs each add up all tiles' lengths for themselves: up to 1000
// loads a CTA instead of an arrival counter and a scan by the last one to arrive.
#include "elias_encode.cuh"
#include "quantize.cuh"

namespace qsgd {

namespace {

using namespace elias;

struct SmallParams {
  QuantizeParams q;           // what quantizing needs; its regions are those of bp
  BucketParams bp;
  uint32_t log2d;             // of a power-of-two bucket size, else 32
  uint32_t* cta_sums;         // bits of every tile
  // one tile:
  uint8_t* out;
  size_t out_capacity;
  uint64_t* out_bits;
  uint32_t* status_dev;
};

// Writes one tile's run of strings: table entries, codes into `stage` (zeroed), the flush.
template <int LB, bool DENSE>
__device__ __forceinline__ void write_tile(const uint32_t* tab, const CodeWords<LB, DENSE>& words, uint32_t* stage, const BucketParams& p,
                                           const Piece<LB>& q, uint32_t mask, int32_t prev, uint32_t bits, uint32_t before,
                                           float A, uint64_t start, uint32_t span, uint64_t payload_bytes, uint8_t* out) {
  const uint32_t lead = (uint32_t)(start & 31);    // bits of the first word that belong to the tile before
  if (q.count && q.c0 == 0u) {                     // this piece opens its bucket's string
    const uint64_t b = (uint64_t)blockIdx.x * p.nbc + q.bucket;
    uint64_t* table = reinterpret_cast<uint64_t*>(out + payload_bytes);
    table[b] = start + before;
    if (b == p.B - 1) table[p.B] = start + span;   // the last bucket ends its tile's run
  }
  if (bits) emit_piece<LB, DENSE>(tab, words, stage, lead + before, q, mask, prev, A);
  __syncthreads();
  const uint64_t next = (uint64_t)(blockIdx.x + 1u) * p.nbc;
  flush_run(reinterpret_cast<uint32_t*>(out) + (start >> 5), stage, lead, span, next >= p.B, p.A + next,
            (uint32_t)(payload_bytes / 4 - (start >> 5)));
}

// A complete tile of power-of-two buckets: scale, levels and signs of this thread's 16 coordinates.
template <int LB, int NORM>
__device__ __forceinline__ float quantize_tile(const SmallParams& p, float* wsum, double* wsum64, uint32_t (&lw)[4], uint32_t& sw) {
  constexpr uint32_t kAll = 0xffffffffu;
  const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, t = blockIdx.x;
  const float4* src = reinterpret_cast<const float4*>(p.q.g + (size_t)t * kTile) + tid * 4;
  float v[16];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const float4 a = __ldcs(src + j);
    v[4 * j] = a.x; v[4 * j + 1] = a.y; v[4 * j + 2] = a.z; v[4 * j + 3] = a.w;
  }
  float part = 0.f;
#pragma unroll
  for (int e = 0; e < 16; ++e) {
    if (NORM == QSGD_NORM_L2) part = fmaf(v[e], v[e], part);
    else part = fmaxf(part, fabsf(v[e]));
  }
  const uint32_t team_w = p.log2d >= 9u ? 32u : 1u << (p.log2d - 4u);      // lanes that share a bucket inside a warp
#pragma unroll
  for (uint32_t o = 16; o > 0; o >>= 1) {
    const float q = __shfl_xor_sync(kAll, part, o);
    const float merged = (NORM == QSGD_NORM_L2) ? part + q : fmaxf(part, q);
    part = (o < team_w) ? merged : part;
  }
  // an fp32 sum of squares outside [8e-28, 1e30] may have lost bits: again in fp64
  const bool shaky = NORM == QSGD_NORM_L2 && !(part >= 8.0e-28f && part <= 1.0e30f);
  double wide = 0.0;
  auto wide_sum = [&]() {
#pragma unroll
    for (int e = 0; e < 16; ++e) wide = fma((double)v[e], (double)v[e], wide);
#pragma unroll
    for (uint32_t o = 16; o > 0; o >>= 1) {
      const double q = __shfl_xor_sync(kAll, wide, o);
      wide = (o < team_w) ? wide + q : wide;
    }
  };
  float A;
  if (p.log2d <= 9u) {
    A = NORM == QSGD_NORM_L2 ? __fsqrt_rn(part) : part;
    if (__any_sync(kAll, shaky)) {
      wide_sum();
      if (shaky) A = __double2float_rn(sqrt(wide));
    }
  } else {                                          // 2, 4 or 8 warps share a bucket
    const uint32_t wpb = 1u << (p.log2d - 9u), w0 = warp & ~(wpb - 1u);
    if (lane == 0) wsum[warp] = part;
    const bool again = __syncthreads_or(shaky ? 1 : 0) != 0;
    float acc = 0.f;
    bool mine = false;
    for (uint32_t w = 0; w < wpb; ++w) {
      const float q = wsum[w0 + w];
      acc = (NORM == QSGD_NORM_L2) ? acc + q : fmaxf(acc, q);
      mine |= NORM == QSGD_NORM_L2 && !(q >= 8.0e-28f && q <= 1.0e30f);
    }
    A = NORM == QSGD_NORM_L2 ? __fsqrt_rn(acc) : acc;
    if (again) {
      wide_sum();
      if (lane == 0) wsum64[warp] = wide;
      __syncthreads();
      wide = 0.0;
      for (uint32_t w = 0; w < wpb; ++w) wide += wsum64[w0 + w];
      if (mine) A = __double2float_rn(sqrt(wide));
    }
  }
  if (!(A >= FLT_MIN)) A = 0.f;                     // zero bucket: Q(0) = 0
  const float r = A > 0.f ? __frcp_rn(A) : 0.f;
  const float sf = (float)p.q.s;
  float um[16];
  philox_uniforms16(t * (kTile / 4) + tid * 4, p.q.pc, um);
  quantize16<LB, true>(v, um, r, sf, kTwo23 + sf, lw, sw);
  if (LB != 8) sw &= nonzero_fields16<LB>(lw);      // canonical sign: 0 where the level is 0
  return A;
}

template <int LB, int NORM, bool DENSE, bool ONE>
__global__ void __launch_bounds__(kThreads) elias_quantize_length_kernel(const __grid_constant__ SmallParams p) {
  extern __shared__ uint32_t stage[];               // ONE: the strings
  __shared__ __align__(16) float tile[kTile];
  __shared__ float part[kTile / 8];
  __shared__ float s_rcp[kMaxBucketsPerTile];
  __shared__ uint32_t slots[2][kWarps];
  __shared__ uint32_t tab[17];
  __shared__ CodeWords<ONE ? LB : 1, DENSE> words;
  __shared__ SymbolLengths<DENSE ? LB : 1> lengths;
  fill_code_table(tab);
  if (DENSE) fill_symbol_lengths<DENSE ? LB : 1>(lengths);
  if (ONE) fill_code_words(words);
  chain_wait();
  const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  Piece<LB> q;
  float A = 0.f;
  if (p.log2d < 32u && (uint64_t)(blockIdx.x + 1u) * kTile <= p.q.n) {
    uint32_t lw[4], sw;
    A = quantize_tile<LB, NORM>(p, part, reinterpret_cast<double*>(tile), lw, sw);
    q.bucket = (tid * 16u) >> p.log2d;
    q.c0 = (tid * 16u) & ((1u << p.log2d) - 1u);
    q.count = 16u;
    q.sign = sw & 0xFFFFu;
#pragma unroll
    for (int j = 0; j < Piece<LB>::kWords; ++j) q.level[j] = lw[j];
    if (!ONE) {
      if (q.c0 == 0u) p.q.A_out[((uint64_t)blockIdx.x << (12u - p.log2d)) + q.bucket] = A;
      store_chunk<LB>(p.q.sign_out, p.q.level_out, blockIdx.x * (kTile / 512) + warp, lane, sw, lw);
    }
  } else {
    quantize_generic_tile<LB, NORM, false>(p.q, blockIdx.x, gridDim.x, tile, part, s_rcp);
    __syncthreads();
    q = load_piece<LB>(p.bp);
    if (ONE && q.count && q.c0 == 0u) A = p.bp.A[q.bucket];
  }
  __syncthreads();                                  // the code tables are there
  const uint32_t mask = DENSE ? 0u : piece_mask<LB>(q);
  const int32_t prev = DENSE ? -1 : nonzero_before<LB>(q, mask, slots[0]);
  const uint32_t bits = piece_bits<LB, DENSE>(tab, lengths, q, mask, prev);
  uint32_t total;
  const uint32_t before = cta_sum_before(bits, slots[1], &total);
  if constexpr (!ONE) {
    if (tid == 0) p.cta_sums[blockIdx.x] = total;
  } else {
    uint64_t pay;
    if (!fix_geometry(total, p.bp.B, p.out_capacity, p.out_bits, p.status_dev, true, &pay)) return;
    for (uint32_t j = tid; j < (total + 31u) >> 5; j += kThreads) stage[j] = 0u;
    __syncthreads();
    write_tile<LB, DENSE>(tab, words, stage, p.bp, q, mask, prev, bits, before, A, 0, total, pay, p.out);
  }
}

// Where a tile's run of strings begins and how long the payload is: by sums over groups of tiles, or, in small problems, where
// nothing has cleared those, every CTA adds up the lengths of all tiles.
struct TileScatterArgs {
  BucketParams bp;
  const uint32_t* sums;       // bits of every tile
  const uint64_t* groups;     // of every group of tiles, or null
  uint32_t ctas;
  uint8_t* out;
  size_t out_capacity;
  uint64_t* out_bits;
  uint32_t* status_dev;
};

template <int LB, bool DENSE>
__global__ void __launch_bounds__(kThreads) elias_tile_scatter_kernel(const __grid_constant__ TileScatterArgs a) {
  extern __shared__ uint32_t stage[];
  __shared__ uint32_t slots[2][kWarps];
  __shared__ uint64_t before_s[kWarps], total_s[kWarps];
  __shared__ uint32_t tab[17];
  __shared__ CodeWords<LB, DENSE> words;
  __shared__ SymbolLengths<DENSE ? LB : 1> lengths;
  fill_code_table(tab);
  fill_code_words(words);
  if (DENSE) fill_symbol_lengths<DENSE ? LB : 1>(lengths);
  chain_wait();                                    // fields and sums come from the kernel ahead
  const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const Piece<LB> q = load_piece<LB>(a.bp);
  const float A = q.count && q.c0 == 0u ? a.bp.A[(uint64_t)blockIdx.x * a.bp.nbc + q.bucket] : 0.f;
  uint64_t start, tot;
  const uint32_t span = a.sums[blockIdx.x];
  if (a.groups) {
    if (warp == 0) find_start(a.sums, a.groups, &before_s[0], &total_s[0]);
    __syncthreads();
    start = before_s[0];
    tot = total_s[0];
  } else {
    uint64_t bef = 0;
    tot = 0;
    for (uint32_t i = tid; i < a.ctas; i += kThreads) {
      const uint32_t v = a.sums[i];
      tot += v;
      bef += i < blockIdx.x ? v : 0u;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      bef += __shfl_xor_sync(0xffffffffu, bef, o);
      tot += __shfl_xor_sync(0xffffffffu, tot, o);
    }
    if (lane == 0) { before_s[warp] = bef; total_s[warp] = tot; }
    __syncthreads();
    bef = tot = 0;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) { bef += before_s[w]; tot += total_s[w]; }
    start = bef;
  }
  uint64_t pay;
  if (!fix_geometry(tot, a.bp.B, a.out_capacity, a.out_bits, a.status_dev, blockIdx.x == 0, &pay)) return;
  const uint32_t nwords = ((uint32_t)(start & 31) + span + 31u) >> 5;
  for (uint32_t j = tid; j < nwords; j += kThreads) stage[j] = 0u;
  __syncthreads();                                 // staging zeroed, tables there
  const uint32_t mask = DENSE ? 0u : piece_mask<LB>(q);
  const int32_t prev = DENSE ? -1 : nonzero_before<LB>(q, mask, slots[0]);
  const uint32_t bits = piece_bits<LB, DENSE>(tab, lengths, q, mask, prev);
  uint32_t total;
  const uint32_t before = cta_sum_before(bits, slots[1], &total);
  write_tile<LB, DENSE>(tab, words, stage, a.bp, q, mask, prev, bits, before, A, start, span, pay, a.out);
}

template <int LB, bool DENSE>
int scatter(const TileScatterArgs& a, uint32_t s, cudaStream_t stream) {
  ScopedKernel sk(kKernEliasScatter, stream);
  return (int)launch_chained(elias_tile_scatter_kernel<LB, DENSE>, a.ctas, kThreads, stage_bytes<DENSE>(a.bp.nbc, a.bp.d, s), stream, a);
}

int scatter_any(const TileScatterArgs& a, uint32_t s, bool dense, cudaStream_t stream) {
  switch (level_bits_for(s)) {
    case 1: return dense ? scatter<1, true>(a, s, stream) : scatter<1, false>(a, s, stream);
    case 2: return dense ? scatter<2, true>(a, s, stream) : scatter<2, false>(a, s, stream);
    case 4: return dense ? scatter<4, true>(a, s, stream) : scatter<4, false>(a, s, stream);
    default: return dense ? scatter<8, true>(a, s, stream) : scatter<8, false>(a, s, stream);
  }
}

template <int LB, int NORM, bool DENSE>
int quantize(const SmallParams& p, uint32_t ctas, cudaStream_t stream) {
  ScopedKernel sk(kKernQuantize, stream);
  if (ctas == 1u) {
    const size_t smem = stage_bytes<DENSE>(p.bp.nbc, p.bp.d, p.q.s);
    return (int)launch_chained(elias_quantize_length_kernel<LB, NORM, DENSE, true>, 1u, kThreads, smem, stream, p);
  }
  return (int)launch_chained(elias_quantize_length_kernel<LB, NORM, DENSE, false>, ctas, kThreads, 0, stream, p);
}

template <int LB>
int quantize_lb(const SmallParams& p, int norm_kind, bool dense, uint32_t ctas, cudaStream_t stream) {
  if (norm_kind == QSGD_NORM_L2)
    return dense ? quantize<LB, QSGD_NORM_L2, true>(p, ctas, stream) : quantize<LB, QSGD_NORM_L2, false>(p, ctas, stream);
  return dense ? quantize<LB, QSGD_NORM_MAX, true>(p, ctas, stream) : quantize<LB, QSGD_NORM_MAX, false>(p, ctas, stream);
}

}  // namespace

namespace elias {

int launch_tile_scatter(const BucketParams& bp, const EliasWs& w, uint32_t s, bool dense, uint8_t* out, size_t out_capacity,
                        uint64_t* out_bits, uint32_t* status_dev, cudaStream_t stream) {
  TileScatterArgs a;
  a.bp = bp; a.sums = w.tile_sums; a.groups = w.tile_groups; a.ctas = (uint32_t)((bp.B + bp.nbc - 1) / bp.nbc); a.out = out;
  a.out_capacity = out_capacity; a.out_bits = out_bits; a.status_dev = status_dev;
  return scatter_any(a, s, dense, stream);
}

int launch_elias_encode_small(const float* g, uint64_t n, uint32_t d, uint32_t s, int norm_kind, bool dense, uint64_t seed,
                              uint32_t step, uint32_t worker, uint8_t* out, size_t out_capacity, uint64_t* out_bits,
                              const EliasWs& w, uint32_t* status_dev, cudaStream_t stream) {
  const FixedLayout L = make_fixed_layout(n, d, s);
  SmallParams p;
  p.q.g = g; p.q.n = n; p.q.d = d; p.q.s = s; p.q.map = no_map();
  p.q.tile_coords = (kTile / d) * d;
  p.q.coord_base = 0;
  p.q.pc = make_philox_consts(seed, step, worker);
  p.q.A_out = reinterpret_cast<float*>(w.fixed);
  p.q.sign_out = reinterpret_cast<uint32_t*>(w.fixed + L.off_sign);
  p.q.level_out = reinterpret_cast<uint32_t*>(w.fixed + L.off_level);
  p.q.B = L.B; p.q.sign_words = L.sign_words; p.q.level_words = L.level_words;
  p.q.tiles = 0; p.q.status = status_dev; p.q.info = nullptr; p.q.total_bytes = L.total; p.q.clear = ClearWords{nullptr, 0};
  p.bp.A = p.q.A_out; p.bp.sign = p.q.sign_out; p.bp.level = p.q.level_out;
  p.bp.n = n; p.bp.d = d; p.bp.B = L.B; p.bp.lpb = 0; p.bp.seg = 16; p.bp.nbc = tile_buckets(d);
  p.log2d = 32;
  if ((d & (d - 1u)) == 0)
    for (p.log2d = 0; (1u << p.log2d) < d; ++p.log2d) {}
  p.cta_sums = w.tile_sums;
  p.out = out; p.out_capacity = out_capacity; p.out_bits = out_bits; p.status_dev = status_dev;
  const uint32_t ctas = (uint32_t)((L.B + p.bp.nbc - 1) / p.bp.nbc);
  int st;
  switch (L.lb) {
    case 1: st = quantize_lb<1>(p, norm_kind, dense, ctas, stream); break;
    case 2: st = quantize_lb<2>(p, norm_kind, dense, ctas, stream); break;
    case 4: st = quantize_lb<4>(p, norm_kind, dense, ctas, stream); break;
    default: st = quantize_lb<8>(p, norm_kind, dense, ctas, stream); break;
  }
  if (st || ctas == 1u) return st;
  TileScatterArgs a;
  a.bp = p.bp; a.sums = w.tile_sums; a.groups = nullptr; a.ctas = ctas; a.out = out;
  a.out_capacity = out_capacity; a.out_bits = out_bits; a.status_dev = status_dev;
  return scatter_any(a, s, dense, stream);
}

}  // namespace elias
}  // namespace qsgd
