// Decode-and-aggregate, Elias path, optionally fused with the SGD step (Section 3.1, end of
// "Efficient Coding of Gradients": the receiver takes the 32-bit scale off the front of a string and
// then walks the (gap, sign, level) codes; Appendix A.2 for the integer decoder; Algorithm 1 for the
// sum and the step).
//
// A string S can only be parsed front to back, but buckets and peers are independent once the
// per-bucket offset table gives each string's first bit. A warp owns a group of G buckets.
// Phase 1 (parse): lane (g, k) reads peer k's string of bucket g through a register
// window (a word ahead) and rebuilds that peer's *fixed-width fields* -- level fields
// and sign bitmap -- for the bucket in shared memory. Phase 2 (apply): every lane takes 16 coordinates and adds
// the peers' fields in ascending k, which fixes the summation order however phase 1 was scheduled. Which shapes come here and which are read by teams of lanes: use_teams in elias_decode.cu.
#include "elias_decode.cuh"

namespace qsgd {

namespace {

// Reconstruction by arithmetic: A * (level / s), the quotient rounded to nearest as the definition has it, without a
// table. The table took 32 KB of a CTA, so fewer warps fitted, and the parse waits on latency: 42.5 us with it, 39.7 us
// without (n = 1 M, d = 96, s = 255, K = 5). The fixed-width decoder does nothing else than this, and was faster with
// the table that it had then (335 against 376 us at n = 60 M, K = 16; with signs in the table 263). With 1 / s = hi + lo in two floats, RN(level * hi + RN(level * lo)) is
// RN(level / s) for every s <= 255 and level <= s (checked exhaustively in rational arithmetic). The level comes as the
// float 2^23 + level, made by one byte permute. All steps work on pairs (f32x2).
struct LevelQuotient {
  unsigned long long hi, lo, klo, m23, m0;      // 1 / s; its rest; -2^23 * rest; -2^23; -0
};

// `minus_zero` is -0 that the compiler cannot see (a kernel parameter): the product with A is an fma with it, because
// ptxas contracts a mul.rn.f32x2 in front of an add.rn.f32x2.
__device__ __forceinline__ LevelQuotient level_quotient(uint32_t s, float minus_zero) {
  const float hi = __fdiv_rn(1.f, (float)s);
  const float lo = __double2float_rn(1.0 / (double)s - (double)hi);
  LevelQuotient q;
  q.hi = pair2(hi, hi); q.lo = pair2(lo, lo);
  q.klo = pair2(-8388608.f * lo, -8388608.f * lo); q.m23 = pair2(-8388608.f, -8388608.f);
  q.m0 = pair2(minus_zero, minus_zero);
  return q;
}

// acc += +-A * (level / s) for two coordinates: levels in bytes j0 of w0 and j1 of w1, signs in bits e and e + 1 of sb.
__device__ __forceinline__ void add_level_pair(float& acc0, float& acc1, uint32_t w0, uint32_t j0, uint32_t w1, uint32_t j1, uint32_t sb,
                                               uint32_t e, float A, const LevelQuotient& lq) {
  const float f0 = __uint_as_float(__byte_perm(w0, 0x4B000000u, 0x7440u | j0));
  const float f1 = __uint_as_float(__byte_perm(w1, 0x4B000000u, 0x7440u | j1));
  const unsigned long long f = pair2(f0, f1);
  const unsigned long long q = fma2(add2(f, lq.m23), lq.hi, fma2(f, lq.lo, lq.klo));
  const float a0 = __uint_as_float(__float_as_uint(A) ^ ((sb << (31u - e)) & 0x80000000u));
  const float a1 = __uint_as_float(__float_as_uint(A) ^ ((sb << (30u - e)) & 0x80000000u));
  const unsigned long long r = add2(pair2(acc0, acc1), fma2(pair2(a0, a1), q, lq.m0));
  asm("mov.b64 {%0, %1}, %2;" : "=f"(acc0), "=f"(acc1) : "l"(r));
}

// 16 one-byte levels in w.
__device__ __forceinline__ void add_peer_bytes(float (&acc)[16], const uint32_t (&w)[4], uint32_t sb, float A, const LevelQuotient& lq) {
#pragma unroll
  for (uint32_t h = 0; h < 4; ++h) {
    add_level_pair(acc[4 * h], acc[4 * h + 1], w[h], 0, w[h], 1, sb, 4 * h, A, lq);
    add_level_pair(acc[4 * h + 2], acc[4 * h + 3], w[h], 2, w[h], 3, sb, 4 * h + 2, A, lq);
  }
}

// One lane, one string. Every code goes the same way (code_entry), so that lanes with different codes stay together, and
// nothing is read back: a level is a byte, and the signs of 32 coordinates are gathered in a register. The loop is a chain
// of dependent instructions and bound by their latency. Against tables of whole codes with a way around them for the
// others, and fields OR-ed in shared memory: 39.9 -> 36.2 us at n = 1 M, d = 96, s = 255, K = 5 (2-norm), 914 -> 664 at
// n = 16.8 M, d = 256, K = 8 (max-norm), 1124 -> 799 at d = 128, K = 16.
// ONES: most gaps are 1, the single bit 0, and their lookup is left out.
template <bool ONES>
__device__ __forceinline__ uint32_t read_codes(Window& in, uint32_t end, uint32_t db, uint32_t d, uint32_t s, const uint2* code,
                                               uint32_t* __restrict__ row) {
  uint8_t* levels = reinterpret_cast<uint8_t*>(row);
  uint32_t* signs = row + (d >> 2);
  uint32_t bad = 0, at = 0xFFFFFFFFu;               // position of the previous nonzero (-1)
  uint32_t gathered = 0, block = 0;                 // signs of the coordinates 32 * block ..
  while (in.bp < end) {
    const uint32_t w = in.peek();
    uint32_t body = 0u, gap = 1u, y = w;
    if (!ONES || w >> 31) {
      const uint2 c = code[w >> 25];
      body = code_body(c);
      gap = code_value(w, c);
      y = in.peek_at(body);
    }
    const uint32_t z = y << 2;
    const uint2 e = code[z >> 25];
    const uint32_t level = code_value(z, e), lb = code_body(e);
    at += gap;
    bad |= y | (z << lb);                           // the two closing bits
    if (at >= db || level > s) return at >= db ? QSGD_DEV_POSITION : QSGD_DEV_LEVEL;
    levels[at] = (uint8_t)level;
    if (at >> 5 != block) { signs[block] = gathered; gathered = 0u; block = at >> 5; }
    gathered |= ((y >> 30) & 1u) << (at & 31u);
    uint32_t bits = body + lb + 3u;
    if (bits > 32u) { in.drop_even(body, end); bits -= body; }
    in.drop_even(bits, end);
  }
  signs[block] = gathered;
  return bad >> 31 || in.bp != end ? QSGD_DEV_OVERRUN : 0u;
}

__device__ __forceinline__ uint32_t parse_to_fields(const StringRef& ref, bool ones, uint32_t db, uint32_t d, uint32_t s, const uint2* code,
                                                    uint32_t* __restrict__ row, float* A_out) {
  *A_out = 0.f;
  if (ref.err) return ref.err;
  Window in;
  in.open(ref.words, ref.lo);
  const uint32_t end = in.bp + 32u + ref.total;
  *A_out = __uint_as_float(in.peek());
  in.drop_even(32u, end);
  return ones ? read_codes<true>(in, end, db, d, s, code, row) : read_codes<false>(in, end, db, d, s, code, row);
}

template <bool FUSED>
__global__ void __launch_bounds__(320) decode_elias_fields_kernel(const __grid_constant__ FieldParams p) {
  constexpr int LB = 8;
  extern __shared__ __align__(16) uint32_t fsm[];
  __shared__ uint2 code[kCodeEntries];
  chain_wait();                                   // the messages come from the kernels ahead
  if (p.when.lo && mean_below(p.when.lo, p.peers, p.K, p.B)) return;
  const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = blockDim.x >> 5;
  for (uint32_t i = tid; i < kCodeEntries; i += blockDim.x) code[i] = code_entry(i);
  __syncthreads();
  const LevelQuotient lq = level_quotient(p.s, p.minus_zero);

  const uint32_t warp_words = p.G * p.bucket_words;
  uint32_t* words = fsm + (size_t)warp * warp_words;
  const uint32_t level_words = (p.d * LB) >> 5;
  const uint32_t pg = lane / p.K, pk = lane % p.K;            // parse role: bucket in group, peer
  const uint32_t slots_per_bucket = p.d >> 4;                 // 16-coordinate lane slots
  const uint32_t total_slots = p.G * slots_per_bucket;
  const uint64_t groups = (p.B + p.G - 1) / p.G;

  for (uint64_t grp = (uint64_t)blockIdx.x * nwarps + warp; grp < groups; grp += (uint64_t)gridDim.x * nwarps) {
    const uint64_t b0 = grp * p.G;
    for (uint32_t q = lane; q < (warp_words >> 2); q += 32) reinterpret_cast<uint4*>(words)[q] = make_uint4(0u, 0u, 0u, 0u);
    __syncwarp();
    // ---- phase 1: one lane per (bucket, peer) ------------------------------------------------
    const bool mine = pg < p.G && b0 + pg < p.B;
    const uint32_t db = mine ? (uint32_t)min((uint64_t)p.d, p.n - (b0 + pg) * p.d) : 0u;
    StringRef ref;
    ref.words = nullptr; ref.lo = 0; ref.total = 0; ref.err = 0;
    if (mine) ref = string_ref(p.peers, pk, b0 + pg, p.B, db);
    // More than 9.5 bits per coordinate in all strings of the warp: nearly all levels are nonzero (n = 33 M, d = 96, K = 5, N(0, 1),
    // 10 bits 578 -> 528 us; strings of 9 to 9.5 bits that have zeros among their levels lost up to 8 %). All lanes vote.
    const bool ones = __all_sync(0xffffffffu, !mine || ref.err || 2u * ref.total > 19u * db);
    if (mine) {
      uint32_t* bucket = words + pg * p.bucket_words;
      float A;
      const uint32_t st = parse_to_fields(ref, ones, db, p.d, p.s, code, bucket + pk * p.row_words, &A);
      reinterpret_cast<float*>(bucket + p.K * p.row_words)[pk] = A;
      if (st) atomicOr(p.status, st);
    }
    __syncwarp();
    // ---- phase 2: the fixed-width decoder's inner loop over the rebuilt fields ----------------
    for (uint32_t s0 = 0; s0 < total_slots; s0 += 32) {
      const uint32_t slot = s0 + lane;
      const uint32_t g = slot / slots_per_bucket, c = (slot - g * slots_per_bucket) << 4;
      const uint64_t b = b0 + g;
      const uint64_t i0 = b * p.d + c;
      const bool live = slot < total_slots && b < p.B && i0 < p.n;
      const uint32_t* bucket = words + (live ? g : 0) * p.bucket_words;
      const float* scales = reinterpret_cast<const float*>(bucket + p.K * p.row_words);
      float acc[16];
#pragma unroll
      for (int e = 0; e < 16; ++e) acc[e] = 0.f;
#pragma unroll 2
      for (uint32_t k = 0; k < p.K; ++k) {
        const uint32_t* row = bucket + k * p.row_words;
        uint32_t w[4] = {0u, 0u, 0u, 0u};
        uint32_t sb = 0;
        float A = 0.f;
        if (live) {
          A = scales[k];
          sb = (row[level_words + (c >> 5)] >> (c & 31)) & 0xFFFFu;
          const uint4 t = *reinterpret_cast<const uint4*>(row + (c >> 2));
          w[0] = t.x; w[1] = t.y; w[2] = t.z; w[3] = t.w;
        }
        add_peer_bytes(acc, w, sb, A, lq);
      }
      if (live) {
        if (p.map.src) store_span16<FUSED>(out_span(p.out, p.map, b, c, p.d, p.n, 16u), acc, p.c);
        else store_lane16<FUSED>(p.out + i0, acc, i0, p.n, p.c);
      }
    }
    __syncwarp();
  }
}

}  // namespace

int launch_elias_fields(FieldParams& p, bool fused, cudaStream_t stream) {
  static KernelSite site[2];
  int max_smem = 0;
  const int st0 = device_shared_memory(&max_smem);
  if (st0) return st0;
  const uint32_t level_words = p.d >> 2, sign_words = p.d >> 5;
  p.row_words = (level_words + sign_words + 3u) & ~3u;
  p.bucket_words = (p.K * p.row_words + p.K + 3u) & ~3u;
  // CTAs of w warps that an SM holds: the code table and what CUDA reserves are per CTA, the fields per warp; 32 warps by registers.
  const size_t per_cta = 2112, per_sm = 227u << 10;
  constexpr uint32_t kResident = 32, kMostWarps = 10;
  auto ctas_of = [&](uint32_t w, size_t per_warp) {
    if (w * per_warp + per_cta > (size_t)max_smem) return 0u;
    const uint32_t by_memory = (uint32_t)(per_sm / (w * per_warp + per_cta)), by_registers = kResident / w;
    return by_memory < by_registers ? by_memory : by_registers;
  };
  // Warps per CTA: the count that leaves the most resident, since the parse is latency-bound; from four on, so that all schedulers
  // of an SM have some.
  auto most_resident = [&](size_t per_warp, uint32_t* warps) {
    uint32_t best = 0;
    for (uint32_t w = 4; w <= kMostWarps; ++w)
      if (ctas_of(w, per_warp) * w > best) { best = ctas_of(w, per_warp) * w; *warps = w; }
    for (uint32_t w = 3; best == 0u && w >= 1u; --w)
      if (ctas_of(w, per_warp)) { best = ctas_of(w, per_warp) * w; *warps = w; }
    return best;
  };
  int sms = 0, occ = 0;
  int st = device_sms(&sms);
  if (st) return st;
  // Buckets to a warp: a power of two, within 16 KB; or as many as it has lanes for (K = 5, d = 96: 6, where a power of two leaves
  // 12 lanes idle, n = 33 M 792 -> 530 us), where that leaves room for 32 warps on an SM (n = 12 M, d = 256, K = 5: 6 with 25 warps
  // 347 us, 4 with 32 286) and at least ten warps with work to each (n = 769 K, d = 256, K = 9: 3 62 us, 2 54).
  uint32_t G = 32 / p.K, power = 1, warps = 1;
  while (2u * power <= G && (size_t)(2u * power) * p.bucket_words * 4 <= (16u << 10)) power *= 2u;
  while (G > power && most_resident((size_t)G * p.bucket_words * 4, &warps) < kResident) --G;
  if (p.B < 10ull * sms * G) G = power;
  p.G = G;
  const size_t per_warp = (size_t)G * p.bucket_words * 4;
  const uint64_t groups = (p.B + G - 1) / G;
  if (groups <= (uint64_t)sms * most_resident(per_warp, &warps)) {
    // all warps are resident at once: the count that spreads them evenly over the SMs
    uint64_t least = ~0ull;
    for (uint32_t w = kMostWarps; w >= 4u; --w) {
      const uint64_t ctas = ((groups + w - 1) / w + sms - 1) / sms;
      if (ctas * w < least && ctas <= ctas_of(w, per_warp)) { least = ctas * w; warps = w; }
    }
  }
  auto kern = fused ? decode_elias_fields_kernel<true> : decode_elias_fields_kernel<false>;
  const size_t smem = (size_t)warps * per_warp;
  st = site[fused ? 1 : 0].lookup_dynamic(kern, (int)warps * 32, smem, &sms, &occ);
  if (st) return st;
  const uint64_t want = (groups + warps - 1) / warps;
  const uint64_t cap = (uint64_t)sms * occ;
  ScopedKernel sk(kKernDecodeEliasFields, stream);
  return (int)launch_chained(kern, (uint32_t)(want < cap ? want : cap), warps * 32u, smem, stream, p);
}

}  // namespace qsgd
