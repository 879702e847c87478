// Quantizing and packing as the fixed-width encoder (quantize_fixed.cu) and the encoder of small Elias messages
// (elias_encode_small.cu) share it: Philox uniforms, stochastic rounding and bit packing of 16 coordinates of a
// thread, and the tile code for any bucket size.
#pragma once

#include <float.h>

#include "qsgd_common.cuh"

namespace qsgd {

constexpr int kQuantizeThreads = 256;
constexpr int kTile = 4096;           // coordinates per tile

// What of a Philox block's work depends on seed, step and worker alone (philox_q).
struct PhiloxConsts {
  uint32_t y0;        // worker ^ k1[0]
  uint32_t z0;        // lo(M1 * step) ^ k0[1]
  uint32_t z1;        // hi(M0 * x0) ^ k1[1],  x0 = hi(M1 * step) ^ k0[0]
  uint32_t z2;        // lo(M0 * x0) ^ k1[2]
  uint32_t k0_2;      // k0[2]
  uint32_t k[7][2];   // round keys 3 .. 9
};

struct QuantizeParams {
  const float* g;
  uint64_t n;
  uint32_t d;
  uint32_t s;
  uint32_t tile_coords;   // generic kernel: coordinates per tile = whole buckets, <= kTile
  uint64_t coord_base;    // generic kernel: first coordinate it is responsible for
  float* A_out;
  uint32_t* sign_out;
  uint32_t* level_out;
  uint64_t B, sign_words, level_words;
  uint64_t tiles;
  uint32_t* status;
  uint64_t* info;         // optional: the four message-info words of a fixed-width message
  uint64_t total_bytes;
  ClearWords clear;
  BucketMap map;          // per-tensor policy: where each bucket lives in g, or no map
  PhiloxConsts pc;
};

// By all threads of one CTA.
__device__ __forceinline__ void clear_words(const ClearWords& c) {
  for (uint32_t i = threadIdx.x; i < c.count; i += kQuantizeThreads) c.at[i] = 0ull;
}

__device__ __forceinline__ float fma_rn(float a, float b, float c) {
  float r;
  asm("fma.rn.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}

// ---------------------------------------------------------------------------------------------
// Philox4x32-10 for the counter (q, 0, step, worker) with everything that does not depend on q
// folded into kernel-uniform constants on the host: after round 0 two of the four words are
// constants, which also makes one product of round 1 a constant. 37 instead of 40
// multiply / xor instructions per block of four uniforms.
// ---------------------------------------------------------------------------------------------

constexpr uint32_t kM0 = 0xD2511F53u, kM1 = 0xCD9E8D57u;

__device__ __forceinline__ uint4 philox_q(uint32_t q, const PhiloxConsts& pc) {
  // round 0: (q, 0, step, worker) -> (x0, l1, hi(M0 q) ^ y0, lo(M0 q))
  uint64_t p0 = (uint64_t)kM0 * q;
  uint32_t a2 = (uint32_t)(p0 >> 32) ^ pc.y0, a3 = (uint32_t)p0;
  // round 1: (x0, l1, a2, a3) -> (hi(M1 a2) ^ z0, lo(M1 a2), a3 ^ z1, lo(M0 x0))
  uint64_t p1 = (uint64_t)kM1 * a2;
  uint32_t c0 = (uint32_t)(p1 >> 32) ^ pc.z0, c1 = (uint32_t)p1, c2 = a3 ^ pc.z1;
  // round 2: c3 = lo(M0 x0) is folded into z2
  p0 = (uint64_t)kM0 * c0;
  p1 = (uint64_t)kM1 * c2;
  c0 = (uint32_t)(p1 >> 32) ^ c1 ^ pc.k0_2;
  c1 = (uint32_t)p1;
  c2 = (uint32_t)(p0 >> 32) ^ pc.z2;
  uint32_t c3 = (uint32_t)p0;
  // rounds 3 .. 9: the high and low halves by separate multiplies (measured slightly faster than the
  // 64-bit products here; the first rounds stay as they are, where it measured slower)
#pragma unroll
  for (int r = 0; r < 7; ++r) {
    const uint32_t h0 = __umulhi(kM0, c0), l0 = kM0 * c0;
    const uint32_t h1 = __umulhi(kM1, c2), l1 = kM1 * c2;
    c0 = h1 ^ c1 ^ pc.k[r][0];
    c1 = l1;
    c2 = h0 ^ c3 ^ pc.k[r][1];
    c3 = l0;
  }
  return make_uint4(c0, c1, c2, c3);
}

// The uniforms of the 16 coordinates of one thread (Philox blocks q0 .. q0 + 3) as fp32 bit
// patterns m = word >> 8 (see quantize_one).
__device__ __forceinline__ void philox_uniforms16(uint32_t q0, const PhiloxConsts& pc, float (&um)[16]) {
#pragma unroll
  for (int b = 0; b < 4; ++b) {
    const uint4 w = philox_q(q0 + b, pc);
    um[4 * b] = __uint_as_float(w.x >> 8);
    um[4 * b + 1] = __uint_as_float(w.y >> 8);
    um[4 * b + 2] = __uint_as_float(w.z >> 8);
    um[4 * b + 3] = __uint_as_float(w.w >> 8);
  }
}

constexpr float kTwo23 = 8388608.0f;
constexpr uint32_t kTwo23Bits = 0x4B000000u;

constexpr float kTwo125 = 4.253529586511730793292182592897102643e+37f;

// One coordinate. Returns the raw bits of 2^23 + level (level clamped to s when CLAMP); pushes the
// sign bit into `sw`. `um` is the bit pattern m = top 24 Philox bits read as an fp32, i.e. m * 2^-149.
// RAW_SIGN: push the sign bit of v as it is; the caller clears the signs of zero levels afterwards
// with a mask derived from the packed level words (cheaper than two more operations per coordinate
// when a word holds many fields). NAN_ZERO: a t that is no number (a NaN coordinate, or an infinite one in its own
// infinite scale) gives level 0 instead of s.
template <bool RAW_SIGN, bool CLAMP, bool NAN_ZERO = false>
__device__ __forceinline__ uint32_t quantize_one(float v, float r, float sf, float cap, float um,
                                                 uint32_t& sw) {
  float t = __fmul_rn(__fmul_rn(sf, fabsf(v)), r);
  if (NAN_ZERO) t = fmaxf(t, 0.0f);
  const float c = fma_rn(um, kTwo125, t);                    // t + m * 2^-24, one rounding
  float fl = __fadd_rd(c, kTwo23);                           // 2^23 + floor(c)
  if (CLAMP) fl = fminf(fl, cap);                            // 2^23 + min(floor(c), s)
  if (RAW_SIGN) {
    sw = __funnelshift_l(__float_as_uint(v), sw, 1);
  } else {
    const float lf = __fsub_rn(fl, kTwo23);                 // the level as a float, exact
    const float sv = fma_rn(lf, v, 0.0f);                   // sign set iff level > 0 and v < 0
    sw = __funnelshift_l(__float_as_uint(sv), sw, 1);
  }
  return __float_as_uint(fl);
}

// Rounds and packs the 16 coordinates of a thread, highest first: level fields by Horner
// multiply-adds on the raw float bits (the constant exponent bits are removed once per word),
// sign bits by funnel shifts; signs of zero levels are cleared at the end.
template <int LB, bool CLAMP>
__device__ __forceinline__ void quantize16(const float (&v)[16], const float (&um)[16], float r, float sf,
                                           float cap, uint32_t (&lw)[4], uint32_t& sw) {
  sw = 0;
#pragma unroll
  for (int j = 0; j < 4; ++j) lw[j] = 0u;                 // LB = 8: 4 words; 4: 2; 2: 1; 1: half
#pragma unroll
  for (int c4 = 3; c4 >= 0; --c4) {
#pragma unroll
    for (int e = 3; e >= 0; --e) {
      const uint32_t bits = quantize_one<LB != 8, CLAMP>(v[4 * c4 + e], r, sf, cap, um[4 * c4 + e], sw);
      if (LB == 8) lw[c4] = lw[c4] * 256u + bits;
      else if (LB == 4) lw[c4 >> 1] = lw[c4 >> 1] * 16u + bits;
      else if (LB == 2) lw[0] = lw[0] * 4u + bits;
      else lw[0] = lw[0] * 2u + bits;
    }
  }
  // remove the exponent bits that rode along: sum over the fields of 0x4B000000 << (LB * e)
  if (LB == 8) {
#pragma unroll
    for (int j = 0; j < 4; ++j) lw[j] -= kTwo23Bits * 0x01010101u;
  } else if (LB == 4) {
    lw[0] -= kTwo23Bits * 0x11111111u;
    lw[1] -= kTwo23Bits * 0x11111111u;
  } else if (LB == 2) {
    lw[0] -= kTwo23Bits * 0x55555555u;
  } else {
    lw[0] = (lw[0] - kTwo23Bits * 0xFFFFu) & 0xFFFFu;
  }
}

// Bit e of the result is set iff level field e of the 16 coordinates packed in lw is nonzero.
template <int LB>
__device__ __forceinline__ uint32_t nonzero_fields16(const uint32_t (&lw)[4]) {
  if (LB == 1) return lw[0] & 0xFFFFu;
  if (LB == 2) {
    uint32_t y = (lw[0] | (lw[0] >> 1)) & 0x55555555u;
    y = (y | (y >> 1)) & 0x33333333u;
    y = (y | (y >> 2)) & 0x0F0F0F0Fu;
    y = (y | (y >> 4)) & 0x00FF00FFu;
    return (y | (y >> 8)) & 0xFFFFu;
  }
  uint32_t m = 0;                                           // LB == 4: two words of eight fields
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    uint32_t y = lw[h] | (lw[h] >> 1);
    y = (y | (y >> 2)) & 0x11111111u;
    y = (y | (y >> 3)) & 0x03030303u;
    y = (y | (y >> 6)) & 0x000F000Fu;
    m |= ((y | (y >> 12)) & 0xFFu) << (8 * h);
  }
  return m;
}

// Stores the sign and level words of the 16 coordinates of every lane of a warp; `c` is the index
// of the warp's chunk of 512 coordinates (complete chunks only: no bounds to check).
template <int LB>
__device__ __forceinline__ void store_chunk(uint32_t* sign_out, uint32_t* level_out, uint32_t c, uint32_t lane,
                                            uint32_t sw, const uint32_t (&lw)[4]) {
  {
    uint32_t w = (sw & 0xFFFFu) << (16 * (lane & 1));
    w |= __shfl_xor_sync(0xffffffffu, w, 1);
    if ((lane & 1) == 0) sign_out[c * 16u + (lane >> 1)] = w;
  }
  if (LB == 8) {
    *reinterpret_cast<uint4*>(level_out + ((size_t)c * 128u + lane * 4u)) = make_uint4(lw[0], lw[1], lw[2], lw[3]);
  } else if (LB == 4) {
    *reinterpret_cast<uint2*>(level_out + ((size_t)c * 64u + lane * 2u)) = make_uint2(lw[0], lw[1]);
  } else if (LB == 2) {
    level_out[(size_t)c * 32u + lane] = lw[0];
  } else {
    uint32_t w = lw[0] << (16 * (lane & 1));
    w |= __shfl_xor_sync(0xffffffffu, w, 1);
    if ((lane & 1) == 0) level_out[c * 16u + (lane >> 1)] = w;
  }
}

// ---------------------------------------------------------------------------------------------
// Generic tile: any bucket size that is a multiple of 32. One CTA per tile of whole buckets.
// ---------------------------------------------------------------------------------------------
constexpr int kGroupsPerThread = kTile / 8 / kQuantizeThreads;  // 2
constexpr int kMaxBucketsPerTile = kTile / 32;          // 128

// One tile of the generic path. `block` / `nblocks` play the role of blockIdx / gridDim so that the
// main kernel can run the ragged last tile in one extra CTA of its own grid.
template <int LB, int NORM, bool MAPPED>
__device__ __forceinline__ void quantize_generic_tile(const QuantizeParams& p, uint32_t block, uint32_t nblocks,
                                                      float* tile, float* part, float* s_rcp) {
  const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint64_t t0 = p.coord_base + (uint64_t)block * p.tile_coords;   // first coordinate
  if (block == 0 && tid == 0 && p.info) {
    p.info[0] = 8 * p.total_bytes; p.info[1] = 0; p.info[2] = p.total_bytes; p.info[3] = 0;
  }
  const uint64_t left = p.n - t0;
  const uint32_t valid = left < p.tile_coords ? (uint32_t)left : p.tile_coords;
  if (valid == 0) {                            // nothing left to encode: only the padding
    if (tid < 4) {
      if (p.B + tid < ((p.B + 3) & ~3ull)) p.A_out[p.B + tid] = 0.f;
      if (p.sign_words + tid < ((p.sign_words + 3) & ~3ull)) p.sign_out[p.sign_words + tid] = 0u;
      if (p.level_words + tid < ((p.level_words + 3) & ~3ull)) p.level_out[p.level_words + tid] = 0u;
    }
    return;
  }

  for (uint32_t i = tid * 4; i < p.tile_coords; i += kQuantizeThreads * 4) {
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (MAPPED) {
      // per-tensor policy: four coordinates of one bucket (d is a multiple of 32) from the
      // bucket's own place; what lies behind the bucket's length is zero padding
      if (i < valid) {
        const uint32_t bi = i / p.d, c = i - bi * p.d;
        const uint64_t b = t0 / p.d + bi;
        const uint32_t L = __ldg(p.map.len + b);
        const float* src = p.g + __ldg(p.map.src + b) + c;
        if (c + 4 <= L && (reinterpret_cast<uintptr_t>(src) & 15u) == 0) {
          v = __ldcs(reinterpret_cast<const float4*>(src));
        } else {
          float t[4] = {0.f, 0.f, 0.f, 0.f};
          for (uint32_t j = 0; j < 4 && c + j < L; ++j) t[j] = src[j];
          v = make_float4(t[0], t[1], t[2], t[3]);
        }
      }
    } else if (i + 4 <= valid) {
      v = __ldcs(reinterpret_cast<const float4*>(p.g + t0 + i));
    } else if (i < valid) {
      float t[4] = {0.f, 0.f, 0.f, 0.f};
      for (uint32_t j = 0; i + j < valid; ++j) t[j] = p.g[t0 + i + j];
      v = make_float4(t[0], t[1], t[2], t[3]);
    }
    *reinterpret_cast<float4*>(tile + i) = v;
  }
  __syncthreads();

  float v[kGroupsPerThread][8];
  const uint32_t groups = p.tile_coords >> 3;
#pragma unroll
  for (int j = 0; j < kGroupsPerThread; ++j) {
    const uint32_t grp = tid + j * kQuantizeThreads;
    float4 a = make_float4(0.f, 0.f, 0.f, 0.f), b = a;
    if (grp < groups) {
      a = *reinterpret_cast<const float4*>(tile + grp * 8);
      b = *reinterpret_cast<const float4*>(tile + grp * 8 + 4);
    }
    v[j][0] = a.x; v[j][1] = a.y; v[j][2] = a.z; v[j][3] = a.w;
    v[j][4] = b.x; v[j][5] = b.y; v[j][6] = b.z; v[j][7] = b.w;
    float acc = 0.f;
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      if (NORM == QSGD_NORM_L2) acc = fmaf(v[j][e], v[j][e], acc);
      else acc = fmaxf(acc, fabsf(v[j][e]));
    }
    if (grp < groups) part[grp] = acc;
  }
  __syncthreads();

  const uint32_t nb = p.tile_coords / p.d;     // buckets in a full tile
  const uint32_t gpb = p.d >> 3;               // groups per bucket
  const uint64_t b0 = t0 / p.d;                // first bucket of the tile
  for (uint32_t b = warp; b < nb; b += kQuantizeThreads / 32) {
    float A;
    if (NORM == QSGD_NORM_L2) {
      // fp32 partials of 8 squares each; redo in fp64 from the tile when they may have lost bits:
      // a nonzero partial outside [8e-28, 1e30], or a bucket total below that range (a zero total
      // too: squares below 1.4e-45 vanish in fp32 while the values do not in fp64)
      double acc = 0.0;
      bool shaky = false;
      for (uint32_t j = lane; j < gpb; j += 32) {
        const float q = part[b * gpb + j];
        shaky |= !(q >= 8.0e-28f && q <= 1.0e30f) && q != 0.f;
        acc += (double)q;
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
      if (__any_sync(0xffffffffu, shaky) || !(acc >= 8.0e-28)) {
        acc = 0.0;
        for (uint32_t i = lane; i < p.d; i += 32) {
          const double x = (double)tile[b * p.d + i];
          acc = fma(x, x, acc);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
      }
      A = __double2float_rn(__dsqrt_rn(acc));
    } else {
      float acc = 0.f;
      for (uint32_t j = lane; j < gpb; j += 32) acc = fmaxf(acc, part[b * gpb + j]);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) acc = fmaxf(acc, __shfl_xor_sync(0xffffffffu, acc, o));
      A = acc;
    }
    if (!(A >= FLT_MIN)) A = 0.f;
    if (lane == 0) {
      s_rcp[b] = A > 0.f ? __frcp_rn(A) : 0.f;
      if (b0 + b < p.B) p.A_out[b0 + b] = A;
    }
  }
  __syncthreads();

  const float sf = (float)p.s;
#pragma unroll
  for (int j = 0; j < kGroupsPerThread; ++j) {
    const uint32_t grp = tid + j * kQuantizeThreads;
    const uint32_t bl = (grp * 8) / p.d;
    const float r = (grp < groups) ? s_rcp[bl] : 0.f;
    const uint32_t q = (uint32_t)((t0 + (uint64_t)grp * 8) >> 2);        // n <= 2^32
    const uint4 ra = philox_q(q, p.pc), rb = philox_q(q + 1u, p.pc);
    const uint32_t rnd[8] = {ra.x, ra.y, ra.z, ra.w, rb.x, rb.y, rb.z, rb.w};
    uint32_t sb = 0, lo = 0, hi = 0;             // fields of coordinates 0 .. 3 and 4 .. 7 (LB = 8), else of all in lo
#pragma unroll
    for (int e = 7; e >= 0; --e) {
      const uint32_t bits = quantize_one<false, true, true>(v[j][e], r, sf, kTwo23 + sf, __uint_as_float(rnd[e] >> 8), sb);
      if (LB == 8 && e >= 4) hi = hi * 256u + bits;
      else lo = lo * (1u << LB) + bits;
    }
    // the exponent bits that rode along (they leave the low 24 bits alone)
    if (LB == 8) { lo -= kTwo23Bits * 0x01010101u; hi -= kTwo23Bits * 0x01010101u; }
    else if (LB == 4) lo -= kTwo23Bits * 0x11111111u;
    else lo &= (1u << (8 * LB & 31)) - 1u;
    uint32_t sw = (sb & 0xFFu) << (8 * (lane & 3));
    sw |= __shfl_xor_sync(0xffffffffu, sw, 1);
    sw |= __shfl_xor_sync(0xffffffffu, sw, 2);
    const uint64_t sidx = (t0 >> 5) + (grp >> 2);
    if ((lane & 3) == 0 && grp < groups && sidx < p.sign_words) p.sign_out[sidx] = sw;

    if (LB == 8) {
      const uint32_t w0 = lo, w1 = hi;
      const uint64_t widx = (t0 >> 2) + (uint64_t)grp * 2;
      if (grp < groups) {
        if (widx + 1 < p.level_words) *reinterpret_cast<uint2*>(p.level_out + widx) = make_uint2(w0, w1);
        else if (widx < p.level_words) p.level_out[widx] = w0;
      }
    } else if (LB == 4) {
      const uint32_t w = lo;
      const uint64_t widx = (t0 >> 3) + grp;
      if (grp < groups && widx < p.level_words) p.level_out[widx] = w;
    } else if (LB == 2) {
      uint32_t w = lo << (16 * (lane & 1));
      w |= __shfl_xor_sync(0xffffffffu, w, 1);
      const uint64_t widx = (t0 >> 4) + (grp >> 1);
      if ((lane & 1) == 0 && grp < groups && widx < p.level_words) p.level_out[widx] = w;
    } else {
      uint32_t w = lo << (8 * (lane & 3));
      w |= __shfl_xor_sync(0xffffffffu, w, 1);
      w |= __shfl_xor_sync(0xffffffffu, w, 2);
      const uint64_t widx = (t0 >> 5) + (grp >> 2);
      if ((lane & 3) == 0 && grp < groups && widx < p.level_words) p.level_out[widx] = w;
    }
  }

  if (block == nblocks - 1 && tid < 4) {
    if (p.B + tid < ((p.B + 3) & ~3ull)) p.A_out[p.B + tid] = 0.f;
    if (p.sign_words + tid < ((p.sign_words + 3) & ~3ull)) p.sign_out[p.sign_words + tid] = 0u;
    if (p.level_words + tid < ((p.level_words + 3) & ~3ull)) p.level_out[p.level_words + tid] = 0u;
  }
}

inline PhiloxConsts make_philox_consts(uint64_t seed, uint32_t step, uint32_t worker) {
  uint32_t k0[10], k1[10];
  k0[0] = (uint32_t)seed; k1[0] = (uint32_t)(seed >> 32);
  for (int r = 1; r < 10; ++r) { k0[r] = k0[r - 1] + 0x9E3779B9u; k1[r] = k1[r - 1] + 0xBB67AE85u; }
  const uint64_t ps = (uint64_t)kM1 * step;
  const uint32_t x0 = (uint32_t)(ps >> 32) ^ k0[0], l1 = (uint32_t)ps;
  const uint64_t px = (uint64_t)kM0 * x0;
  PhiloxConsts pc;
  pc.y0 = worker ^ k1[0];
  pc.z0 = l1 ^ k0[1];
  pc.z1 = (uint32_t)(px >> 32) ^ k1[1];
  pc.z2 = (uint32_t)px ^ k1[2];
  pc.k0_2 = k0[2];
  for (int r = 0; r < 7; ++r) { pc.k[r][0] = k0[r + 3]; pc.k[r][1] = k1[r + 3]; }
  return pc;
}

}  // namespace qsgd
