// What the decoders share: reconstruction of +-A * (level / s) from the fields of a fixed-width message, the places of
// coordinates in the output, stores of sums and of the step.
#pragma once

#include "qsgd_common.cuh"

namespace qsgd {

__device__ __forceinline__ float shfl_f(float v, uint32_t src) {
  return __shfl_sync(0xffffffffu, v, (int)src);
}

// Two floats in a register pair, and the operations on both at once: one issue slot for two.
typedef unsigned long long float2p;
__device__ __forceinline__ float2p pair2(float a, float b) {
  float2p r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ float2 unpair2(float2p v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ float2p fma2(float2p a, float2p b, float2p c) {
  float2p r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ float2p add2(float2p a, float2p b) {
  float2p r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
// acc + RN(A * v). The product is an fma with -0 that the compiler cannot see (a kernel parameter), because ptxas contracts a
// mul.rn.f32x2 in front of an add.rn.f32x2.
__device__ __forceinline__ float2p add_product2(float2p acc, float A, float v0, float v1, float minus_zero) {
  return add2(acc, fma2(pair2(A, A), pair2(v0, v1), pair2(minus_zero, minus_zero)));
}

// Adds peer k's 16 values to acc[] (coordinates 2 j and 2 j + 1 in acc[j]). SINGLE: the whole chunk lies in one bucket and
// `lut` is already scaled by A; otherwise `lut` holds +-(level / s) and A is this lane's bucket scale.
template <bool SINGLE>
__device__ __forceinline__ float2p add_pair_lut(float2p acc, uint32_t i0, uint32_t i1, float lut, float A, float minus_zero) {
  const float a = shfl_f(lut, i0), b = shfl_f(lut, i1);
  return SINGLE ? add2(acc, pair2(a, b)) : add_product2(acc, A, a, b, minus_zero);
}

template <int LB, bool SINGLE, int W>
__device__ __forceinline__ void add_peer_lut(float2p (&acc)[8], const uint32_t (&w)[W], uint32_t sb,
                                             float lut, float A, float minus_zero) {
  if (LB == 4) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const uint32_t word = w[h % W], s8 = sb >> (8 * h);
      const uint32_t ev = word & 0x0F0F0F0Fu, od = (word >> 4) & 0x0F0F0F0Fu;
      const uint32_t ie = (((s8 & 0x55u) * 0x00410410u) & 0x10101010u) | ev;   // coords 0,2,4,6
      const uint32_t io = (((s8 & 0xAAu) * 0x00208208u) & 0x10101010u) | od;   // coords 1,3,5,7
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[4 * h + j] = add_pair_lut<SINGLE>(acc[4 * h + j], ie >> (8 * j), io >> (8 * j), lut, A, minus_zero);
    }
  } else if (LB == 2) {
    // 16 two-bit levels in w[0]. Per half (8 coordinates) spread the levels to nibble spacing
    // and drop the sign bit at bit 2 of each nibble; the lookup table repeats every 8 lanes, so
    // whatever follows in the shifted word is ignored by the shuffle (it reads 5 index bits).
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      uint32_t x = (w[0] >> (16 * h)) & 0xFFFFu;
      x = (x | (x << 8)) & 0x00FF00FFu;
      x = (x | (x << 4)) & 0x0F0F0F0Fu;
      x = (x | (x << 2)) & 0x33333333u;
      uint32_t y = (sb >> (8 * h)) & 0xFFu;
      y = (y | (y << 12)) & 0x000F000Fu;
      y = (y | (y << 6)) & 0x03030303u;
      y = (y | (y << 3)) & 0x11111111u;
      const uint32_t z = x | (y << 2);
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[4 * h + j] = add_pair_lut<SINGLE>(acc[4 * h + j], z >> (8 * j), z >> (8 * j + 4), lut, A, minus_zero);
    }
  } else {
    // LB = 1: interleave the 16 level bits (even positions) with the 16 sign bits (odd); the
    // lookup table repeats every 4 lanes.
    uint32_t x = w[0] & 0xFFFFu, y = sb & 0xFFFFu;
    x = (x | (x << 8)) & 0x00FF00FFu; y = (y | (y << 8)) & 0x00FF00FFu;
    x = (x | (x << 4)) & 0x0F0F0F0Fu; y = (y | (y << 4)) & 0x0F0F0F0Fu;
    x = (x | (x << 2)) & 0x33333333u; y = (y | (y << 2)) & 0x33333333u;
    x = (x | (x << 1)) & 0x55555555u; y = (y | (y << 1)) & 0x55555555u;
    const uint32_t z = x | (y << 1);
#pragma unroll
    for (int j = 0; j < 8; ++j) acc[j] = add_pair_lut<SINGLE>(acc[j], z >> (4 * j), z >> (4 * j + 2), lut, A, minus_zero);
  }
}

// LB = 8: table lookup of +-(level / s) in shared memory: level l, sign g of lane t at byte 256 l + 128 g + 4 t behind the
// address 65536, so that lanes never meet in a bank and one byte permute makes an address: of the level's byte, a byte that
// holds 128 g + 4 t, and the base.
template <int W>
__device__ __forceinline__ void add_peer_tab(float2p (&acc)[8], const uint32_t (&w)[W], uint32_t sb, uint32_t lane, float A,
                                             float minus_zero) {
#pragma unroll
  for (int h = 0; h < 4; ++h) {
    // the signs of four coordinates into the highest bits of four bytes: bit j times 2^(7 + 7 j) (no two products meet)
    const uint32_t four = h & 1 ? ((sb >> (4 * (h & 2))) & 0xF0u) * 0x01020408u : ((sb >> (4 * (h & 2))) & 0x0Fu) * 0x10204080u;
    const uint32_t t = (four & 0x80808080u) | lane * 0x04040404u;
    const uint32_t t01 = __byte_perm(t, 1u, 0x5410u), t23 = __byte_perm(t, 1u, 0x5432u);
    float v[4];
#pragma unroll
    for (uint32_t j = 0; j < 4; ++j)
      asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v[j]) : "r"(__byte_perm(w[h % W], j < 2 ? t01 : t23, 0x7600u | j << 4 | (4u + (j & 1u)))));
#pragma unroll
    for (int j = 0; j < 2; ++j) acc[2 * h + j] = add_product2(acc[2 * h + j], A, v[2 * j], v[2 * j + 1], minus_zero);
  }
}

// Writes 16 accumulated values of one lane: acc as it is, or the SGD step x <- x - c * acc.
template <bool FUSED>
__device__ __forceinline__ void store_lane16(float* o, const float (&acc)[16], uint64_t i0, uint64_t n,
                                             float c) {
  if (i0 + 16 <= n) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      float4 r = make_float4(acc[4 * j], acc[4 * j + 1], acc[4 * j + 2], acc[4 * j + 3]);
      if (FUSED) {
        const float4 x = *reinterpret_cast<const float4*>(o + 4 * j);
        r.x = __fsub_rn(x.x, __fmul_rn(c, r.x)); r.y = __fsub_rn(x.y, __fmul_rn(c, r.y));
        r.z = __fsub_rn(x.z, __fmul_rn(c, r.z)); r.w = __fsub_rn(x.w, __fmul_rn(c, r.w));
      }
      *reinterpret_cast<float4*>(o + 4 * j) = r;
    }
  } else {
#pragma unroll
    for (int e = 0; e < 16; ++e)
      if (i0 + e < n) o[e] = FUSED ? __fsub_rn(o[e], __fmul_rn(c, acc[e])) : acc[e];
  }
}

// Where `want` consecutive coordinates of bucket b, starting at bucket-relative position c0, live in
// the output array, and how many of them exist.
struct OutSpan {
  float* ptr;
  uint32_t valid;
};

__device__ __forceinline__ OutSpan out_span(float* out, const BucketMap& map, uint64_t b, uint32_t c0, uint32_t d,
                                            uint64_t n, uint32_t want) {
  OutSpan sp;
  if (map.src) {
    const uint32_t L = __ldg(map.len + b);
    sp.ptr = out + __ldg(map.src + b) + c0;
    sp.valid = c0 < L ? min(want, L - c0) : 0u;
  } else {
    const uint64_t i0 = b * d + c0;
    sp.ptr = out + i0;
    sp.valid = i0 < n ? (uint32_t)min((uint64_t)want, n - i0) : 0u;
  }
  return sp;
}

// store_lane16 through a span: vector accesses when all 16 values exist and the place is 16-byte
// aligned, element by element otherwise.
template <bool FUSED>
__device__ __forceinline__ void store_span16(const OutSpan& sp, const float (&acc)[16], float c) {
  if (sp.valid == 16u && (reinterpret_cast<uintptr_t>(sp.ptr) & 15u) == 0) {
    store_lane16<FUSED>(sp.ptr, acc, 0, 16, c);
  } else {
#pragma unroll
    for (int e = 0; e < 16; ++e)
      if ((uint32_t)e < sp.valid) sp.ptr[e] = FUSED ? __fsub_rn(sp.ptr[e], __fmul_rn(c, acc[e])) : acc[e];
  }
}

// The same for 8 values.
template <bool FUSED>
__device__ __forceinline__ void store_span8(const OutSpan& sp, const float (&acc)[8], float c) {
  if (sp.valid == 8u && (reinterpret_cast<uintptr_t>(sp.ptr) & 15u) == 0) {
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      float4 r = make_float4(acc[4 * j], acc[4 * j + 1], acc[4 * j + 2], acc[4 * j + 3]);
      if (FUSED) {
        const float4 x = *reinterpret_cast<const float4*>(sp.ptr + 4 * j);
        r.x = __fsub_rn(x.x, __fmul_rn(c, r.x)); r.y = __fsub_rn(x.y, __fmul_rn(c, r.y));
        r.z = __fsub_rn(x.z, __fmul_rn(c, r.z)); r.w = __fsub_rn(x.w, __fmul_rn(c, r.w));
      }
      *reinterpret_cast<float4*>(sp.ptr + 4 * j) = r;
    }
  } else {
#pragma unroll
    for (int e = 0; e < 8; ++e)
      if ((uint32_t)e < sp.valid) sp.ptr[e] = FUSED ? __fsub_rn(sp.ptr[e], __fmul_rn(c, acc[e])) : acc[e];
  }
}

// A warp's chunk of 512 sums, 16 consecutive ones a lane: acc as it is, or the SGD step. Where the chunk lies in one piece, the
// lanes pass their quads through `turn` (2 KB of the warp's shared memory), so that accesses to `out` are to 512 consecutive
// bytes: with 16 bytes out of every 64 they were a quarter of the fixed-width decoder's L1 wavefronts. The chunk at the end of
// the vector goes the same way, a quad at a time (by its lanes' 16 sums, with code of its own, a ragged decode of some thousand
// coordinates took 0.3 to 0.5 us of 3 longer). SINGLE: the chunk lies in one bucket.
template <bool FUSED, bool SINGLE>
__device__ __forceinline__ void store_chunk16(float* out, const BucketMap& map, const float2p (&acc)[8], uint32_t turn, uint32_t ch,
                                              uint32_t log2_chunks_per_bucket, uint32_t d, uint64_t n, float c, uint32_t lane) {
  const uint64_t i0 = (uint64_t)ch * 512u, i = i0 + lane * 16u;
  if (SINGLE || !map.src) {
    OutSpan sp;
    if (map.src) {
      const uint32_t b = ch >> log2_chunks_per_bucket;
      sp = out_span(out, map, b, (ch - (b << log2_chunks_per_bucket)) * 512u, d, n, 512u);
    } else {
      sp.ptr = out + i0;
      sp.valid = (uint32_t)min((uint64_t)512u, n - i0);
    }
    const bool quads = (reinterpret_cast<uintptr_t>(sp.ptr) & 15u) == 0;
    // quad j of lane l at 4 l + (j ^ (l / 2 & 3)): eight lanes at a time in eight groups of banks, both ways
#pragma unroll
    for (uint32_t j = 0; j < 4; ++j) {
      const float2 a = unpair2(acc[2 * j]), b = unpair2(acc[2 * j + 1]);
      asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(turn + (lane * 4u + (j ^ ((lane >> 1) & 3u))) * 16u),
                   "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y) : "memory");
    }
    float* o = sp.ptr + lane * 4u;                                        // quad 32 j + lane: from o + 128 j on
    const uint32_t from = turn + (lane ^ ((lane >> 3) & 3u)) * 16u;
    const uint32_t left = sp.valid > lane * 4u ? sp.valid - lane * 4u : 0u;
    if (quads && sp.valid == 512u) {              // nothing to ask for each quad: 1 % of a large decode
      float4 x[4];
      if (FUSED)
#pragma unroll
        for (uint32_t j = 0; j < 4; ++j) x[j] = *reinterpret_cast<const float4*>(o + j * 128u);
      __syncwarp();
#pragma unroll
      for (uint32_t j = 0; j < 4; ++j) {
        float4 r;
        asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(r.x), "=f"(r.y), "=f"(r.z), "=f"(r.w) : "r"(from + j * 512u) : "memory");
        if (FUSED) {
          r.x = __fsub_rn(x[j].x, __fmul_rn(c, r.x)); r.y = __fsub_rn(x[j].y, __fmul_rn(c, r.y));
          r.z = __fsub_rn(x[j].z, __fmul_rn(c, r.z)); r.w = __fsub_rn(x[j].w, __fmul_rn(c, r.w));
        }
        *reinterpret_cast<float4*>(o + j * 128u) = r;
      }
      __syncwarp();                               // before the next chunk's quads
      return;
    }
    float4 x[4];
    if (FUSED)
#pragma unroll
      for (uint32_t j = 0; j < 4; ++j) {
        if (quads && left >= j * 128u + 4u) {
          x[j] = *reinterpret_cast<const float4*>(o + j * 128u);
        } else {
          x[j] = make_float4(0.f, 0.f, 0.f, 0.f);
          if (left > j * 128u) x[j].x = o[j * 128u];
          if (left > j * 128u + 1u) x[j].y = o[j * 128u + 1u];
          if (left > j * 128u + 2u) x[j].z = o[j * 128u + 2u];
          if (left > j * 128u + 3u) x[j].w = o[j * 128u + 3u];
        }
      }
    __syncwarp();
#pragma unroll
    for (uint32_t j = 0; j < 4; ++j) {
      float4 r;
      asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(r.x), "=f"(r.y), "=f"(r.z), "=f"(r.w) : "r"(from + j * 512u) : "memory");
      if (FUSED) {
        r.x = __fsub_rn(x[j].x, __fmul_rn(c, r.x)); r.y = __fsub_rn(x[j].y, __fmul_rn(c, r.y));
        r.z = __fsub_rn(x[j].z, __fmul_rn(c, r.z)); r.w = __fsub_rn(x[j].w, __fmul_rn(c, r.w));
      }
      if (quads && left >= j * 128u + 4u) {
        *reinterpret_cast<float4*>(o + j * 128u) = r;
      } else {
        if (left > j * 128u) o[j * 128u] = r.x;
        if (left > j * 128u + 1u) o[j * 128u + 1u] = r.y;
        if (left > j * 128u + 2u) o[j * 128u + 2u] = r.z;
        if (left > j * 128u + 3u) o[j * 128u + 3u] = r.w;
      }
    }
    __syncwarp();                                 // before the next chunk's quads
    return;
  }
  if (i >= n) return;                             // per-tensor policy, several buckets to a chunk: each lives elsewhere
  float v[16];
#pragma unroll
  for (int j = 0; j < 8; ++j) { const float2 a = unpair2(acc[j]); v[2 * j] = a.x; v[2 * j + 1] = a.y; }
  const uint64_t b = i / d;
  store_span16<FUSED>(out_span(out, map, b, (uint32_t)(i - b * d), d, n, 16u), v, c);
}

}  // namespace qsgd
