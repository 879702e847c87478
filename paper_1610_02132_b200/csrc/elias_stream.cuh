// What the decoders with a lane per stream share (elias_decode_ring.cu, elias_decode_dense.cu): accesses to shared memory by
// address and copies in the background. (The sums of a step are written out in each: they differ by the lookup of a value, and by
// what the compiler makes of the loop around it.)
#pragma once

#include "elias_decode.cuh"

namespace qsgd {

__device__ __forceinline__ uint32_t shared_address(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
// A store and a load that happen where `when` holds, without a branch.
__device__ __forceinline__ void store_byte_if(uint32_t when, uint32_t addr, uint32_t v) {
  asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %0, 0;\n\t@p st.shared.u8 [%1], %2;\n\t}" ::"r"(when), "r"(addr), "r"(v)
               : "memory");
}
__device__ __forceinline__ void load_word_if(bool when, uint32_t& v, uint32_t addr) {
  asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %1, 0;\n\t@p ld.shared.u32 %0, [%2];\n\t}" : "+r"(v) : "r"((uint32_t)when), "r"(addr)
               : "memory");
}
__device__ __forceinline__ void store_byte(uint32_t addr, uint32_t v) {
  asm volatile("st.shared.u8 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}
__device__ __forceinline__ uint32_t load_word(uint32_t addr) {
  uint32_t v;
  asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ void load_words(uint32_t addr, uint32_t& a, uint32_t& b) {
  asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(a), "=r"(b) : "r"(addr) : "memory");
}
// 16 bytes from global to shared memory, in the background; and the wait for all of this thread's.
__device__ __forceinline__ void copy16(uint32_t addr, const void* from) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(addr), "l"(from) : "memory");
}
__device__ __forceinline__ void copies_done() { asm volatile("cp.async.wait_all;" ::: "memory"); }
__device__ __forceinline__ void zero_quad(uint32_t addr) {
  asm volatile("st.shared.v4.u32 [%0], {%1, %1, %1, %1};" ::"r"(addr), "r"(0) : "memory");
}

}  // namespace qsgd
