// Exchange words of the persistent 2D kernels: tile-edge values tagged with
// their step in aligned 64-bit words.
#pragma once

#include "internal.h"

namespace pat {

using u64 = unsigned long long;

// Exchange words.  The buffer is filled with 0xff bytes before every launch,
// so no stale word can carry a valid tag.
//   forward: [step (32 bits)][P (32 bits)]
//   adjoint: [W_lo with its low 8 mantissa bits replaced by step mod 128][W_hi]
//            (W_lo is a correction ~2^-24 of W_hi; dropping 8 of its bits is
//            far below FP32 rounding of W)
template <bool ADJ>
__device__ __forceinline__ u64 pack(float hi, float lo, unsigned step) {
  if (!ADJ) return ((u64)step << 32) | (u64)__float_as_uint(hi);
  const unsigned l = (__float_as_uint(lo) & ~0xffu) | (step & 0x7fu);
  return ((u64)l << 32) | (u64)__float_as_uint(hi);
}
template <bool ADJ>
__device__ __forceinline__ bool tag_ok(u64 w, unsigned step) {
  const unsigned h = (unsigned)(w >> 32);
  return ADJ ? (h & 0xffu) == (step & 0x7fu) : h == step;
}
__device__ __forceinline__ float word_hi(u64 w) { return __uint_as_float((unsigned)(w & 0xffffffffull)); }
__device__ __forceinline__ float word_lo(u64 w) { return __uint_as_float((unsigned)(w >> 32) & ~0xffu); }

// Exchange words are written with relaxed GPU-scope stores straight from the
// owning threads (aligned 64-bit elements: single-copy atomic) and read with
// relaxed GPU-scope loads.
__device__ __forceinline__ void st_word2(u64* p, u64 a, u64 b) {
  asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(p), "l"(a), "l"(b) : "memory");
}
__device__ __forceinline__ void st_word(u64* p, u64 a) {
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(a) : "memory");
}
__device__ __forceinline__ u64 ld_word(const u64* p) {
  u64 a;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(a) : "l"(p) : "memory");
  return a;
}
__device__ __forceinline__ void ld_word2(const u64* p, u64& a, u64& b) {
  asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "l"(p) : "memory");
}

}  // namespace pat
