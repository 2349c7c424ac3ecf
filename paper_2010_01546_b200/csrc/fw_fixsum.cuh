// Sums of products in more than fp32 without fp64 (whose conversions, 16 per clock and SM, would bound the kernels):
// two fp32 numbers, the first anchored at a power of two above every partial sum.  See fw_recursion_team.cu.
#ifndef FW_FIXSUM_CUH_
#define FW_FIXSUM_CUH_
#include <stdint.h>

#include "fw_lanes.cuh"

namespace fw {

// The running sum s + l of products whose partial sums are bounded by B, two at a time (packed fp32 pairs).
__device__ __forceinline__ float anchor(float B) {
  // 1.5 * 2^k with 2^k >= 2 B: s stays between 2^k and 2^(k+1)
  // (too large or not finite: infinity, and the result is not finite either)
  const uint32_t ex = (__float_as_uint(B) >> 23) & 0xffu;
  return __uint_as_float(min((max(ex, 26u) + 2u) << 23 | 0x00400000u, 0x7f800000u));
}
__device__ __forceinline__ void fix_add(u64& s, u64& l, u64 a, u64 x) {
  u64 n, d, e;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(n) : "l"(a), "l"(x), "l"(s));
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(s), "l"(n));
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(e) : "l"(a), "l"(x), "l"(d));
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(l) : "l"(l), "l"(e));
  s = n;
}
// The value of a sum as two fp32 numbers: d = s - C, a multiple of ulp(C), and l.  Sums of d over lanes and warps stay
// exact in fp32: every one of them is bounded like the whole product.
__device__ __forceinline__ float2 fix_value(u64 s, u64 l, float C) {
  float s0, s1, l0, l1;
  unpack2(s, s0, s1);
  unpack2(l, l0, l1);
  return make_float2(__fadd_rn(__fsub_rn(s0, C), __fsub_rn(s1, C)), l0 + l1);
}
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return make_float2(__fadd_rn(a.x, b.x), a.y + b.y); }
__device__ __forceinline__ float2 shfl_xor2(float2 a, int o) {
  return make_float2(__shfl_xor_sync(0xffffffffu, a.x, o), __shfl_xor_sync(0xffffffffu, a.y, o));
}

}  // namespace fw
#endif
