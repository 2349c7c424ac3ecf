// Small device helpers that several kernels share: packed fp32 pairs, warp sums, the rank update of Phi_y.
#ifndef FW_LANES_CUH_
#define FW_LANES_CUH_

namespace fw {

// ---- two fp32 numbers in a 64-bit register ----
typedef unsigned long long u64;
__device__ __forceinline__ u64 pack2(float x, float y) {
  u64 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
  return r;
}
__device__ __forceinline__ void unpack2(u64 r, float& x, float& y) { asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(r)); }
__device__ __forceinline__ u64 add2(u64 a, u64 b) { u64 r; asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b)); return r; }
__device__ __forceinline__ u64 fmadd2(u64 a, u64 b, u64 c) {
  u64 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
// (not for a product that is added to: see mul2)
__device__ __forceinline__ u64 times2(u64 a, u64 b) { u64 r; asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b)); return r; }
// A product rounded by itself: the compiler fuses a packed multiplication with the addition that follows it, .rn or not, so
// the product is an fma with z = (-0, -0), which the compiler must not know (callers read it from shared memory).
__device__ __forceinline__ u64 mul2(u64 a, u64 b, u64 z) {
  u64 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(z));
  return r;
}

// p + (a (vi u_j + ui v_j) + l vi v_j) of two or four entries j (l = a^2 lambda_e; va, vb, ua, ub: v_j and u_j of the first and
// the last two), a rounding per operation and symmetric in (i, j), on packed pairs: half the issue slots.
__device__ __forceinline__ u64 rank2(u64 p, u64 vi, u64 ui, u64 vj, u64 uj, u64 a, u64 l, u64 z) {
  return add2(p, add2(mul2(a, add2(mul2(vi, uj, z), mul2(ui, vj, z)), z), mul2(l, mul2(vi, vj, z), z)));
}
__device__ __forceinline__ float4 rank2(float4 p, u64 vi, u64 ui, u64 va, u64 vb, u64 ua, u64 ub, u64 a, u64 l, u64 z) {
  const u64 x = rank2(pack2(p.x, p.y), vi, ui, va, ua, a, l, z), y = rank2(pack2(p.z, p.w), vi, ui, vb, ub, a, l, z);
  unpack2(x, p.x, p.y);
  unpack2(y, p.z, p.w);
  return p;
}

struct Quad { u64 lo, hi; };       // four neighbouring entries of a row, as packed pairs

// Sums of four values over the warp in 6 shuffles instead of 20: halves of the warp keep two of the values, quarters
// one, and the four totals are handed to every lane.
__device__ __forceinline__ float4 warp_sum4(float y0, float y1, float y2, float y3) {
  const int lane = threadIdx.x & 31;
  const bool hi = (lane & 16) != 0, mid = (lane & 8) != 0;
  float u0 = hi ? y2 : y0, u1 = hi ? y3 : y1;
  u0 += __shfl_xor_sync(0xffffffffu, hi ? y0 : y2, 16);
  u1 += __shfl_xor_sync(0xffffffffu, hi ? y1 : y3, 16);
  float z = mid ? u1 : u0;
  z += __shfl_xor_sync(0xffffffffu, mid ? u0 : u1, 8);
  z += __shfl_xor_sync(0xffffffffu, z, 4);
  z += __shfl_xor_sync(0xffffffffu, z, 2);
  z += __shfl_xor_sync(0xffffffffu, z, 1);
  return make_float4(__shfl_sync(0xffffffffu, z, 0), __shfl_sync(0xffffffffu, z, 8), __shfl_sync(0xffffffffu, z, 16),
                     __shfl_sync(0xffffffffu, z, 24));
}

// sum over the warp, the same bits in every lane
template <class T>
__device__ __forceinline__ T warp_sum(T x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  return x;
}

// a 2^-896 as fp64: the bits moved into place.  Exact for every finite a, zero and subnormal numbers included.
__device__ __forceinline__ double widen(float a) {
  const int b = __float_as_int(a);
  return __hiloint2double((b >> 3) & 0x8fffffff, b << 29);
}
constexpr double kWiden = 0x1p896;

// What two orders of an fp64 sum of products of fp32 numbers are taken to differ by at most, over ||row|| ||x||: 16 x 2^-53.
// Found for M = 640 ... 8192 (20000 rows each, the orders the kernels use): up to 4.3 x 2^-53 for random, sign-definite,
// decaying, sparse and eigenvector-like rows, up to M / 128 x 2^-53 for rows of repeated entries.  The worst case, about
// M / 16 x 2^-53, would send most passes of a layer of M = 4608 through a second sum (1.2 -> 1.7 ms for four steps); past
// the window the two orders' roundings differ with a probability near 1e-7 a row.
constexpr float kOrderWindow = 0x1p-49f;

// 1/sqrt(n2) refined by one Newton step, 0 when n2 is not a positive finite number
__device__ __forceinline__ float inv_norm(float n2) {
  float inv = (n2 > 0.f && isfinite(n2)) ? rsqrtf(n2) : 0.f;
  return inv > 0.f ? inv * (1.5f - 0.5f * n2 * inv * inv) : 0.f;
}

}  // namespace fw
#endif
