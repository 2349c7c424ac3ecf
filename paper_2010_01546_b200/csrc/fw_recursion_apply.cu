// The rank-one terms of a reduction call in T and Q (Eqs. 42, 44), applied after
// the recursion.  A step's term needs t = T^T v_e with the T of that step, but
// the recursion needs neither t nor T nor Q: it works on Phi_y alone.  So the
// recursion kernels only record (v_e, a_e) of their steps and these two kernels
// take all of a call's steps at once: T and Q each cross memory once per call
// (up to kHist steps) instead of once per step, and the recursion keeps its
// shared memory for Phi_y.
//
//   apply_t   a row of T^T is held in registers; for each step in order
//             t[i] = T^T[i, :] . v,  T^T[i, :] += a t[i] v^T.  Rows are independent.
//             Every element sees the operations of a step-by-step update in the same order.
//   apply_q   Q[i][j] += a (a + 2) t[i] t[j], step after step, then (last steps of a call)
//             the smoothing of Eq. 35.
//
// Both are bound by reading and writing their matrix once (L2 or HBM).
#include <cstring>

#include "fw_fixsum.cuh"
#include "fw_internal.h"
#include "fw_lanes.cuh"

namespace fw {
namespace {

constexpr int AT = 256;             // threads per CTA
constexpr int AWARPS = AT / 32;
constexpr int kWarpRowMax = 1280;   // longest row a single warp holds (40 floats per lane); above, the CTA shares a row

struct ApplyArgs {
  GroupDev g;
  int32_t block0[FW_MAX_GROUP + 1];   // first CTA of each layer in the flat grid
  int32_t K, smooth;
};

__device__ __forceinline__ int apply_layer(const ApplyArgs& a, int block) {
  int li = 0;
#pragma unroll 1
  for (int i = 1; i < a.g.n; ++i)
    if (block >= a.block0[i]) li = i;
  return li;
}

// One row of T^T, NV units of V floats per thread, units `t`, `t` + T, ... of the row for thread t of the T that share it.
// Bound by issue: the conversions of an fp64 sum (16 per clock and SM) made 64 layers of M = 1152 and eight steps 470 us,
// now 355.  FIX: the dot product as an anchored sum of two fp32 numbers (where the recursion on Phi_y accumulates in more than fp32);
// ||v|| = 1, so ||row|| bounds it, and a step adds at most |a t| to that norm.
template <int NV, int V, bool FIX, bool BLOCK>
__device__ __forceinline__ void row_steps(float* __restrict__ row, const LayerDev* L, int i, int K, float2* red) {
  constexpr int T = BLOCK ? AT : 32, H = NV * V / 2;
  const int M = L->M, MU = M / V;
  const int t = BLOCK ? (int)threadIdx.x : (int)(threadIdx.x & 31);
  static_assert((NV * V) % 2 == 0 || !FIX, "pairs");
  float r[NV][V];
  float* rf = &r[0][0];
#pragma unroll
  for (int n = 0; n < NV; ++n) {
    const int c = t + n * T;
#pragma unroll
    for (int e = 0; e < V; ++e) r[n][e] = 0.f;
    if (c < MU) {
      if (V == 4) *reinterpret_cast<float4*>(r[n]) = reinterpret_cast<const float4*>(row)[c];
      else r[n][0] = row[c];
    }
  }
  // sum over the threads of the row
  auto total = [&](float2 y) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) y = add2(y, shfl_xor2(y, o));
    if (BLOCK) {
      if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = y;
      __syncthreads();
      y = red[0];
#pragma unroll
      for (int w = 1; w < AWARPS; ++w) y = add2(y, red[w]);
      __syncthreads();
    }
    return y;
  };
  float rn = 0.f;
  if (FIX) {
    float q = 0.f;
#pragma unroll
    for (int n = 0; n < NV * V; ++n) q = fmaf(rf[n], rf[n], q);
    rn = sqrtf(total(make_float2(q, 0.f)).x);
  }
  for (int k = 0; k < K; ++k) {
    const float a = L->ah[k];
    if (a == 0.f) continue;                        // no step taken (uniform)
    const float* v = L->vh + (size_t)k * M;
    float x[NV][V];
    float* xf = &x[0][0];
#pragma unroll
    for (int n = 0; n < NV; ++n) {
      const int c = t + n * T;
#pragma unroll
      for (int e = 0; e < V; ++e) x[n][e] = 0.f;
      if (c < MU) {
        if (V == 4) *reinterpret_cast<float4*>(x[n]) = __ldg(reinterpret_cast<const float4*>(v) + c);
        else x[n][0] = __ldg(v + c);
      }
    }
    float ti;
    if (FIX) {
      const float C = anchor(1.01f * rn);
      u64 s = pack2(C, C), l = 0;
#pragma unroll
      for (int h = 0; h < H; ++h) fix_add(s, l, pack2(rf[2 * h], rf[2 * h + 1]), pack2(xf[2 * h], xf[2 * h + 1]));
      const float2 y = total(fix_value(s, l, C));
      ti = y.x + y.y;
    } else {
      float acc = 0.f;
#pragma unroll
      for (int n = 0; n < NV * V; ++n) acc = fmaf(rf[n], xf[n], acc);
      ti = warp_sum(acc);
    }
    const float ati = a * ti;
    if (FIX) rn += fabsf(ati);
    if (t == 0) L->th[(size_t)k * M + i] = ti;
#pragma unroll
    for (int n = 0; n < NV * V; ++n) rf[n] = fmaf(ati, xf[n], rf[n]);
  }
#pragma unroll
  for (int n = 0; n < NV; ++n) {
    const int c = t + n * T;
    if (c < MU) {
      if (V == 4) reinterpret_cast<float4*>(row)[c] = *reinterpret_cast<const float4*>(r[n]);
      else row[c] = r[n][0];
    }
  }
}

// rows of M <= 1280 take a warp each; longer rows a CTA each
__global__ void __launch_bounds__(AT) apply_t_kernel(const __grid_constant__ ApplyArgs a) {
  dep_sync();
  __shared__ float2 red[AWARPS];
  const int li = apply_layer(a, (int)blockIdx.x);
  const LayerDev* L = a.g.layer[li];
  const int M = L->M, K = a.K;
  const int blk = (int)blockIdx.x - a.block0[li];
  if (M > kWarpRowMax) {
    float* row = L->Tt + (size_t)blk * M;
    if ((M & 3) == 0) {
      if (M <= 4 * 3 * AT) row_steps<3, 4, true, true>(row, L, blk, K, red);
      else row_steps<8, 4, true, true>(row, L, blk, K, red);
    } else {
      row_steps<32, 1, true, true>(row, L, blk, K, red);
    }
    return;
  }
  const int i = blk * AWARPS + (threadIdx.x >> 5);
  if (i >= M) return;
  float* row = L->Tt + (size_t)i * M;
  if ((M & 3) == 0) {
    if (M <= 256) row_steps<2, 4, false, false>(row, L, i, K, nullptr);
    else if (M <= 640) row_steps<5, 4, false, false>(row, L, i, K, nullptr);
    else row_steps<10, 4, true, false>(row, L, i, K, nullptr);
  } else {
    if (M <= 160) row_steps<5, 1, false, false>(row, L, i, K, nullptr);
    else if (M <= 640) row_steps<20, 1, false, false>(row, L, i, K, nullptr);
    else row_steps<40, 1, true, false>(row, L, i, K, nullptr);
  }
}

// A thread takes QR rows of V columns (V = 4, or 1 for rows of odd length) of a layer's Q, whose
// loads are all in flight together, and takes them through the steps.  Threads are numbered along the
// columns, then along the groups of rows, so a CTA is full whatever M is (64 layers of M = 1152, eight steps: 480 us with
// a CTA per 1024 columns and two rows in flight, 240 us so, 104 at HBM rate).
constexpr int QR = 8;
__host__ __device__ inline int q_units(int M) { return (M & 3) == 0 ? M / 4 : M; }

template <int V>
__device__ __forceinline__ void q_tile(const LayerDev* L, int row0, int c, int K, bool smooth) {
  const int M = L->M;
  float q[QR][V];
#pragma unroll
  for (int r = 0; r < QR; ++r) {
    if (row0 + r >= M) continue;
    const float* qp = L->Q + (size_t)(row0 + r) * M + (size_t)c * V;
    if (V == 4) *reinterpret_cast<float4*>(q[r]) = *reinterpret_cast<const float4*>(qp); else q[r][0] = *qp;
  }
#pragma unroll 2
  for (int k = 0; k < K; ++k) {
    const float a = L->ah[k], aq = a * (a + 2.f);
    if (aq == 0.f) continue;
    const float* t = L->th + (size_t)k * M;
    float tj[V], ti[QR];
    if (V == 4) {
      *reinterpret_cast<float4*>(tj) = __ldg(reinterpret_cast<const float4*>(t) + c);
#pragma unroll
      for (int h = 0; h < QR / 4; ++h)            // row0 and M are multiples of four
        if (row0 + 4 * h < M) *reinterpret_cast<float4*>(ti + 4 * h) = __ldg(reinterpret_cast<const float4*>(t + row0) + h);
    } else {
      tj[0] = __ldg(t + c);
#pragma unroll
      for (int r = 0; r < QR; ++r) ti[r] = __ldg(t + min(row0 + r, M - 1));
    }
#pragma unroll
    for (int r = 0; r < QR; ++r)
#pragma unroll
      for (int e = 0; e < V; ++e) q[r][e] = __fadd_rn(q[r][e], __fmul_rn(aq, __fmul_rn(ti[r], tj[e])));
  }
  const float beta = L->beta;
  smooth = smooth && L->Qs != L->Q;
#pragma unroll
  for (int r = 0; r < QR; ++r) {
    if (row0 + r >= M) continue;
    const size_t at = (size_t)(row0 + r) * M + (size_t)c * V;
    float* qp = L->Q + at;
    if (V == 4) *reinterpret_cast<float4*>(qp) = *reinterpret_cast<const float4*>(q[r]); else *qp = q[r][0];
    if (smooth) {
      float* sp = L->Qs + at;
      float s[V];
      if (V == 4) *reinterpret_cast<float4*>(s) = *reinterpret_cast<const float4*>(sp); else s[0] = *sp;
#pragma unroll
      for (int e = 0; e < V; ++e) s[e] = fmaf(beta, s[e], (1.f - beta) * q[r][e]);
      if (V == 4) *reinterpret_cast<float4*>(sp) = *reinterpret_cast<const float4*>(s); else *sp = s[0];
    }
  }
}

__global__ void __launch_bounds__(AT) apply_q_kernel(const __grid_constant__ ApplyArgs a) {
  dep_sync();
  const int li = apply_layer(a, (int)blockIdx.x);
  const LayerDev* L = a.g.layer[li];
  const int M = L->M;
  const int units = q_units(M);
  const int64_t idx = (int64_t)((int)blockIdx.x - a.block0[li]) * AT + threadIdx.x;
  const int row0 = (int)(idx / units) * QR, c = (int)(idx % units);
  if (row0 >= M) return;
  if ((M & 3) == 0) q_tile<4>(L, row0, c, a.K, a.smooth != 0);
  else q_tile<1>(L, row0, c, a.K, a.smooth != 0);
}

}  // namespace

cudaError_t launch_recursion_apply(const GroupDev& g, const int* layer_M, int K, bool smooth, cudaStream_t s) {
  if (K < 1 || K > kHist) return cudaErrorInvalidValue;
  ApplyArgs a;
  memset(&a, 0, sizeof(a));
  a.g = g; a.K = K; a.smooth = smooth ? 1 : 0;
  int n = 0;
  for (int i = 0; i < g.n; ++i) {
    a.block0[i] = n;
    n += layer_M[i] > kWarpRowMax ? layer_M[i] : (layer_M[i] + AWARPS - 1) / AWARPS;
  }
  a.block0[g.n] = n;
  { ProfScope ps(FW_PROF_RECUR_UPD, s); launch_dep(apply_t_kernel, n, AT, 0, s, a); }
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  n = 0;
  for (int i = 0; i < g.n; ++i) {
    const int M = layer_M[i];
    a.block0[i] = n;
    n += (int)(((int64_t)q_units(M) * ((M + QR - 1) / QR) + AT - 1) / AT);
  }
  a.block0[g.n] = n;
  { ProfScope ps(FW_PROF_RECUR_UPD, s); launch_dep(apply_q_kernel, n, AT, 0, s, a); }
  return cudaGetLastError();
}

}  // namespace fw
