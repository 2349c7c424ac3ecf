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

#include "fw_internal.h"

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

template <class T>
__device__ __forceinline__ T warp_sum(T x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  return x;
}

// One row of T^T, NV units of V floats per thread, units `t`, `t` + T, ... of the row for thread t of the T that share it.
// D: accumulator of the dot products (double where the recursion on Phi_y accumulates in more than fp32).
template <int NV, int V, class D, bool BLOCK>
__device__ __forceinline__ void row_steps(float* __restrict__ row, const LayerDev* L, int i, int K, D* red) {
  constexpr int T = BLOCK ? AT : 32;
  const int M = L->M, MU = M / V;
  const int t = BLOCK ? (int)threadIdx.x : (int)(threadIdx.x & 31);
  float r[NV][V];
#pragma unroll
  for (int n = 0; n < NV; ++n) {
    const int c = t + n * T;
    if (c < MU) {
      if (V == 4) *reinterpret_cast<float4*>(r[n]) = reinterpret_cast<const float4*>(row)[c];
      else r[n][0] = row[c];
    }
  }
  for (int k = 0; k < K; ++k) {
    const float a = L->ah[k];
    if (a == 0.f) continue;                        // no step taken (uniform)
    const float* v = L->vh + (size_t)k * M;
    float x[NV][V];
    D acc = 0;
#pragma unroll
    for (int n = 0; n < NV; ++n) {
      const int c = t + n * T;
#pragma unroll
      for (int e = 0; e < V; ++e) x[n][e] = 0.f;
      if (c < MU) {
        if (V == 4) *reinterpret_cast<float4*>(x[n]) = __ldg(reinterpret_cast<const float4*>(v) + c);
        else x[n][0] = __ldg(v + c);
#pragma unroll
        for (int e = 0; e < V; ++e) acc = fma((D)r[n][e], (D)x[n][e], acc);
      }
    }
    acc = warp_sum(acc);
    if (BLOCK) {
      if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
      __syncthreads();
      acc = 0;
#pragma unroll
      for (int w = 0; w < AWARPS; ++w) acc += red[w];
      __syncthreads();
    }
    const float ti = (float)acc, ati = a * ti;
    if (t == 0) L->th[(size_t)k * M + i] = ti;
#pragma unroll
    for (int n = 0; n < NV; ++n)
#pragma unroll
      for (int e = 0; e < V; ++e) r[n][e] = fmaf(ati, x[n][e], r[n][e]);
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
  __shared__ double red[AWARPS];
  const int li = apply_layer(a, (int)blockIdx.x);
  const LayerDev* L = a.g.layer[li];
  const int M = L->M, K = a.K;
  const int blk = (int)blockIdx.x - a.block0[li];
  if (M > kWarpRowMax) {
    float* row = L->Tt + (size_t)blk * M;
    if ((M & 3) == 0) {
      if (M <= 4 * 3 * AT) row_steps<3, 4, double, true>(row, L, blk, K, red);
      else row_steps<8, 4, double, true>(row, L, blk, K, red);
    } else {
      row_steps<32, 1, double, true>(row, L, blk, K, red);
    }
    return;
  }
  const int i = blk * AWARPS + (threadIdx.x >> 5);
  if (i >= M) return;
  float* row = L->Tt + (size_t)i * M;
  if ((M & 3) == 0) {
    if (M <= 256) row_steps<2, 4, float, false>(row, L, i, K, nullptr);
    else if (M <= 640) row_steps<5, 4, float, false>(row, L, i, K, nullptr);
    else row_steps<10, 4, double, false>(row, L, i, K, nullptr);
  } else {
    if (M <= 160) row_steps<5, 1, float, false>(row, L, i, K, nullptr);
    else if (M <= 640) row_steps<20, 1, float, false>(row, L, i, K, nullptr);
    else row_steps<40, 1, double, false>(row, L, i, K, nullptr);
  }
}

// A CTA takes QR rows by 4 AT (V = 4) or AT (V = 1) columns of a layer's Q: the vectors' entries of a thread's columns
// stay in registers across the rows.
constexpr int QR = 8;
__host__ __device__ inline int q_blocks_x(int M) { return (M & 3) == 0 ? (M / 4 + AT - 1) / AT : (M + AT - 1) / AT; }

template <int V>
__device__ __forceinline__ void q_tile(const LayerDev* L, int row0, int c, int K, bool smooth) {
  const int M = L->M;
  const bool in = c * V < M;
  for (int k0 = 0; k0 < K; k0 += 8) {
    float tj[8][V], aq[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const float a = k0 + k < K ? L->ah[k0 + k] : 0.f;
      aq[k] = a * (a + 2.f);
#pragma unroll
      for (int e = 0; e < V; ++e) tj[k][e] = 0.f;
      if (a != 0.f && in) {
        const float* t = L->th + (size_t)(k0 + k) * M;
        if (V == 4) *reinterpret_cast<float4*>(tj[k]) = __ldg(reinterpret_cast<const float4*>(t) + c);
        else tj[k][0] = __ldg(t + c);
      }
    }
    if (!in) continue;
    const bool last = k0 + 8 >= K;
#pragma unroll 2
    for (int r = 0; r < QR; ++r) {
      const int i = row0 + r;
      if (i >= M) break;
      float* qp = L->Q + (size_t)i * M + (size_t)c * V;
      float q[V];
      if (V == 4) *reinterpret_cast<float4*>(q) = *reinterpret_cast<const float4*>(qp); else q[0] = *qp;
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        if (aq[k] != 0.f) {
          const float ti = __ldg(L->th + (size_t)(k0 + k) * M + i);
#pragma unroll
          for (int e = 0; e < V; ++e) q[e] = __fadd_rn(q[e], __fmul_rn(aq[k], __fmul_rn(ti, tj[k][e])));
        }
      }
      if (V == 4) *reinterpret_cast<float4*>(qp) = *reinterpret_cast<const float4*>(q); else *qp = q[0];
      if (last && smooth && L->Qs != L->Q) {
        const float beta = L->beta;
        float* sp = L->Qs + (size_t)i * M + (size_t)c * V;
        float s[V];
        if (V == 4) *reinterpret_cast<float4*>(s) = *reinterpret_cast<const float4*>(sp); else s[0] = *sp;
#pragma unroll
        for (int e = 0; e < V; ++e) s[e] = fmaf(beta, s[e], (1.f - beta) * q[e]);
        if (V == 4) *reinterpret_cast<float4*>(sp) = *reinterpret_cast<const float4*>(s); else *sp = s[0];
      }
    }
  }
}

__global__ void __launch_bounds__(AT) apply_q_kernel(const __grid_constant__ ApplyArgs a) {
  dep_sync();
  const int li = apply_layer(a, (int)blockIdx.x);
  const LayerDev* L = a.g.layer[li];
  const int M = L->M;
  const int blk = (int)blockIdx.x - a.block0[li];
  if ((M & 3) == 0 && M <= 2 * AT) {
    // short rows: several rows side by side
    const int M4 = M >> 2, side = AT / M4;                 // side >= 2
    const int g = (int)threadIdx.x / M4, c = (int)threadIdx.x - g * M4;
    if (g < side) q_tile<4>(L, (blk * side + g) * QR, c, a.K, a.smooth != 0);
    return;
  }
  const int bx = q_blocks_x(M);
  const int by = blk / bx;
  const int c = (blk - by * bx) * AT + (int)threadIdx.x;
  if ((M & 3) == 0) q_tile<4>(L, by * QR, c, a.K, a.smooth != 0);
  else q_tile<1>(L, by * QR, c, a.K, a.smooth != 0);
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
    if ((M & 3) == 0 && M <= 2 * AT) {
      const int rows = (AT / (M >> 2)) * QR;
      n += (M + rows - 1) / rows;
    } else {
      n += q_blocks_x(M) * ((M + QR - 1) / QR);
    }
  }
  a.block0[g.n] = n;
  { ProfScope ps(FW_PROF_RECUR_UPD, s); launch_dep(apply_q_kernel, n, AT, 0, s, a); }
  return cudaGetLastError();
}

}  // namespace fw
