// The rank-one terms of a reduction call in T and Q (Eqs. 42, 44), applied after
// the recursion.  A step's term needs t = T^T v_e with the T of that step, but
// the recursion needs neither t nor T nor Q: it works on Phi_y alone.  So the
// recursion kernels only record (v_e, a_e) of their steps and these two kernels
// take all of a call's steps at once: T and Q each cross memory once per call
// (up to kHist steps) instead of once per step, and the recursion keeps its
// shared memory for Phi_y.
//
//   apply_t   a warp holds a row of T^T; for each step in order
//             t[i] = T^T[i, :] . v,  T^T[i, :] += a t[i] v^T.  Rows are independent.
//             Every element sees the operations of a step-by-step update in the same order.
//   apply_q   Q[i][j] += a (a + 2) t[i] t[j], step after step, then (last steps of a call)
//             the smoothing of Eq. 35.
//
// apply_q is bound by reading and writing its matrix (L2 or HBM), apply_t by its fp64 sums.
#include <algorithm>
#include <cstring>

#include "fw_internal.h"
#include "fw_lanes.cuh"
#include "fw_sm100.cuh"

namespace fw {
namespace {

constexpr int AT = 256;             // threads per CTA
constexpr int AWARPS = AT / 32;
constexpr int kWarpRowMax = 1280;   // longest row a single warp holds (40 floats per lane); above, the CTA shares a row

struct ApplyArgs {
  GroupDev g;
  int32_t block0[FW_MAX_GROUP + 1];   // first CTA of each layer in the flat grid
  int32_t K, smooth;
  int32_t exchanges;
};

__device__ __forceinline__ int apply_layer(const ApplyArgs& a, int block) {
  int li = 0;
#pragma unroll 1
  for (int i = 1; i < a.g.n; ++i)
    if (block >= a.block0[i]) li = i;
  return li;
}

// t[i] is an fp64 sum as the products of the recursion are: a lane takes every 32nd float4 of the row (rows that are not whole
// float4s: every 32nd entry) in ascending order, then a butterfly over the lanes.  An SM converts 16 numbers per clock to fp64
// and both factors need it, so the row's are widened by integer operations instead, which holds for
// finite numbers: `plain` is for rows that are or may become anything else.  64 layers of M = 1152, eight steps: 430 us, of which the
// conversions alone are 150; sums in fp32 pairs took 350, but some rounded otherwise.
template <bool PLAIN>
__device__ __forceinline__ double dot4(float4 r, float4 x, double acc) {
  if (PLAIN) {
    acc = fma((double)r.x, (double)x.x, acc); acc = fma((double)r.y, (double)x.y, acc);
    acc = fma((double)r.z, (double)x.z, acc); acc = fma((double)r.w, (double)x.w, acc);
  } else {
    acc = fma(widen(r.x), (double)x.x * kWiden, acc); acc = fma(widen(r.y), (double)x.y * kWiden, acc);
    acc = fma(widen(r.z), (double)x.z * kWiden, acc); acc = fma(widen(r.w), (double)x.w * kWiden, acc);
  }
  return acc;
}
__device__ __forceinline__ float4 axpy4(float a, float4 x, float4 r) {
  return make_float4(fmaf(a, x.x, r.x), fmaf(a, x.y, r.y), fmaf(a, x.z, r.z), fmaf(a, x.w, r.w));
}
// on the TF32 grid (the operand of the re-sync products that a layer with round_t keeps)
__device__ __forceinline__ float4 rounded4(float4 r) {
  return make_float4(sm100::tf32_rna(r.x), sm100::tf32_rna(r.y), sm100::tf32_rna(r.z), sm100::tf32_rna(r.w));
}
__device__ __forceinline__ float abs4(float4 r) { return fabsf(r.x) + fabsf(r.y) + fabsf(r.z) + fabsf(r.w); }
constexpr float kFinite = 1e37f;    // numbers whose absolute values sum to less are finite

// One row of T^T of at most 32 V NV entries in the registers of a warp, in units of V = 4 or 1 floats.
template <int NV, int V>
__device__ __forceinline__ void row_steps(float* __restrict__ row, const LayerDev* L, int i, int K) {
  const int M = L->M, MU = M / V, t = threadIdx.x & 31;
  float4 r4[V == 4 ? NV : 1];
  float r1[V == 4 ? 1 : NV];
  float top = 0.f;
#pragma unroll
  for (int n = 0; n < NV; ++n) {
    const int c = t + 32 * n;
    if (V == 4) {
      r4[n] = c < MU ? reinterpret_cast<const float4*>(row)[c] : make_float4(0.f, 0.f, 0.f, 0.f);
      top += abs4(r4[n]);
    } else {
      r1[n] = c < MU ? row[c] : 0.f;
    }
  }
  bool plain = V == 1 || __any_sync(0xffffffffu, !(top < kFinite));
  for (int k = 0; k < K; ++k) {
    const float a = L->ah[k];
    if (a == 0.f) continue;                        // no step taken (uniform)
    const float* v = L->vh + (size_t)k * M;
    // all of v before any of it is used: a load at a time is a chain of latencies
    float4 x4[V == 4 ? NV : 1];
    float x1[V == 4 ? 1 : NV];
#pragma unroll
    for (int n = 0; n < NV; ++n) {
      const int c = t + 32 * n;
      if (V == 4) x4[n] = c < MU ? __ldg(reinterpret_cast<const float4*>(v) + c) : make_float4(0.f, 0.f, 0.f, 0.f);
      else x1[n] = c < MU ? __ldg(v + c) : 0.f;
    }
    double acc = 0.0;
    if (V == 1) {
#pragma unroll
      for (int n = 0; n < NV; ++n) acc = fma((double)r1[n], (double)x1[n], acc);
    } else if (plain) {
#pragma unroll
      for (int n = 0; n < NV; ++n) acc = dot4<true>(r4[n], x4[n], acc);
    } else {
#pragma unroll
      for (int n = 0; n < NV; ++n) acc = dot4<false>(r4[n], x4[n], acc);
    }
    const float ti = (float)warp_sum(acc), ati = a * ti;
    plain = plain || !(fabsf(ati) < kFinite / kHist);
    if (t == 0) L->th[(size_t)k * M + i] = ti;
#pragma unroll
    for (int n = 0; n < NV; ++n) {
      if (V == 4) r4[n] = axpy4(ati, x4[n], r4[n]);
      else r1[n] = fmaf(ati, x1[n], r1[n]);
    }
  }
#pragma unroll
  for (int n = 0; n < NV; ++n) {
    const int c = t + 32 * n;
    if (c >= MU) continue;
    if (V == 4) {
      reinterpret_cast<float4*>(row)[c] = r4[n];
      if (L->round_t) reinterpret_cast<float4*>(L->tmp + (size_t)i * M)[c] = rounded4(r4[n]);
    } else {
      row[c] = r1[n];
    }
  }
}
// A longer row in the registers of a CTA, at most AT V NV entries.  The sum runs over all threads, in another order; where
// numbers as close to it as the two orders may be round to different fp32 numbers, the first warp forms the sum of record
// from a copy of the row in shared memory (`copy`).  rn bounds ||row|| (||v|| = 1, so a step adds at most |a t|); a row that
// is not finite always takes that way.
template <int NV, int V>
__device__ __forceinline__ void long_row_steps(float* __restrict__ row, float* copy, double* red, const LayerDev* L, int i, int K) {
  const int M = L->M, MU = M / V, t = threadIdx.x;
  float r[NV][V];
#pragma unroll
  for (int n = 0; n < NV; ++n) {
    const int c = t + AT * n;
#pragma unroll
    for (int e = 0; e < V; ++e) r[n][e] = 0.f;
    if (c < MU) {
      if (V == 4) *reinterpret_cast<float4*>(r[n]) = reinterpret_cast<const float4*>(row)[c];
      else r[n][0] = row[c];
    }
  }
  auto total = [&](double y) {
    y = warp_sum(y);
    if ((t & 31) == 0) red[t >> 5] = y;
    __syncthreads();
    y = red[0];
#pragma unroll
    for (int w = 1; w < AWARPS; ++w) y += red[w];
    __syncthreads();
    return y;
  };
  float q = 0.f;
#pragma unroll
  for (int n = 0; n < NV; ++n)
#pragma unroll
    for (int e = 0; e < V; ++e) q = fmaf(r[n][e], r[n][e], q);
  float rn = 1.01f * sqrtf((float)total((double)q));
  for (int k = 0; k < K; ++k) {
    const float a = L->ah[k];
    if (a == 0.f) continue;
    const float* v = L->vh + (size_t)k * M;
    float x[NV][V];
#pragma unroll
    for (int n = 0; n < NV; ++n) {
      const int c = t + AT * n;
#pragma unroll
      for (int e = 0; e < V; ++e) x[n][e] = 0.f;
      if (c < MU) {
        if (V == 4) *reinterpret_cast<float4*>(x[n]) = __ldg(reinterpret_cast<const float4*>(v) + c);
        else x[n][0] = __ldg(v + c);
      }
    }
    double acc = 0.0;
#pragma unroll
    for (int n = 0; n < NV; ++n)
#pragma unroll
      for (int e = 0; e < V; ++e) acc = fma(widen(r[n][e]), (double)x[n][e] * kWiden, acc);
    double y = total(acc);
    const double w = (double)(rn * kOrderWindow);
    if ((float)(y - w) != (float)(y + w)) {          // uniform in the CTA
#pragma unroll
      for (int n = 0; n < NV; ++n)
#pragma unroll
        for (int e = 0; e < V; ++e)
          if (t + AT * n < MU) copy[V * (t + AT * n) + e] = r[n][e];
      __syncthreads();
      if (t < 32) {
        double z = 0.0;
        for (int c = t; c < MU; c += 32)
#pragma unroll
          for (int e = 0; e < V; ++e) z = fma((double)copy[V * c + e], (double)__ldg(v + V * c + e), z);
        z = warp_sum(z);
        if (t == 0) red[0] = z;
      }
      __syncthreads();
      y = red[0];
      __syncthreads();
    }
    const float ti = (float)y, ati = a * ti;
    rn += 1.01f * fabsf(ati);
    if (t == 0) L->th[(size_t)k * M + i] = ti;
#pragma unroll
    for (int n = 0; n < NV; ++n)
#pragma unroll
      for (int e = 0; e < V; ++e) r[n][e] = fmaf(ati, x[n][e], r[n][e]);
  }
#pragma unroll
  for (int n = 0; n < NV; ++n) {
    const int c = t + AT * n;
    if (c < MU) {
      if (V == 4) {
        const float4 q = *reinterpret_cast<const float4*>(r[n]);
        reinterpret_cast<float4*>(row)[c] = q;
        if (L->round_t) reinterpret_cast<float4*>(L->tmp + (size_t)i * M)[c] = rounded4(q);
      } else {
        row[c] = r[n][0];
      }
    }
  }
}

__global__ void __launch_bounds__(AT, 2) apply_t_kernel(const __grid_constant__ ApplyArgs a) {
  dep_sync();
  const int li = apply_layer(a, (int)blockIdx.x);
  const LayerDev* L = a.g.layer[li];
  const int M = L->M;
  const int i = ((int)blockIdx.x - a.block0[li]) * AWARPS + (threadIdx.x >> 5);
  if (i >= M) return;
  float* row = L->Tt + (size_t)i * M;
  if ((M & 3) == 0) row_steps<kWarpRowMax / 128, 4>(row, L, i, a.K);
  else row_steps<kWarpRowMax / 32, 1>(row, L, i, a.K);
}

template <int NV, int V>
__global__ void __launch_bounds__(AT, NV == 3 ? 4 : 2) apply_t_long_kernel(const __grid_constant__ ApplyArgs a) {
  dep_sync();
  extern __shared__ __align__(16) float copy[];
  __shared__ double red[AWARPS];
  const int li = apply_layer(a, (int)blockIdx.x);
  const LayerDev* L = a.g.layer[li];
  const int M = L->M, i = (int)blockIdx.x - a.block0[li];
  long_row_steps<NV, V>(L->Tt + (size_t)i * M, copy, red, L, i, a.K);
}
// which kernel takes a layer's T: 0 a warp per row; a CTA per row of whole float4s, up to three or eight per thread, or of
// single entries.  A kernel each: together they would all have the registers of the largest (16 warps per SM).
inline int t_kind(int M) { return M <= kWarpRowMax ? 0 : (M & 3) != 0 ? 3 : M <= 4 * 3 * AT ? 1 : 2; }

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
  if (idx == 0) L->iscal[IS_EXCHANGE] = (int32_t)((uint32_t)L->iscal[IS_EXCHANGE] + (uint32_t)a.exchanges);   // the team launch has ended
  if (row0 >= M) return;
  if ((M & 3) == 0) q_tile<4>(L, row0, c, a.K, a.smooth != 0);
  else q_tile<1>(L, row0, c, a.K, a.smooth != 0);
}

}  // namespace

cudaError_t launch_recursion_apply(const GroupDev& g, const int* layer_M, int K, bool smooth, int exchanges, cudaStream_t s) {
  if (K < 1 || K > kHist) return cudaErrorInvalidValue;
  ApplyArgs a;
  memset(&a, 0, sizeof(a));
  a.g = g; a.K = K; a.smooth = smooth ? 1 : 0; a.exchanges = exchanges;
  void (*const kernels[])(const ApplyArgs) = {apply_t_kernel, apply_t_long_kernel<3, 4>, apply_t_long_kernel<8, 4>,
                                              apply_t_long_kernel<32, 1>};
  int n = 0;
  for (int kind = 0; kind < 4; ++kind) {
    int longest = 0;
    n = 0;
    for (int i = 0; i < g.n; ++i) {
      const int M = layer_M[i];
      a.block0[i] = n;
      if (t_kind(M) != kind) continue;
      n += kind ? M : (M + AWARPS - 1) / AWARPS;
      longest = std::max(longest, M);
    }
    a.block0[g.n] = n;
    if (n == 0) continue;
    ProfScope ps(FW_PROF_RECUR_UPD, s);
    const cudaError_t e = launch_dep(kernels[kind], n, AT, kind ? sizeof(float) * longest : 0, s, a);      // at most 32 KB
    if (e != cudaSuccess) return e;
  }
  n = 0;
  for (int i = 0; i < g.n; ++i) {
    const int M = layer_M[i];
    a.block0[i] = n;
    n += (int)(((int64_t)q_units(M) * ((M + QR - 1) / QR) + AT - 1) / AT);
  }
  a.block0[g.n] = n;
  ProfScope ps(FW_PROF_RECUR_UPD, s);
  return launch_dep(apply_q_kernel, n, AT, 0, s, a);
}

}  // namespace fw
