// Grouped fp32 (FFMA) GEMM used by the FP32 engine and by layers the tensor-core kernels do not take:
//   - the Gram pass X^T X with fused column sums (Eqs. 3, 5: the covariance sum),
//   - G * Qs with the optional fused SGD epilogue (Eqs. 27, 29),
//   - the re-sync products T Phix and (T Phix) T^T.
// One launch covers every problem of a group; a CTA finds its problem, tile and K-split from its block index.
//
// A group of 128 threads computes a 64 x 64 tile, 8 x 4 accumulators per thread, from 16-deep slabs staged through
// registers (where the Gram pass subtracts its shift) into two shared-memory buffers.  It is bound by the FP32 pipe when
// the tiles fill the machine; when they do not, what counts is the length of the chain of slabs, so 2 or 4 groups of a
// CTA share the tile, each a contiguous part of K, and their sums are added in order at the end: the chain is that much
// shorter and the SM has that many more warps to hide it.  Products of the ResNet-20-shaped set at batch 32 (Gram /
// re-sync / G Qs): 1028 / 310 / 101 us with 4 x 4 accumulators, scalar loads and one group; see launch_gemm_ffma.
#include <cstring>

#include "fw_internal.h"

namespace fw {

namespace {

constexpr int BM = 64, BN = 64, BK = 16, NT = 128;   // tile, slab, threads of a group
constexpr int TM = 8, TN = 4;                        // accumulators per thread: 8 x 16 threads
constexpr int LDA = BM + 4, LDB = BN + 4;            // shared-memory rows
constexpr int kSlab = BK * (LDA + LDB);              // floats of one buffer

// The kernel's argument block carries as many problems as the launch needs: a launch costs 0.7 us per KB of arguments.
template <int CAP>
struct GemmBlock {
  int32_t n;
  GemmProblem p[CAP];
};

__device__ __forceinline__ float ld_elem(const void* base, int64_t idx, int bf16) {
  if (bf16) return __bfloat162float(reinterpret_cast<const __nv_bfloat16*>(base)[idx]);
  return reinterpret_cast<const float*>(base)[idx];
}

// A slab of a matrix stored k x n (row-major, n contiguous): element (k, n) at P[k ld + n]; 64 columns from n0.  Thread t
// of a group holds entries (k, n) as two float4 of one column quad (vec) or eight scalars.
struct SlabRegs { float v[8]; };
__device__ __forceinline__ void load_kmajor(SlabRegs& r, const void* P, int64_t ld, int64_t k0, int64_t ke, int n0, int n, int t,
                                            bool vec, int bf16) {
  if (vec) {
    const int c = n0 + 4 * (t & 15);
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const int64_t k = k0 + (t >> 4) + 8 * e;
      float4 q = make_float4(0.f, 0.f, 0.f, 0.f);
      if (k < ke && c < n) q = *reinterpret_cast<const float4*>(reinterpret_cast<const float*>(P) + k * ld + c);
      *reinterpret_cast<float4*>(r.v + 4 * e) = q;
    }
  } else {
    const int c = n0 + (t & 63);
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const int64_t k = k0 + (t >> 6) + 2 * e;
      r.v[e] = (k < ke && c < n) ? ld_elem(P, k * ld + c, bf16) : 0.f;
    }
  }
}
// shift: subtracted from the elements inside the matrix (zero for the padding)
__device__ __forceinline__ void store_kmajor(float* S, int lds, const SlabRegs& r, const float (&sh)[4], int64_t k0, int64_t ke,
                                             int t, bool vec) {
  if (vec) {
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const int kk = (t >> 4) + 8 * e;
      float4 q = *reinterpret_cast<const float4*>(r.v + 4 * e);
      if (k0 + kk < ke) { q.x -= sh[0]; q.y -= sh[1]; q.z -= sh[2]; q.w -= sh[3]; }
      *reinterpret_cast<float4*>(S + kk * lds + 4 * (t & 15)) = q;
    }
  } else {
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const int kk = (t >> 6) + 2 * e;
      S[kk * lds + (t & 63)] = k0 + kk < ke ? r.v[e] - sh[0] : r.v[e];
    }
  }
}
// A stored m x k (row-major, k contiguous): a thread takes quads of k of row t % 64, stored transposed
__device__ __forceinline__ void load_mmajor(SlabRegs& r, const float* P, int64_t ld, int64_t k0, int64_t ke, int m0, int m, int t,
                                            bool vec) {
  const int row = m0 + (t & 63);
  const float* p = P + (int64_t)row * ld;
#pragma unroll
  for (int e = 0; e < 2; ++e) {
    const int64_t k = k0 + 4 * ((t >> 6) + 2 * e);
    float4 q = make_float4(0.f, 0.f, 0.f, 0.f);
    if (row < m) {
      if (vec && k + 4 <= ke) q = *reinterpret_cast<const float4*>(p + k);
      else {
        if (k < ke) q.x = p[k];
        if (k + 1 < ke) q.y = p[k + 1];
        if (k + 2 < ke) q.z = p[k + 2];
        if (k + 3 < ke) q.w = p[k + 3];
      }
    }
    *reinterpret_cast<float4*>(r.v + 4 * e) = q;
  }
}
__device__ __forceinline__ void store_mmajor(float* S, const SlabRegs& r, int t) {
#pragma unroll
  for (int e = 0; e < 2; ++e)
#pragma unroll
    for (int i = 0; i < 4; ++i) S[(4 * ((t >> 6) + 2 * e) + i) * LDA + (t & 63)] = r.v[4 * e + i];
}

extern __shared__ __align__(16) float gsm[];

template <int KG, int CAP>
__global__ void __launch_bounds__(NT * KG) gemm_ffma_kernel(const __grid_constant__ GemmBlock<CAP> g) {
  // locate the problem this CTA works on
  const int cta = blockIdx.x;
  int pi = 0;
#pragma unroll 1
  for (int i = 1; i < g.n; ++i)
    if (cta >= g.p[i].first_cta) pi = i;
  const GemmProblem& pr = g.p[pi];
  const int local = cta - pr.first_cta;
  const int split = local / pr.ntiles;
  const int tile = local - split * pr.ntiles;
  int tm, tn;
  if (pr.sym) tri_decode(tile, pr.tiles_n, tm, tn);
  else { tm = tile / pr.tiles_n; tn = tile - tm * pr.tiles_n; }
  const int m0 = tm * BM, n0 = tn * BN;
  const int t = threadIdx.x % NT, grp = threadIdx.x / NT;
  // K range of this split, then of this group, in multiples of BK
  const int64_t kslabs = (pr.k + BK - 1) / BK;
  const int64_t per = (kslabs + pr.splits - 1) / pr.splits;
  const int64_t sb = (int64_t)split * per, se = min(sb + per, kslabs);
  const int64_t gper = (max(se - sb, (int64_t)0) + KG - 1) / KG;
  const int64_t kb = (sb + grp * gper) * BK, ke = min(min(sb + (grp + 1) * gper, se) * BK, pr.k);

  float* slab = gsm + grp * 2 * kSlab;
  const int tx = t & 15, ty = t >> 4;
  float acc[TM][TN];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) acc[i][j] = 0.f;
  const bool a_km = pr.a_kmajor != 0;
  const bool same = a_km && pr.A == pr.B && pr.lda == pr.ldb && m0 == n0;        // diagonal Gram tile: one operand
  const bool vec_a = pr.vec_a != 0, vec_b = pr.vec_b != 0;
  const bool want_colsum = pr.colsum != nullptr && tm == tn;
  float colacc = 0.f;        // thread t < BM of a group: column m0 + t
  float sha[4], shb[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int ca = vec_a ? m0 + 4 * (t & 15) + i : m0 + (t & 63), cb = vec_b ? n0 + 4 * (t & 15) + i : n0 + (t & 63);
    sha[i] = pr.shift && ca < pr.m ? pr.shift[ca] : 0.f;
    shb[i] = pr.shift && cb < pr.n ? pr.shift[cb] : 0.f;
  }
  SlabRegs ra, rb;
  auto load = [&](int64_t k0) {
    if (a_km) load_kmajor(ra, pr.A, pr.lda, k0, ke, m0, pr.m, t, vec_a, pr.in_bf16);
    else load_mmajor(ra, reinterpret_cast<const float*>(pr.A), pr.lda, k0, ke, m0, pr.m, t, vec_a);
    if (!same) load_kmajor(rb, pr.B, pr.ldb, k0, ke, n0, pr.n, t, vec_b, pr.in_bf16);
  };
  auto store = [&](int64_t k0, int buf) {
    float* As = slab + buf * kSlab;
    if (a_km) store_kmajor(As, LDA, ra, sha, k0, ke, t, vec_a);
    else store_mmajor(As, ra, t);
    if (!same) store_kmajor(As + BK * LDA, LDB, rb, shb, k0, ke, t, vec_b);
  };
  auto sync = [&] {
    if (KG == 1) __syncthreads();
    else asm volatile("bar.sync %0, %1;" ::"r"(grp + 1), "r"(NT) : "memory");
  };

  int buf = 0;
  if (kb < ke) {
    load(kb);
    store(kb, 0);
  }
  sync();
  for (int64_t k0 = kb; k0 < ke; k0 += BK) {
    const bool more = k0 + BK < ke;
    if (more) load(k0 + BK);
    const float* As = slab + buf * kSlab;
    const float* Bs = same ? As : As + BK * LDA;
#pragma unroll
    for (int kk = 0; kk < BK; ++kk) {
      const float4 a0 = *reinterpret_cast<const float4*>(As + kk * LDA + TM * ty);
      const float4 a1 = *reinterpret_cast<const float4*>(As + kk * LDA + TM * ty + 4);
      const float4 b4 = *reinterpret_cast<const float4*>(Bs + kk * LDB + TN * tx);
      const float a[TM] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
      const float b[TN] = {b4.x, b4.y, b4.z, b4.w};
#pragma unroll
      for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
    }
    if (want_colsum && t < BM) {
#pragma unroll
      for (int kk = 0; kk < BK; ++kk) colacc += As[kk * LDA + t];
    }
    if (more) store(k0 + BK, buf ^ 1);
    sync();
    buf ^= 1;
  }

  // the groups' sums, added in order by the first one (thread t of every group holds the same entries)
  if (KG > 1) {
    __syncthreads();
    float4* part = reinterpret_cast<float4*>(gsm);                                // [group - 1][8][NT] float4, then column sums
    float* cols = gsm + (KG - 1) * TM * TN * NT;
    if (grp > 0) {
#pragma unroll
      for (int i = 0; i < TM; ++i)
        part[((grp - 1) * TM + i) * NT + t] = make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
      if (want_colsum && t < BM) cols[(grp - 1) * BM + t] = colacc;
    }
    __syncthreads();
    if (grp > 0) return;
#pragma unroll
    for (int q = 0; q < KG - 1; ++q) {
#pragma unroll
      for (int i = 0; i < TM; ++i) {
        const float4 o = part[(q * TM + i) * NT + t];
        acc[i][0] += o.x; acc[i][1] += o.y; acc[i][2] += o.z; acc[i][3] += o.w;
      }
      if (want_colsum && t < BM) colacc += cols[q * BM + t];
    }
  }

  // epilogue
  float* C = pr.C + (int64_t)split * pr.c_split_stride;
  const bool vec_c = pr.vec_c != 0;
  const int ng0 = n0 + TN * tx, mg0 = m0 + TM * ty;
  bool bad = false;
#pragma unroll
  for (int i = 0; i < TM; ++i) {
    const int mg = mg0 + i;
    if (mg >= pr.m || ng0 >= pr.n) continue;
    float* c = C + (int64_t)mg * pr.ldc + ng0;
    const bool quad = vec_c && ng0 + TN <= pr.n;
    float o[TN] = {0.f, 0.f, 0.f, 0.f};
    if (pr.epi == EPI_SGD) {
      if (quad) *reinterpret_cast<float4*>(o) = *reinterpret_cast<const float4*>(c);
      else
#pragma unroll
        for (int j = 0; j < TN; ++j) if (ng0 + j < pr.n) o[j] = c[j];
    }
#pragma unroll
    for (int j = 0; j < TN; ++j) {
      bad |= ng0 + j < pr.n && !isfinite(acc[i][j]);
      if (pr.epi == EPI_SGD) o[j] = fmaf(-pr.lr, acc[i][j], o[j]);
      else o[j] = pr.colbias && ng0 + j < pr.n ? acc[i][j] - pr.colbias[ng0 + j] : acc[i][j];
    }
    if (pr.epi == EPI_SYMM && tm == tn) {
      // both images of a diagonal tile come from its upper triangle
#pragma unroll
      for (int j = 0; j < TN; ++j)
        if (ng0 + j < pr.n && ng0 + j >= mg) { c[j] = o[j]; C[(int64_t)(ng0 + j) * pr.ldc + mg] = o[j]; }
      continue;
    }
    if (quad) *reinterpret_cast<float4*>(c) = *reinterpret_cast<const float4*>(o);
    else
#pragma unroll
      for (int j = 0; j < TN; ++j) if (ng0 + j < pr.n) c[j] = o[j];
  }
  if (pr.epi == EPI_SYMM && tm != tn) {
    // the mirror image: a thread's eight rows are eight consecutive entries of each of its four columns' rows
#pragma unroll
    for (int j = 0; j < TN; ++j) {
      if (ng0 + j >= pr.n) continue;
      float* c = C + (int64_t)(ng0 + j) * pr.ldc + mg0;
      if (vec_c && mg0 + TM <= pr.m) {
        *reinterpret_cast<float4*>(c) = make_float4(acc[0][j], acc[1][j], acc[2][j], acc[3][j]);
        *reinterpret_cast<float4*>(c + 4) = make_float4(acc[4][j], acc[5][j], acc[6][j], acc[7][j]);
      } else {
#pragma unroll
        for (int i = 0; i < TM; ++i) if (mg0 + i < pr.m) c[i] = acc[i][j];
      }
    }
  }
  if (want_colsum && t < BM && m0 + t < pr.m) pr.colsum[(int64_t)split * pr.m + m0 + t] = colacc;
  if (bad && pr.nonfinite) *pr.nonfinite = 1;
}

template <int KG, int CAP>
cudaError_t launch(const GemmGroup& g, int total, cudaStream_t s) {
  static SmemAttrCache attr;
  const size_t part = (KG - 1) * (size_t)(TM * TN * NT + BM), slabs = (size_t)KG * 2 * kSlab;
  const size_t smem = (part > slabs ? part : slabs) * sizeof(float);
  cudaError_t e = ensure_dyn_smem(gemm_ffma_kernel<KG, CAP>, smem, attr);
  if (e != cudaSuccess) return e;
  GemmBlock<CAP> b;
  b.n = g.n;
  memcpy(b.p, g.p, g.n * sizeof(GemmProblem));
  gemm_ffma_kernel<KG, CAP><<<total, NT * KG, smem, s>>>(b);
  return cudaGetLastError();
}
template <int KG>
cudaError_t launch_cap(const GemmGroup& g, int total, cudaStream_t s) {
  if (g.n <= 2) return launch<KG, 2>(g, total, s);
  if (g.n <= 16) return launch<KG, 16>(g, total, s);
  return launch<KG, FW_MAX_GROUP>(g, total, s);
}

bool quads(const void* p, int64_t ld) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0 && (ld & 3) == 0; }

}  // namespace

cudaError_t launch_gemm_ffma(GemmGroup& g, cudaStream_t s, int prof_class) {
  int total = 0;
  for (int i = 0; i < g.n; ++i) {
    GemmProblem& p = g.p[i];
    p.tiles_m = (p.m + BM - 1) / BM;
    p.tiles_n = (p.n + BN - 1) / BN;
    p.ntiles = p.sym ? p.tiles_n * (p.tiles_n + 1) / 2 : p.tiles_m * p.tiles_n;
    if (p.splits < 1) p.splits = 1;
    p.first_cta = total;
    total += p.ntiles * p.splits;
    p.vec_a = !p.in_bf16 && quads(p.A, p.lda) && (!p.a_kmajor || (p.m & 3) == 0);
    p.vec_b = !p.in_bf16 && quads(p.B, p.ldb) && (p.n & 3) == 0;
    p.vec_c = quads(p.C, p.ldc) && (p.c_split_stride & 3) == 0;
  }
  g.total_ctas = total;
  if (total == 0) return cudaSuccess;
  ProfScope ps(prof_class, s);
  // groups per tile: with six resident CTAs of one group an SM has all the warps it can use, so from four CTAs per SM on
  // one group suffices; below, the tile's chain is shared
  if (total >= 4 * 148) return launch_cap<1>(g, total, s);
  if (total >= 2 * 148) return launch_cap<2>(g, total, s);
  return launch_cap<4>(g, total, s);
}

}  // namespace fw
