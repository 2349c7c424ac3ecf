// Grouped fp32 (FFMA) GEMM used by the FP32 engine and by layers the tensor-core kernels do not take:
//   - the Gram pass X^T X with fused column sums (Eqs. 3, 5: the covariance sum),
//   - G * Qs with the optional fused SGD epilogue (Eqs. 27, 29),
//   - the re-sync products T Phix and (T Phix) T^T.
// One launch covers every problem of a group; a CTA finds its problem, tile and K-split from its block index.
//
// A group of 64 threads computes a 64 x 64 tile, 8 x 8 accumulators per thread (packed fp32 pairs: one instruction for two
// products), from 16-deep slabs copied asynchronously
// into three shared-memory buffers, where the thread that copied an element subtracts the Gram pass's shift from it.  It is bound by issue and the FP32 pipe when
// the tiles fill the machine (65536 x 576: pipe busy in 66 % of the cycles, 55 % of its rate in products of the tiles; the
// rest are the copies that make a pair of one operand, and latencies; shared memory is at 60 % of its wavefronts); when they do not, what counts is the length of the chain of slabs, so 2, 4 or 8 groups of a
// CTA share the tile, each a contiguous part of K, and their sums are added in order at the end: the chain is that much
// shorter and the SM has that many more warps to hide it.  Products of the ResNet-20-shaped set at batch 32 (Gram /
// re-sync / G Qs): 1028 / 310 / 101 us with 4 x 4 accumulators, scalar loads and one group; see launch_gemm_ffma.
#include <algorithm>
#include <cstring>

#include "fw_internal.h"
#include "fw_lanes.cuh"
#include "fw_sm100.cuh"

namespace fw {

namespace {

constexpr int BM = 64, BN = 64, BK = 16;             // tile, slab
constexpr int TM = 8;                                // rows per thread
constexpr int LDA = BM + 4;                          // shared-memory rows of both operands
constexpr int kSlab = 2 * BK * LDA;                  // floats of one stage
constexpr int kStages = 3;

// The kernel's argument block carries as many problems as the launch needs: a launch costs 0.7 us per KB of arguments.
template <int CAP>
struct GemmBlock {
  int32_t n;
  GemmProblem p[CAP];
};

__device__ __forceinline__ void fma2(u64& c, u64 a, u64 b) { asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(c) : "l"(a), "l"(b)); }

__device__ __forceinline__ void cp_async16(float* d, const float* p, bool in) {
  const uint32_t sa = (uint32_t)__cvta_generic_to_shared(d);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(sa), "l"(p), "r"(in ? 16 : 0) : "memory");
}
__device__ __forceinline__ void cp_async4(float* d, const float* p, bool in) {
  const uint32_t sa = (uint32_t)__cvta_generic_to_shared(d);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(sa), "l"(p), "r"(in ? 4 : 0) : "memory");
}

__device__ __forceinline__ uint32_t cluster_size() {
  uint32_t n;
  asm("mov.u32 %0, %%cluster_nctaid.x;" : "=r"(n));
  return n;
}
__device__ __forceinline__ float4 ld_cluster(uint32_t a) {
  float4 v;
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(a) : "memory");
  return v;
}

// A group's shape: TN columns per thread, so 64 (TN = 8) or 128 (TN = 4) threads.
template <int TN>
struct Shape {
  static constexpr int NT = BM * BN / (TM * TN);
  static constexpr int KV = NT / 16, KS = NT / 64;   // rows of a slab a pass of the group covers: quads, single columns
};

// One operand's slab into shared memory (row k of the slab at S + k LDA), asynchronously.  A thread copies
// quads of columns 4 (t % 16) ... of rows k = t / 16 + KV e, or (not vec) column t % 64 of rows k = t / 64 + KS e from p, its
// first element of the slab; `left` rows of K are inside the matrix, the rest becomes zero (base: an address inside the
// matrix for the copies that read nothing).
template <int TN>
__device__ __forceinline__ void stage_kmajor(float* S, const float* p, const float* base, int64_t ld, int left, bool in, int t,
                                             bool vec) {
  if (vec) {
    constexpr int KV = Shape<TN>::KV;
    const int k0 = t >> 4;
#pragma unroll
    for (int e = 0; e < BK / KV; ++e) {
      const bool ok = in && k0 + KV * e < left;
      cp_async16(S + (k0 + KV * e) * LDA + 4 * (t & 15), ok ? p + KV * e * ld : base, ok);
    }
  } else {
    constexpr int KS = Shape<TN>::KS;
    const int k0 = t >> 6;
#pragma unroll
    for (int e = 0; e < BK / KS; ++e) {
      const bool ok = in && k0 + KS * e < left;
      cp_async4(S + (k0 + KS * e) * LDA + (t & 63), ok ? p + KS * e * ld : base, ok);
    }
  }
}
template <int TN>
__device__ __forceinline__ void stage_bf16(float* S, const __nv_bfloat16* p, int64_t ld, int left, bool in, int t) {
  constexpr int KS = Shape<TN>::KS;
  const int k0 = t >> 6;
#pragma unroll
  for (int e = 0; e < BK / KS; ++e)
    S[(k0 + KS * e) * LDA + (t & 63)] = (in && k0 + KS * e < left) ? __bfloat162float(p[KS * e * ld]) : 0.f;
}
// The shift, subtracted from the elements inside the matrix by the thread that copied them
template <int TN>
__device__ __forceinline__ void centre(float* S, const float (&sh)[4], int left, int t, bool vec) {
  if (vec) {
    constexpr int KV = Shape<TN>::KV;
#pragma unroll
    for (int e = 0; e < BK / KV; ++e) {
      const int kk = (t >> 4) + KV * e;
      float4* q = reinterpret_cast<float4*>(S + kk * LDA + 4 * (t & 15));
      if (kk < left) { float4 x = *q; x.x -= sh[0]; x.y -= sh[1]; x.z -= sh[2]; x.w -= sh[3]; *q = x; }
    }
  } else {
    constexpr int KS = Shape<TN>::KS;
#pragma unroll
    for (int e = 0; e < BK / KS; ++e) {
      const int kk = (t >> 6) + KS * e;
      if (kk < left) S[kk * LDA + (t & 63)] -= sh[0];
    }
  }
}
// An M-major operand (stored m x k) is transposed on its way: a thread (TN = 4) takes quads of k = 4 (t / 64) + 8 e of row
// t % 64 through registers, loaded before a slab's products and stored after them.
struct QuadRegs { float4 q[2]; };
__device__ __forceinline__ void load_mmajor(QuadRegs& r, const float* p, int left, bool in, int t, bool vec) {
#pragma unroll
  for (int e = 0; e < 2; ++e) {
    const int k = 4 * (t >> 6) + 8 * e;
    r.q[e] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (!in) continue;
    if (vec && k + 4 <= left) r.q[e] = *reinterpret_cast<const float4*>(p + k);
    else {
      if (k < left) r.q[e].x = p[k];
      if (k + 1 < left) r.q[e].y = p[k + 1];
      if (k + 2 < left) r.q[e].z = p[k + 2];
      if (k + 3 < left) r.q[e].w = p[k + 3];
    }
  }
}
__device__ __forceinline__ void store_mmajor(float* S, const QuadRegs& r, int t) {
#pragma unroll
  for (int e = 0; e < 2; ++e) {
    float* d = S + (4 * (t >> 6) + 8 * e) * LDA + (t & 63);
    d[0] = r.q[e].x; d[LDA] = r.q[e].y; d[2 * LDA] = r.q[e].z; d[3 * LDA] = r.q[e].w;
  }
}

extern __shared__ __align__(16) float gsm[];

// AKM: A is K-major (copied asynchronously); else M-major, TN = 4
// SHARED: the CTAs of a cluster share a tile's K (an instantiation of its own: even reading the cluster's size costs a launch of
// M = 64 half a microsecond)
template <int TN, bool AKM, int KG, int CAP, bool SHARED>
__global__ void __launch_bounds__(Shape<TN>::NT * KG, TN == 8 ? 8 / KG : 1) gemm_ffma_kernel(const __grid_constant__ GemmBlock<CAP> g) {
  constexpr int NT = Shape<TN>::NT;
  // locate the problem this CTA, or its cluster, works on
  const int kc = SHARED ? (int)cluster_size() : 1, rank = SHARED ? (int)sm100::cluster_ctarank() : 0;
  const int cta = SHARED ? (int)blockIdx.x / kc : (int)blockIdx.x;
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
  const int groups = KG * kc, part_of_k = rank * KG + grp;
  const int64_t gper = (max(se - sb, (int64_t)0) + groups - 1) / groups;
  const int64_t kb = (sb + part_of_k * gper) * BK, ke = min(min(sb + (part_of_k + 1) * gper, se) * BK, pr.k);

  float* slab = gsm + grp * kStages * kSlab;
  const int tx = t % (BN / TN), ty = t / (BN / TN);
  u64 acc2[TM / 2][TN];      // rows 8 ty + 2 i, + 1; columns 4 tx + j (and 32 + 4 tx + j - 4)
#pragma unroll
  for (int i = 0; i < TM / 2; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) acc2[i][j] = 0;
  const bool same = AKM && pr.A == pr.B && pr.lda == pr.ldb && m0 == n0;        // diagonal Gram tile: one operand
  const bool vec_a = pr.vec_a != 0, vec_b = pr.vec_b != 0;
  const int bf16 = pr.in_bf16;
  const bool want_colsum = pr.colsum != nullptr && tm == tn;
  float colacc = 0.f;        // column m0 + t
  // my column (or row) of each operand, and whether it is inside the matrix
  const int ca = AKM && vec_a ? m0 + 4 * (t & 15) : m0 + (t & 63), cb = vec_b ? n0 + 4 * (t & 15) : n0 + (t & 63);
  const bool in_a = ca < pr.m, in_b = cb < pr.n;
  dep_sync();                // so far: parameters only
  float sha[4] = {0.f, 0.f, 0.f, 0.f}, shb[4] = {0.f, 0.f, 0.f, 0.f};
  if (pr.shift) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      if (ca + i < pr.m) sha[i] = pr.shift[ca + i];
      if (cb + i < pr.n) shb[i] = pr.shift[cb + i];
    }
  }
  const int64_t lda = pr.lda, ldb = pr.ldb;
  const float* pa = reinterpret_cast<const float*>(pr.A);
  const float* pb = reinterpret_cast<const float*>(pr.B);
  {
    const int64_t oa = AKM ? (kb + (vec_a ? t >> 4 : t >> 6)) * lda + ca : (int64_t)ca * lda + kb;
    const int64_t ob = (kb + (vec_b ? t >> 4 : t >> 6)) * ldb + cb;
    if (bf16) {
      pa = reinterpret_cast<const float*>(reinterpret_cast<const __nv_bfloat16*>(pr.A) + oa);
      pb = reinterpret_cast<const float*>(reinterpret_cast<const __nv_bfloat16*>(pr.B) + ob);
    } else {
      pa += oa; pb += ob;
    }
  }
  const int64_t step_a = AKM ? BK * lda : BK, step_b = BK * ldb;
  QuadRegs rq;
  auto stage = [&](int left, int buf) {
    float* S = slab + buf * kSlab;
    if (bf16) {
      stage_bf16<TN>(S, reinterpret_cast<const __nv_bfloat16*>(pa), lda, left, in_a, t);
      if (!same) stage_bf16<TN>(S + BK * LDA, reinterpret_cast<const __nv_bfloat16*>(pb), ldb, left, in_b, t);
      pa = reinterpret_cast<const float*>(reinterpret_cast<const __nv_bfloat16*>(pa) + step_a);
      pb = reinterpret_cast<const float*>(reinterpret_cast<const __nv_bfloat16*>(pb) + step_b);
    } else {
      if (AKM) stage_kmajor<TN>(S, pa, reinterpret_cast<const float*>(pr.A), lda, left, in_a, t, vec_a);
      else load_mmajor(rq, pa, left, in_a, t, vec_a);
      if (!same) stage_kmajor<TN>(S + BK * LDA, pb, reinterpret_cast<const float*>(pr.B), ldb, left, in_b, t, vec_b);
      pa += step_a; pb += step_b;
    }
  };
  auto commit = [] { asm volatile("cp.async.commit_group;" ::: "memory"); };
  auto sync = [&] {
    if (KG == 1) __syncthreads();
    else asm volatile("bar.sync %0, %1;" ::"r"(grp + 1), "r"(NT) : "memory");
  };

  int64_t left64 = ke - kb;      // rows of K from the current slab on
  auto rows = [&](int ahead) { return (int)max((int64_t)0, min(left64 - ahead * BK, (int64_t)BK)); };
#pragma unroll
  for (int i = 0; i < kStages - 1; ++i) {
    if (rows(i) > 0) {
      stage(rows(i), i);
      if (!AKM) store_mmajor(slab + i * kSlab, rq, t);
    }
    commit();
  }
  int buf = 0;
  for (; left64 > 0; left64 -= BK) {
    asm volatile("cp.async.wait_group %0;" ::"n"(kStages - 2) : "memory");
    if (pr.shift) {
      float* S = slab + buf * kSlab;
      centre<TN>(S, sha, rows(0), t, vec_a);
      if (!same) centre<TN>(S + BK * LDA, shb, rows(0), t, vec_b);
    }
    sync();                      // the slab is complete, and the one before it is free
    const int nb = buf == 0 ? kStages - 1 : buf - 1;
    const bool more = rows(kStages - 1) > 0;
    if (more) stage(rows(kStages - 1), nb);
    commit();
    const float* As = slab + buf * kSlab;
    const float* Bs = same ? As : As + BK * LDA;
#pragma unroll
    for (int kk = 0; kk < BK; ++kk) {
      const ulonglong2 a0 = *reinterpret_cast<const ulonglong2*>(As + kk * LDA + TM * ty);
      const ulonglong2 a1 = *reinterpret_cast<const ulonglong2*>(As + kk * LDA + TM * ty + 4);
      const float4 b0 = *reinterpret_cast<const float4*>(Bs + kk * LDA + 4 * tx);
      const float4 b1 = TN == 8 ? *reinterpret_cast<const float4*>(Bs + kk * LDA + 32 + 4 * tx) : b0;
      const u64 a[TM / 2] = {a0.x, a0.y, a1.x, a1.y};
      const float bs[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
#pragma unroll
      for (int j = 0; j < TN; ++j) {
        const u64 b = pack2(bs[j], bs[j]);
#pragma unroll
        for (int i = 0; i < TM / 2; ++i) fma2(acc2[i][j], a[i], b);
      }
    }
    if (want_colsum && t < BM) {
#pragma unroll
      for (int kk = 0; kk < BK; ++kk) colacc += As[kk * LDA + t];
    }
    if (!AKM && more) store_mmajor(slab + nb * kSlab, rq, t);
    buf = buf == kStages - 1 ? 0 : buf + 1;
  }
  float acc[TM][TN];
#pragma unroll
  for (int i = 0; i < TM / 2; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) unpack2(acc2[i][j], acc[2 * i][j], acc[2 * i + 1][j]);

  asm volatile("cp.async.wait_group 0;" ::: "memory");
  // the groups' sums, added in order by the first one (thread t of every group holds the same entries)
  if (KG > 1) {
    __syncthreads();
    float4* part = reinterpret_cast<float4*>(gsm);                                // [group - 1][TN / 4 TM][NT] float4, then column sums
    float* cols = gsm + (KG - 1) * TM * TN * NT;
    if (grp > 0) {
#pragma unroll
      for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int h = 0; h < TN / 4; ++h)
          part[((grp - 1) * (TN / 4) * TM + (TN / 4) * i + h) * NT + t] =
              make_float4(acc[i][4 * h], acc[i][4 * h + 1], acc[i][4 * h + 2], acc[i][4 * h + 3]);
      if (want_colsum && t < BM) cols[(grp - 1) * BM + t] = colacc;
    }
    __syncthreads();
    if (grp > 0 && kc == 1) return;
    if (grp == 0) {
#pragma unroll
      for (int q = 0; q < KG - 1; ++q) {
#pragma unroll
        for (int i = 0; i < TM; ++i) {
#pragma unroll
          for (int h = 0; h < TN / 4; ++h) {
            const float4 o = part[(q * (TN / 4) * TM + (TN / 4) * i + h) * NT + t];
            acc[i][4 * h] += o.x; acc[i][4 * h + 1] += o.y; acc[i][4 * h + 2] += o.z; acc[i][4 * h + 3] += o.w;
          }
        }
        if (want_colsum && t < BM) colacc += cols[q * BM + t];
      }
    }
    if (SHARED && kc > 1) {
      // the CTAs' sums, added in order by the first one out of the others' shared memory, which stays until it has read them
      float4* sums = reinterpret_cast<float4*>(gsm + (KG - 1) * (BM * BN + BM));
      if (grp == 0 && rank > 0) {
#pragma unroll
        for (int i = 0; i < TM; ++i) sums[i * NT + t] = make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
      }
      sm100::cluster_arrive();
      sm100::cluster_wait();
      if (grp == 0 && rank == 0) {
        for (int r = 1; r < kc; ++r) {
          const uint32_t p = sm100::mapa_shared((uint32_t)__cvta_generic_to_shared(sums + t), (uint32_t)r);
          float4 o[TM];
#pragma unroll
          for (int i = 0; i < TM; ++i) o[i] = ld_cluster(p + (uint32_t)(i * NT * sizeof(float4)));
#pragma unroll
          for (int i = 0; i < TM; ++i) { acc[i][0] += o[i].x; acc[i][1] += o[i].y; acc[i][2] += o[i].z; acc[i][3] += o[i].w; }
        }
      }
      sm100::cluster_arrive();
      sm100::cluster_wait();
      if (grp > 0 || rank > 0) return;
    }
  }

  // epilogue
  float* C = pr.C + (int64_t)split * pr.c_split_stride;
  const bool vec_c = pr.vec_c != 0;
  const int mg0 = m0 + TM * ty;
  bool bad = false;
#pragma unroll
  for (int h = 0; h < TN / 4; ++h) {
    const int ng0 = n0 + 32 * h + 4 * tx;
#pragma unroll
    for (int i = 0; i < TM; ++i) {
      const int mg = mg0 + i;
      if (mg >= pr.m || ng0 >= pr.n) continue;
      float* c = C + (int64_t)mg * pr.ldc + ng0;
      const bool quad = vec_c && ng0 + 4 <= pr.n;
      float o[4] = {0.f, 0.f, 0.f, 0.f};
      if (pr.epi == EPI_SGD) {
        if (quad) *reinterpret_cast<float4*>(o) = *reinterpret_cast<const float4*>(c);
        else
#pragma unroll
          for (int j = 0; j < 4; ++j) if (ng0 + j < pr.n) o[j] = c[j];
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float x = acc[i][4 * h + j];
        bad |= ng0 + j < pr.n && !isfinite(x);
        if (pr.epi == EPI_SGD) o[j] = fmaf(-pr.lr, x, o[j]);
        else o[j] = pr.colbias && ng0 + j < pr.n ? x - pr.colbias[ng0 + j] : x;
      }
      if (pr.epi == EPI_SYMM && tm == tn) {
        // both images of a diagonal tile come from its upper triangle
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (ng0 + j < pr.n && ng0 + j >= mg) { c[j] = o[j]; C[(int64_t)(ng0 + j) * pr.ldc + mg] = o[j]; }
        continue;
      }
      if (quad) *reinterpret_cast<float4*>(c) = *reinterpret_cast<const float4*>(o);
      else
#pragma unroll
        for (int j = 0; j < 4; ++j) if (ng0 + j < pr.n) c[j] = o[j];
    }
    if (pr.epi == EPI_SYMM && tm != tn) {
      // the mirror image: a thread's eight rows are eight consecutive entries of each of its columns' rows
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        if (ng0 + j >= pr.n) continue;
        float* c = C + (int64_t)(ng0 + j) * pr.ldc + mg0;
        const int q = 4 * h + j;
        if (vec_c && mg0 + TM <= pr.m) {
          *reinterpret_cast<float4*>(c) = make_float4(acc[0][q], acc[1][q], acc[2][q], acc[3][q]);
          *reinterpret_cast<float4*>(c + 4) = make_float4(acc[4][q], acc[5][q], acc[6][q], acc[7][q]);
        } else {
#pragma unroll
          for (int i = 0; i < TM; ++i) if (mg0 + i < pr.m) c[i] = acc[i][q];
        }
      }
    }
  }
  if (want_colsum && t < BM && m0 + t < pr.m) pr.colsum[(int64_t)split * pr.m + m0 + t] = colacc;
  if (bad && pr.nonfinite) *pr.nonfinite = 1;
}

template <int TN, bool AKM, int KG, int CAP, bool SHARED>
cudaError_t launch(const GemmGroup& g, int total, int kc, cudaStream_t s) {
  static SmemAttrCache attr;
  const size_t part = (KG - 1) * (size_t)(BM * BN + BM) + (SHARED ? BM * BN : 0), slabs = (size_t)KG * kStages * kSlab;
  const size_t smem = (part > slabs ? part : slabs) * sizeof(float);
  cudaError_t e = ensure_dyn_smem(gemm_ffma_kernel<TN, AKM, KG, CAP, SHARED>, smem, attr);
  if (e != cudaSuccess) return e;
  GemmBlock<CAP> b;
  b.n = g.n;
  memcpy(b.p, g.p, g.n * sizeof(GemmProblem));
  if (SHARED) return launch_dep_cluster(kc, gemm_ffma_kernel<TN, AKM, KG, CAP, SHARED>, total * kc, Shape<TN>::NT * KG, smem, s, b);
  return launch_dep(gemm_ffma_kernel<TN, AKM, KG, CAP, SHARED>, total, Shape<TN>::NT * KG, smem, s, b);
}
template <int TN, bool AKM, int KG, bool SHARED = false>
cudaError_t launch_cap(const GemmGroup& g, int total, cudaStream_t s, int kc = 1) {
  if (g.n <= 2) return launch<TN, AKM, KG, 2, SHARED>(g, total, kc, s);
  if (g.n <= 16) return launch<TN, AKM, KG, 16, SHARED>(g, total, kc, s);
  return launch<TN, AKM, KG, FW_MAX_GROUP, SHARED>(g, total, kc, s);
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
  // A launch's problems all have the same kind of A.  Groups per tile: an SM holds eight groups of 64 threads (four of
  // 128); with fewer tiles than that the chain of a tile is shared, and below one tile per SM it is what counts, so the
  // groups have 128 threads there.
  const int sms = sm_count();
  // A tile is 64 x 64 x K products on one SM, 9.4 us of its FP32 pipe at K = 576: with few tiles a cluster of CTAs shares each, as
  // long as a group keeps four slabs of the longest K and the clusters fill at most three quarters of the SMs (beyond that two
  // CTAs meet on an SM, and 36 tiles of K = 576 took 30 us on four CTAs each instead of 22 on one).  G Qs, one CTA -> shared:
  // 64 x 576 22 -> 13 us, 256 x 576 22 -> 16, 64 x 1024 36 -> 15, 16 x 2304 68 -> 38; not taken: 16 x 144 8.7 -> 9.7.  The longest
  // K decides for a group of several: it is the last to end, and the others' clusters fit beside it (67 x 27 and 67 x 603 16.9 us,
  // 67 x 603 alone 17.0, both unshared 30.7).  Eight CTAs a tile would need K above 1000 in at most 13 tiles, and there are at least K / 64.
  int kc = 1;
  int64_t kslabs = 0;
  bool whole = true;                  // column sums and row splits are the Gram pass's, whose partition is the caller's
  for (int i = 0; i < g.n; ++i) { kslabs = std::max(kslabs, (g.p[i].k + BK - 1) / BK); whole = whole && !g.p[i].colsum && g.p[i].splits == 1; }
  while (whole && kc < 4 && 8 * kc * total <= 3 * sms && kslabs >= 16 * kc) kc *= 2;
  if (!g.p[0].a_kmajor) {
    if (total >= 4 * sms) return launch_cap<4, false, 1>(g, total, s);
    if (kc > 1) return launch_cap<4, false, 4, true>(g, total, s, kc);
    return launch_cap<4, false, 4>(g, total, s);
  }
  if (total >= 6 * sms) return launch_cap<8, true, 1>(g, total, s);
  if (total >= 3 * sms) return launch_cap<8, true, 2>(g, total, s);
  if (total >= sms) return launch_cap<8, true, 4>(g, total, s);
  if (kc > 1) return launch_cap<4, true, 4, true>(g, total, s, kc);
  return launch_cap<4, true, 4>(g, total, s);
}

}  // namespace fw
