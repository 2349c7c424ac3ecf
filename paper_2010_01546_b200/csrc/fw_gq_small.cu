// G~ = G Qs (Eq. 29) with the optional SGD step (Eq. 27) for small layers of the tensor-core engine: N up to 128 rows, M up to
// 1024.  Such a product is a few dozen MFLOP, so what bounds it is latency: the CTA-pair kernel (fw_umma_gq.cu) takes 7 to 8 us
// for one tile (tensor memory, pipeline fill, 256-wide tiles, a second launch where K is split).  Here a tile is 64 rows by
// 32 columns and its K is shared by a cluster of one, two, four or eight CTAs, at most 168 each: a CTA brings its whole share of both
// operands to shared memory in one go (one trip to memory), multiplies it with warp-level TF32 instructions, and the
// cluster's partial tiles are added in rank order out of shared memory.  With so little to do for each CTA the start-up of tcgen05
// (allocation, descriptors, commit and read-back) costs more than its rate gains.  (Operands go in as they are.  PTX leaves the
// low 13 bits of a TF32 operand open; measured, the instruction ignores them, as tcgen05 does.)
#include <algorithm>
#include <cstdio>
#include <cstring>

#include "fw_sm100.cuh"
#include "fw_umma.h"

namespace fw {

using namespace sm100;

namespace {

constexpr int GS_MAX = 16;             // problems per launch
constexpr int GS_THREADS = 256;
constexpr int GS_N = 64, GS_M = 32;    // rows and columns of a tile
constexpr int GS_KC = 168;             // K a CTA takes at most
constexpr int GS_QLD = GS_M + 8;       // shared-memory rows of Qs and of partial tiles: fragments without bank conflicts
constexpr int GS_PLD = GS_M + 4;
constexpr int GS_WARPS = GS_THREADS / 32;
constexpr int GS_CL = 8;               // largest cluster
constexpr int GS_MAX_N = 128, GS_MAX_M = 1024;

struct GsProblem {
  const float* Qs;
  const float* G;
  float* out;
  int32_t* nonfinite;
  int32_t N, M, tiles_m, first;        // first: tiles before this problem's
};
struct GsArgs {
  GsProblem p[GS_MAX];
  int32_t n, cl, epi;
  float lr;
};

// K per CTA of a cluster of cl: a multiple of 8, so that rows of kc + 4 floats put a fragment's rows on distinct banks
__host__ __device__ inline int gs_share(int M, int cl) { return ((M + cl - 1) / cl + 7) & ~7; }
// no more CTAs than hold K: a larger cluster starts later than it gains (M = 576, eight for four: 8.3 for 6.8 us)
inline int gs_cluster(int M) {
  int cl = 1;
  while (gs_share(M, cl) > GS_KC) cl *= 2;
  return cl;
}
inline size_t gs_smem(int kc) { return sizeof(float) * ((size_t)GS_N * (kc + 4) + (size_t)kc * GS_QLD + 16 * GS_WARPS * GS_PLD); }

__device__ __forceinline__ void copy16(float* dst, const float* src, bool valid) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_u32(dst)), "l"(src), "r"(valid ? 16 : 0) : "memory");
}
// D (16 x 8) += A (16 x 8) B (8 x 8)
__device__ __forceinline__ void mma_16x8x8(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3]) : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

__global__ void __launch_bounds__(GS_THREADS) gq_small_kernel(const __grid_constant__ GsArgs a) {
  extern __shared__ __align__(16) float gs_smem_f[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int cl = a.cl, rank = (int)blockIdx.x % cl, tile = (int)blockIdx.x / cl;
  int pi = 0;
#pragma unroll 1
  for (int i = 1; i < a.n; ++i)
    if (tile >= a.p[i].first) pi = i;
  const GsProblem& pr = a.p[pi];
  const int N = pr.N, M = pr.M;
  const int n0 = (tile - pr.first) / pr.tiles_m * GS_N, m0 = (tile - pr.first) % pr.tiles_m * GS_M;
  const int kc = gs_share(M, cl), k0 = rank * kc, kn = min(kc, M - k0);        // kn <= 0: nothing left for this CTA
  const int ldg = kc + 4;
  float* sG = gs_smem_f;
  float* sQ = sG + GS_N * ldg;
  float* part = sQ + kc * GS_QLD;
  dep_sync();
  // my share of both operands; past the end of K both are zero (entries past N or M reach only results that are not kept)
  for (int r = warp; r < GS_N; r += GS_THREADS / 32) {
    if (n0 + r >= N) break;
    const float* src = pr.G + (int64_t)(n0 + r) * M + k0;
    for (int c = lane; c < (kc >> 2); c += 32) copy16(sG + r * ldg + 4 * c, 4 * c < kn ? src + 4 * c : pr.G, 4 * c < kn);
  }
  for (int i = tid; i < kc * (GS_M / 4); i += GS_THREADS) {
    const int k = i >> 3, c = 4 * (i & 7);
    const bool in = k < kn && m0 + c < M;
    copy16(sQ + k * GS_QLD + c, in ? pr.Qs + (int64_t)(k0 + k) * M + m0 + c : pr.Qs, in);
  }
  asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
  __syncthreads();
  // The tile's rows are one, two or four tiles of 16; the warps beyond that share K.  A warp: 16 rows by all columns, every
  // kq-th part of the k steps.
  const int rt = n0 + 16 >= N ? 1 : n0 + 32 >= N ? 2 : 4, nq = GS_WARPS / rt;
  const int r0 = 16 * (warp % rt), kq = warp / rt, gr = lane >> 2, t = lane & 3;
  float d[GS_M / 8][4];
#pragma unroll
  for (int h = 0; h < GS_M / 8; ++h) d[h][0] = d[h][1] = d[h][2] = d[h][3] = 0.f;
  const float* ga = sG + (r0 + gr) * ldg + t;
  const float* qb = sQ + t * GS_QLD + gr;
#pragma unroll 2
  for (int k = 8 * kq; k < kc; k += 8 * nq) {
    const uint32_t fa[4] = {__float_as_uint(ga[k]), __float_as_uint(ga[k + 8 * ldg]), __float_as_uint(ga[k + 4]), __float_as_uint(ga[k + 8 * ldg + 4])};
#pragma unroll
    for (int h = 0; h < GS_M / 8; ++h)
      mma_16x8x8(d[h], fa, __float_as_uint(qb[k * GS_QLD + 8 * h]), __float_as_uint(qb[(k + 4) * GS_QLD + 8 * h]));
  }
  float* mine = part + (16 * warp + gr) * GS_PLD + 2 * t;          // warp kq rt + i: part kq of rows 16 i and on
#pragma unroll
  for (int h = 0; h < GS_M / 8; ++h) {
    *reinterpret_cast<float2*>(mine + 8 * h) = make_float2(d[h][0], d[h][1]);
    *reinterpret_cast<float2*>(mine + 8 * GS_PLD + 8 * h) = make_float2(d[h][2], d[h][3]);
  }
  // the warps' shares of K, then those of the cluster's CTAs, each of which adds a part of the rows; in order
  const int all = 16 * rt, rows = all / cl;
  if (nq > 1) {
    __syncthreads();
    for (int i = tid; i < all * (GS_M / 4); i += GS_THREADS) {
      float4* p = reinterpret_cast<float4*>(part + (i >> 3) * GS_PLD + 4 * (i & 7));
      float4 v = *p;
      for (int q = 1; q < nq; ++q) {
        const float4 x = p[q * all * (GS_PLD / 4)];
        v.x += x.x; v.y += x.y; v.z += x.z; v.w += x.w;
      }
      *p = v;
    }
  }
  if (cl > 1) { cluster_arrive(); cluster_wait(); }
  else __syncthreads();
  for (int i = tid; i < rows * (GS_M / 4); i += GS_THREADS) {
    const int r = rank * rows + (i >> 3), c = 4 * (i & 7);
    if (n0 + r >= N || m0 + c >= M) continue;
    const uint32_t at = smem_u32(part + r * GS_PLD + c);
    float4* o = reinterpret_cast<float4*>(pr.out + (int64_t)(n0 + r) * M + m0 + c);
    float4 w = make_float4(0.f, 0.f, 0.f, 0.f);
    if (a.epi == EPI_SGD) w = *o;
    float4 x[GS_CL];
#pragma unroll
    for (int q = 0; q < GS_CL; ++q)              // all on their way before any is added
      if (q < cl)
        asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
                     : "=f"(x[q].x), "=f"(x[q].y), "=f"(x[q].z), "=f"(x[q].w) : "r"(mapa_shared(at, (uint32_t)q)) : "memory");
    float4 v = x[0];
#pragma unroll
    for (int q = 1; q < GS_CL; ++q)
      if (q < cl) { v.x += x[q].x; v.y += x[q].y; v.z += x[q].z; v.w += x[q].w; }
    if (pr.nonfinite && !(isfinite(v.x) && isfinite(v.y) && isfinite(v.z) && isfinite(v.w))) *pr.nonfinite = 1;
    if (a.epi == EPI_SGD) {
      w.x = fmaf(-a.lr, v.x, w.x); w.y = fmaf(-a.lr, v.y, w.y); w.z = fmaf(-a.lr, v.z, w.z); w.w = fmaf(-a.lr, v.w, w.w);
      *o = w;
    } else {
      *o = v;
    }
  }
  if (cl > 1) { cluster_arrive(); cluster_wait(); }       // no CTA leaves while a peer may read its partial tile
}

}  // namespace

// Every problem of a launch gets the cluster of the longest (a launch for each size of cluster took longer: 300 x 64 three times beside 144 x
// 32 and 576 x 16, eight layers, 16.0 us for 9.7, by CTA pairs 12.0), so three things are asked for:
// - rows: tiles with the K that they need, counted by their rows, come to no more than 64 rows an SM.  One product of 64 x 576 takes
//   6.8 us here and 8.0 by CTA pairs, 32 x 288 4.9 and 6.9, 128 x 576 7.0 and 8.9, 20 x 1000 5.8 and 9.2; but 64 x 1024 9.8 and 8.4, the
//   fifteen of a ResNet-20-shaped set 19 and 13.5.
// - where K is shared by four CTAs or more, no more tiles than nine to ten SMs for each launch that the pairs need (sixteen layers), however few
//   rows they have: 10 x 576 six times 9.7 and 11.7 us, eight times 12.6 and 11.8, twelve times 17.6 and 11.9; 1 x 1000 four times 13.5 and
//   18.4, eight times 25.3 and 18.7, sixteen times 53 and 20.  (Below that 10 x 300 64 times: 34.9 and 39.9.)
// - CTAs beyond those that the layers' own K takes: no more than one an SM.  10 x 1000 beside fifteen of 16 x 144 is 856 for 331: 14.3 and
//   11.4 us; beside 32 x 576, 32 x 300 and 32 x 64, 496 for 350: 10.1 and 13.6.
// 16-byte accesses throughout: rows of whole float4s and aligned matrices.
bool gq_small_eligible(const UmmaGqItem* items, int n) {
  int64_t rows = 0, tiles = 0, ctas = 0;
  int cl = 1;
  for (int i = 0; i < n; ++i) {
    const UmmaGqItem& it = items[i];
    const uintptr_t p = (uintptr_t)it.Qs | (uintptr_t)it.G | (uintptr_t)it.out;
    if (it.N > GS_MAX_N || it.M > GS_MAX_M || it.M % 4 != 0 || (p & 15) != 0 || it.colbias) return false;
    const int64_t wide = (it.M + GS_M - 1) / GS_M, t = wide * ((it.N + GS_N - 1) / GS_N);
    const int c = gs_cluster(it.M);
    rows += wide * it.N * c; tiles += t; ctas += t * c;
    cl = std::max(cl, c);
  }
  const int64_t sms = sm_count();
  if (rows > GS_N * sms) return false;
  if (cl >= 4 && 10 * tiles > 9 * sms * ((n + GS_MAX - 1) / GS_MAX)) return false;
  return cl * tiles - ctas <= sms;
}

fw_status gq_small_launch(const UmmaGqItem* items, int n, int epi, float lr, int prof_class, cudaStream_t s) {
  static SmemAttrCache attr;
  if (ensure_dyn_smem(gq_small_kernel, gs_smem(GS_KC), attr) != cudaSuccess) { cudaGetLastError(); return FW_ERR_CUDA; }
  for (int base = 0; base < n; base += GS_MAX) {
    GsArgs a;
    memset(&a, 0, sizeof(a));
    a.n = std::min(n - base, GS_MAX); a.epi = epi; a.lr = lr;
    int longest = 0, tiles = 0;
    for (int i = 0; i < a.n; ++i) {
      const UmmaGqItem& it = items[base + i];
      GsProblem& p = a.p[i];
      p.Qs = it.Qs; p.G = it.G; p.out = it.out; p.nonfinite = it.nonfinite; p.N = (int32_t)it.N; p.M = it.M;
      p.tiles_m = (it.M + GS_M - 1) / GS_M; p.first = tiles;
      tiles += p.tiles_m * (int)((it.N + GS_N - 1) / GS_N);
      longest = std::max(longest, it.M);
    }
    a.cl = gs_cluster(longest);
    ProfScope ps(prof_class, s);
    const cudaError_t e = launch_dep_cluster(a.cl, gq_small_kernel, tiles * a.cl, GS_THREADS, gs_smem(gs_share(longest, a.cl)), s, a);
    if (e != cudaSuccess) {
      fprintf(stderr, "[fw] gq_small_kernel launch: %s\n", cudaGetErrorString(e));
      return FW_ERR_CUDA;
    }
  }
  return FW_OK;
}

}  // namespace fw
