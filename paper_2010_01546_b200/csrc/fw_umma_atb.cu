// Re-sync products D = A^T B of square fp32 matrices below M = 1024 (larger ones: fw_umma_pair.cu), all layers of a group
// in one launch: one CTA per 128 x 128 tile, TF32 products accumulated in TMEM over all of K.
//
// What bounds a tile is latency: K = 576 is 24 stages of 24 KB, 2.6 us of tensor time and 6.7 us of staging (45 bytes per
// clock and SM), so as little as possible stands between a load and its MMA.  Operands that were written rounded to TF32 (T
// and the first product of a layer without leakage) go straight to the tensor core; the others are rounded in place by two
// groups of four warps, for alternate stages, so that the round trip through shared memory of one hides the other's.  Tiles are 128 x
// 128 so that the 190 + 120 tiles of a ResNet-20-shaped set (M = 144, 288, 576) fill the chip, two CTAs to an SM where
// there are more; each accumulates in 128 of the SM's 512 TMEM columns.
#include <algorithm>
#include <cstdio>
#include <cstring>
#include <vector>

#include "fw_sm100.cuh"
#include "fw_umma.h"

namespace fw {

using namespace sm100;

namespace {

constexpr int AB_MAX = 16;                       // layers per launch
constexpr int AB_T = 128;                        // rows and columns of a tile
constexpr int AB_SR = 24;                        // K rows per stage: four stages in the shared memory of half an SM
constexpr int AB_CW = 32;                        // columns per chunk
constexpr int AB_NC = AB_T / AB_CW;              // chunks per operand and stage
constexpr uint32_t AB_CHUNK = AB_SR * 128;       // bytes per chunk
constexpr uint32_t AB_STAGE = 2 * AB_NC * AB_CHUNK;
constexpr int AB_STAGES = 4;                     // even: a stage stays with one rounding group, which then sees every phase of its barrier
constexpr int AB_FIX = 4;                        // warps of a rounding group
constexpr int AB_THREADS = 64 + 2 * AB_FIX * 32; // TMA warp, MMA warp, two rounding groups that also write the tile
constexpr int AB_PITCH = AB_T + 4;               // floats per row of the tile in shared memory: rows on distinct banks
constexpr int AB_SMEM = AB_STAGES * AB_STAGE + 1024;
static_assert(AB_STAGES % 2 == 0 && AB_CHUNK % 1024 == 0, "stages and rounding groups; chunks of whole swizzle atoms");
static_assert(AB_T * AB_PITCH * 4 <= AB_STAGES * (int)AB_STAGE, "the tile leaves through the stages");

struct AtbProblem {
  float* C;
  int32_t fix;           // operands to be rounded in shared memory: 1 A, 2 B
  int32_t round_c;       // 1: C is rounded to TF32 (not with sym)
  int32_t* status;       // time-out word of the owning layer
  int32_t M;
  int32_t sym;           // 1: D is symmetric: tiles on and above the diagonal, mirrored
  int32_t box3;          // the maps are chunked 3-D views (M a multiple of 32): one instruction per operand and stage
  int32_t first;         // first CTA
};
struct AtbGroup {
  CUtensorMap a[AB_MAX], b[AB_MAX];
  AtbProblem p[AB_MAX];
  int32_t n;
};

__host__ __device__ inline int atb_tiles(int M, bool sym) {
  const int nb = (M + AB_T - 1) / AB_T;
  return sym ? nb * (nb + 1) / 2 : nb * nb;
}

__global__ void __launch_bounds__(AB_THREADS, 2) atb_umma_kernel(const __grid_constant__ AtbGroup g) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t bar_full[AB_STAGES], bar_ready[AB_STAGES], bar_empty[AB_STAGES], bar_accum;
  __shared__ uint32_t tmem_base_sh;
  __shared__ int abort_flag;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int pi = 0;
#pragma unroll 1
  for (int i = 1; i < g.n; ++i)
    if ((int)blockIdx.x >= g.p[i].first) pi = i;
  const AtbProblem& pr = g.p[pi];
  const int M = pr.M, M16 = (M + 15) & ~15, nb = (M + AB_T - 1) / AB_T;
  int I = 0, J = (int)blockIdx.x - pr.first;
  while (J >= (pr.sym ? nb - I : nb)) { J -= pr.sym ? nb - I : nb; ++I; }
  if (pr.sym) J += I;
  const int row0 = AB_T * I, col0 = AB_T * J, n = min(AB_T, M16 - col0), nk = (M + AB_SR - 1) / AB_SR;
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const volatile int* abortp = &abort_flag;
  if (threadIdx.x == 0) {
    abort_flag = 0;
    for (int s = 0; s < AB_STAGES; ++s) {
      mbar_init(smem_u32(&bar_full[s]), 1);
      mbar_init(smem_u32(&bar_ready[s]), AB_FIX);
      mbar_init(smem_u32(&bar_empty[s]), 1);
    }
    mbar_init(smem_u32(&bar_accum), 1);
    mbar_fence_init();
    tma_prefetch_desc(&g.a[pi]);
    tma_prefetch_desc(&g.b[pi]);
  }
  dep_sync();                                     // so far: parameters and this CTA's own shared memory only
  // stage kb: lane q < 2 NC fetches chunk q % NC of operand q / NC (one lane each operand where one box holds its chunks)
  const int op = lane / AB_NC, ch = lane % AB_NC, x0 = (op ? col0 : row0) + ch * AB_CW;
  const bool mine = op < 2 && (pr.box3 ? ch == 0 : x0 < M);
  const CUtensorMap* map = op ? &g.b[pi] : &g.a[pi];
  const int chunks = pr.box3 ? 2 * AB_NC : min(AB_NC, (M - row0 + AB_CW - 1) / AB_CW) + min(AB_NC, (M - col0 + AB_CW - 1) / AB_CW);
  auto fetch = [&](int kb, int s) {
    const uint32_t fb = smem_u32(&bar_full[s]), dst = base + s * AB_STAGE + (uint32_t)(op * AB_NC + ch) * AB_CHUNK;
    if (lane == 0) mbar_expect_tx(fb, (uint32_t)chunks * AB_CHUNK);
    __syncwarp();
    if (mine) {
      if (pr.box3) tma_load_3d(dst, map, 0, kb * AB_SR, x0 / AB_CW, fb);
      else tma_load_2d(dst, map, x0, kb * AB_SR, fb);
    }
  };
  if (warp == 0) {
    __syncwarp();                                 // the barriers are lane 0's
    for (int kb = 0; kb < min(nk, AB_STAGES); ++kb) fetch(kb, kb);
  } else if (warp == 1) {
    tmem_alloc(smem_u32(&tmem_base_sh), AB_T);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_base_sh;
  if (warp == 0) {
    int s = 0;
    uint32_t ph = 0;
    for (int kb = AB_STAGES; kb < nk; ++kb) {
      const bool got = mbar_wait(smem_u32(&bar_empty[s]), ph, abortp);
      if (!__all_sync(0xffffffffu, got)) { if (lane == 0) { abort_flag = 1; atomicExch(pr.status, 211); } break; }
      fetch(kb, s);
      if (++s == AB_STAGES) { s = 0; ph ^= 1; }
    }
  } else if (warp == 1) {
    if (elect_one()) {
      // chunks along the tile are AB_CHUNK apart, 4-row atoms 512 bytes, k-steps (8 rows) 1024
      const uint64_t ad = make_smem_desc(base, AB_CHUNK, 512, kSwizzle128B32);
      const uint64_t bd = make_smem_desc(base + AB_NC * AB_CHUNK, AB_CHUNK, 512, kSwizzle128B32);
      const uint32_t idesc = make_idesc(2, (uint32_t)n, 1, 1);
      int s = 0;
      uint32_t ph = 0, accum = 0;
      bool ok = true;
      for (int kb = 0; kb < nk; ++kb) {
        if (!mbar_wait(smem_u32(pr.fix ? &bar_ready[s] : &bar_full[s]), ph, abortp)) { abort_flag = 1; atomicExch(pr.status, 212); ok = false; break; }
        tc_fence_after();
#pragma unroll
        for (int ks = 0; ks < AB_SR / 8; ++ks) {
          const uint64_t off = (uint64_t)(s * (AB_STAGE >> 4) + ks * 64);
          mma_tf32(tmem, ad + off, bd + off, idesc, accum);
          accum = 1;
        }
        mma_commit(smem_u32(&bar_empty[s]));
        if (++s == AB_STAGES) { s = 0; ph ^= 1; }
      }
      if (ok) mma_commit(smem_u32(&bar_accum));
    }
  } else {
    const int group = (warp - 2) / AB_FIX, t = (int)threadIdx.x - 64 - group * AB_FIX * 32;
    bool got = true;
    for (int kb = group; pr.fix && kb < nk && got; kb += 2) {
      const int s = kb % AB_STAGES;
      got = mbar_wait(smem_u32(&bar_full[s]), (uint32_t)(kb / AB_STAGES) & 1, abortp);
      float4* st = reinterpret_cast<float4*>(smem_raw + (base - smem_u32(smem_raw)) + s * AB_STAGE) + t;
      constexpr int NV = (int)AB_STAGE / 2 / 16 / (AB_FIX * 32);      // of an operand
#pragma unroll
      for (int o = 0; o < 2; ++o) {
        if (!(pr.fix >> o & 1)) continue;
        float4 v[NV];
#pragma unroll
        for (int i = 0; i < NV; ++i) v[i] = st[(o * NV + i) * AB_FIX * 32];
#pragma unroll
        for (int i = 0; i < NV; ++i)
          st[(o * NV + i) * AB_FIX * 32] = make_float4(tf32_rna(v[i].x), tf32_rna(v[i].y), tf32_rna(v[i].z), tf32_rna(v[i].w));
      }
      fence_proxy_async_smem();                   // generic-proxy writes -> visible to the tensor core's reads
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&bar_ready[s]));
    }
    const int q = warp & 3;                       // TMEM lane quarter of this warp; two warps share one, half the columns each
    got = got && mbar_wait(smem_u32(&bar_accum), 0, abortp);
    if (!got) { abort_flag = 1; atomicExch(pr.status, 213); }
    asm volatile("bar.sync 1, 256;" ::: "memory");
    if (*abortp == 0) {
      // A TMEM lane is a row of the tile: the rows leave through shared memory (every MMA has completed) as 512 bytes per warp
      // instruction; the mirror image straight from the registers, where the lanes are neighbours in an output row.
      tc_fence_after();
      float* const C = pr.C;
      float* tile = reinterpret_cast<float*>(smem_raw) + ((base - smem_u32(smem_raw)) >> 2);
      const int row = row0 + q * 32 + lane;
      float* trow = tile + (q * 32 + lane) * AB_PITCH;
      for (int c0 = 16 * group; c0 < n; c0 += 32) {
        uint32_t r[16];
        tmem_ld16(tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)c0, r);
        tmem_ld_wait();
#pragma unroll
        for (int j = 0; j < 16; j += 4)
          *reinterpret_cast<float4*>(trow + c0 + j) = make_float4(__uint_as_float(r[j]), __uint_as_float(r[j + 1]),
                                                                  __uint_as_float(r[j + 2]), __uint_as_float(r[j + 3]));
        if (pr.sym && row < M) {
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            const int col = col0 + c0 + j;
            if (col > row && col < M) C[(int64_t)col * M + row] = __uint_as_float(r[j]);
          }
        }
      }
      asm volatile("bar.sync 1, 256;" ::: "memory");
      const int col = col0 + 4 * lane;            // M is a multiple of four: a group of four columns is inside or outside
      for (int t0 = 16 * group; t0 < 16 * group + 16; t0 += 8) {
        float4 v[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) v[i] = *reinterpret_cast<const float4*>(tile + (q * 32 + t0 + i) * AB_PITCH + 4 * lane);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const int r = row0 + q * 32 + t0 + i;
          if (r >= M || col >= M) continue;
          float* p = C + (int64_t)r * M + col;
          if (pr.round_c) v[i] = make_float4(tf32_rna(v[i].x), tf32_rna(v[i].y), tf32_rna(v[i].z), tf32_rna(v[i].w));
          if (!pr.sym || col >= r) {
            *reinterpret_cast<float4*>(p) = v[i];
          } else if (col + 3 >= r) {              // the diagonal runs through these four
            if (col + 1 >= r) p[1] = v[i].y;
            if (col + 2 >= r) p[2] = v[i].z;
            p[3] = v[i].w;
          }
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, AB_T);
  }
}

}  // namespace

fw_status umma_atb_launch(const UmmaAtbItem* items, int n, cudaStream_t s) {
  static SmemAttrCache attr;
  if (ensure_dyn_smem(atb_umma_kernel, AB_SMEM, attr) != cudaSuccess) {
    cudaGetLastError();
    return FW_ERR_CUDA;
  }
  // the longest tiles first: they spread over the SMs, the short ones become the second CTA of some
  std::vector<UmmaAtbItem> by_size(items, items + n);
  std::stable_sort(by_size.begin(), by_size.end(), [](const UmmaAtbItem& x, const UmmaAtbItem& y) { return x.M > y.M; });
  for (int base = 0; base < n; base += AB_MAX) {
    AtbGroup g;
    memset(&g, 0, sizeof(g));
    g.n = std::min(n - base, AB_MAX);
    int ctas = 0;
    for (int i = 0; i < g.n; ++i) {
      const UmmaAtbItem& it = by_size[base + i];
      AtbProblem& p = g.p[i];
      p.C = it.C; p.fix = it.fix; p.round_c = it.round_c; p.status = it.status; p.M = it.M; p.sym = it.sym; p.box3 = it.M % AB_CW == 0; p.first = ctas;
      ctas += atb_tiles(it.M, it.sym != 0);
      auto encode = [&](CUtensorMap* m, const float* x) {
        const uint64_t M = (uint64_t)it.M;
        return p.box3 ? tmap_encode_chunked_3d(m, false, x, M, M, M, AB_SR, AB_NC, AB_CW) : tmap_encode_2d(m, false, x, M, M, M, AB_CW, AB_SR);
      };
      if (!encode(&g.a[i], it.A) || !encode(&g.b[i], it.B)) {
        fprintf(stderr, "[fw] tensor-map encoding failed (A^T B)\n");
        return FW_ERR_CUDA;
      }
    }
    ProfScope ps(FW_PROF_RESYNC, s);
    const cudaError_t e = launch_dep(atb_umma_kernel, ctas, AB_THREADS, AB_SMEM, s, g);
    if (e != cudaSuccess) {
      fprintf(stderr, "[fw] atb_umma_kernel launch: %s\n", cudaGetErrorString(e));
      return FW_ERR_CUDA;
    }
  }
  return FW_OK;
}

}  // namespace fw
