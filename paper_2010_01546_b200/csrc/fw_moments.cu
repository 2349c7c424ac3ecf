// Moment kernels around the Gram pass (Eqs. 2-5, 37-38, 31):
//   pilot_mean     column means of the first rows of X, used to centre X inside
//                  the Gram pass so that the one-pass covariance does not cancel
//   moments_vec    reduce the split column sums, update mu, phi, lam_bar
//   moments_mat    reduce the split Gram partials, centre on the updated mean,
//                  running average into Phix, mirror to the lower triangle
//   bias_comp      b += W (mu_new - mu_old), carried by extra CTAs of the moments_mat launch
//   accumulate     a call that leaves its block open: its split sums are added to the block's accumulators
#include <algorithm>
#include <cstring>

#include "fw_internal.h"
#include "fw_sm100.cuh"

namespace fw {
namespace {

constexpr int kPilotRows = 512;     // rows sampled for the pilot mean
constexpr int kPilotTY = 16;        // row lanes per block

// f(r0) + f(r0 + STEP) + ... below n, added in that order.  The loads of eight terms are in flight together, the last ones
// too: what a sum of a few dozen terms costs is the chain of load latencies (the pilot mean of M = 2304: 22 us with one
// load at a time, 13 so).
template <int STEP, class F>
__device__ __forceinline__ float strided_sum(int64_t r0, int64_t n, F f) {
  float s = 0.f;
  for (; r0 < n; r0 += 8 * STEP) {
    float v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) v[u] = r0 + u * STEP < n ? f(r0 + u * STEP) : 0.f;
#pragma unroll
    for (int u = 0; u < 8; ++u) if (r0 + u * STEP < n) s += v[u];
  }
  return s;
}

__global__ void pilot_mean_kernel(const __grid_constant__ GroupDev g, const __grid_constant__ PtrTable X,
                                  const __grid_constant__ Rows64 rows, const __grid_constant__ Rows64 ldx,
                                  int in_bf16, int to_pmean) {
  dep_sync();
  const LayerDev* L = g.layer[blockIdx.y];
  const int M = L->M;
  const int col = blockIdx.x * 32 + threadIdx.x;
  if (blockIdx.x * 32 >= M) return;
  int64_t R = rows.v[blockIdx.y];
  if (R > kPilotRows) R = kPilotRows;
  const int64_t ld = ldx.v[blockIdx.y];
  float acc = 0.f;
  if (col < M) {
    if (in_bf16) {
      const __nv_bfloat16* x = reinterpret_cast<const __nv_bfloat16*>(X.p[blockIdx.y]);
      acc = strided_sum<kPilotTY>(threadIdx.y, R, [&](int64_t r) { return __bfloat162float(x[r * ld + col]); });
    } else {
      const float* x = reinterpret_cast<const float*>(X.p[blockIdx.y]);
      acc = strided_sum<kPilotTY>(threadIdx.y, R, [&](int64_t r) { return x[r * ld + col]; });
    }
  }
  __shared__ float sm[kPilotTY][33];
  sm[threadIdx.y][threadIdx.x] = acc;
  __syncthreads();
  if (threadIdx.y == 0 && col < M) {
    float s = 0.f;
#pragma unroll
    for (int i = 0; i < kPilotTY; ++i) s += sm[i][threadIdx.x];
    (to_pmean ? L->pmean : L->shift)[col] = s / (float)R;
  }
}

struct MomentArgs {
  int32_t splits[FW_MAX_GROUP];
  int32_t first[FW_MAX_GROUP];
  int32_t use_acc[FW_MAX_GROUP];     // add the sums accumulated by the block's earlier calls (accumulate kernel:
                                     // 0 = overwrite the accumulators, 1 = add to them)
  float corr[FW_MAX_GROUP];          // > 0: corr c c^T was taken out of this call's Gram sums (c = rounded pmean)
  TileTable tt;                      // flat grid over the upper-triangle 32x32 tiles of all layers
  int32_t sum_blocks;                // CTAs of moments_vec_kernel behind its one per layer that add the split partials of a tile each into
                                     // gram_acc; 0: moments_mat_kernel adds them
  int32_t bias_blocks;               // CTAs per layer placed before the tiles for b += W (mu_new - mu_old); 0: none
};

// s, d += the split partials [k0, k1) of a column's sum and of its diagonal entry, in split order; the loads of eight splits are
// issued together, the last ones too (the chain of additions is short, the chain of load latencies is what a plain loop
// would pay).
__device__ __forceinline__ void split_sums(const float* cp, const float* gp, int64_t M, int64_t MM, int k0, int k1, float& s, float& d) {
  for (int k = k0; k < k1; k += 8) {
    float sv[8], dv[8];
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (k + u < k1) { sv[u] = cp[(int64_t)(k + u) * M]; dv[u] = gp[(int64_t)(k + u) * MM]; }
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (k + u < k1) { s += sv[u]; d += dv[u]; }
  }
}

// Four consecutive entries of a row, i fixed: V4 in one access (rows of whole float4s), else one by one below M.
template <bool V4>
__device__ __forceinline__ float4 load_quad(const float* p, int j, int M) {
  if (V4) return *reinterpret_cast<const float4*>(p);
  float4 r = make_float4(0.f, 0.f, 0.f, 0.f);
  r.x = p[0];
  if (j + 1 < M) r.y = p[1];
  if (j + 2 < M) r.z = p[2];
  if (j + 3 < M) r.w = p[3];
  return r;
}
template <bool V4>
__device__ __forceinline__ void store_quad(float* p, int j, int M, float4 v) {
  if (V4) { *reinterpret_cast<float4*>(p) = v; return; }
  p[0] = v.x;
  if (j + 1 < M) p[1] = v.y;
  if (j + 2 < M) p[2] = v.z;
  if (j + 3 < M) p[3] = v.w;
}

// Entries (i, j) ... (i, j + 3) of a layer's Gram sums: split partials in split order, eight loads in flight at a time, the last
// ones too; then what was taken out of them and the block's earlier calls.
template <bool V4>
__device__ __forceinline__ float4 gram_quad(const LayerDev* L, const MomentArgs& a, int li, int i, int j) {
  const int M = L->M, S = a.splits[li];
  const int64_t off = (int64_t)i * M + j, MM = (int64_t)M * M;
  float4 s2 = make_float4(0.f, 0.f, 0.f, 0.f);
  const float* gp = L->gram_part + off;
  for (int k0 = 0; k0 < S; k0 += 8) {
    float4 v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (k0 + u < S) v[u] = load_quad<V4>(gp + (int64_t)(k0 + u) * MM, j, M);
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (k0 + u < S) { s2.x += v[u].x; s2.y += v[u].y; s2.z += v[u].z; s2.w += v[u].w; }
  }
  const float corr = a.corr[li];
  if (corr > 0.f) {                                                // symmetric in (i, j)
    const int xbf = L->x_dtype == FW_BF16;
    const float ci = corr_round(L->pmean[i], xbf);
    const float4 pm = load_quad<V4>(L->pmean + j, j, M);
    s2.x = fmaf(corr, __fmul_rn(ci, corr_round(pm.x, xbf)), s2.x); s2.y = fmaf(corr, __fmul_rn(ci, corr_round(pm.y, xbf)), s2.y);
    s2.z = fmaf(corr, __fmul_rn(ci, corr_round(pm.z, xbf)), s2.z); s2.w = fmaf(corr, __fmul_rn(ci, corr_round(pm.w, xbf)), s2.w);
  }
  if (a.use_acc[li]) {
    const float4 g4 = load_quad<V4>(L->gram_acc + off, j, M);
    s2.x += g4.x; s2.y += g4.y; s2.z += g4.z; s2.w += g4.w;
  }
  return s2;
}

// One entry, by the same operations in the same order; sixteen loads in flight.
__device__ __forceinline__ float gram_sum(const LayerDev* L, const MomentArgs& a, int li, int i, int j) {
  const int M = L->M, S = a.splits[li];
  const int64_t off = (int64_t)i * M + j, MM = (int64_t)M * M;
  const float* gp = L->gram_part + off;
  float s2 = 0.f;
  for (int k0 = 0; k0 < S; k0 += 16) {
    float v[16];
#pragma unroll
    for (int u = 0; u < 16; ++u)
      if (k0 + u < S) v[u] = gp[(int64_t)(k0 + u) * MM];
#pragma unroll
    for (int u = 0; u < 16; ++u)
      if (k0 + u < S) s2 += v[u];
  }
  const float corr = a.corr[li];
  if (corr > 0.f) {
    const int xbf = L->x_dtype == FW_BF16;
    s2 = fmaf(corr, __fmul_rn(corr_round(L->pmean[i], xbf), corr_round(L->pmean[j], xbf)), s2);
  }
  return s2;
}

// the layer and the 32 x 32 tile (bi <= bj) of its upper triangle that a place in the flat list of tiles stands for
__device__ __forceinline__ int find_tile(const GroupDev& g, const MomentArgs& a, int tile_id, int& bi, int& bj) {
  int li = 0;
#pragma unroll 1
  for (int i = 1; i < g.n; ++i)
    if (tile_id >= a.tt.tile0[i]) li = i;
  tri_decode(tile_id - a.tt.tile0[li], (g.layer[li]->M + 31) / 32, bi, bj);
  return li;
}

// One CTA per layer, 1024 threads (one column each for M <= 1024), and a.sum_blocks CTAs that meanwhile add the split partials
// of a tile each, a thread an entry.
__global__ void __launch_bounds__(1024) moments_vec_kernel(const __grid_constant__ GroupDev g,
                                                          const __grid_constant__ Rows64 rows,
                                                          const __grid_constant__ MomentArgs a) {
  dep_sync();
  if ((int)blockIdx.x >= g.n) {
    int bi, bj;
    const int li = find_tile(g, a, (int)blockIdx.x - g.n, bi, bj);
    const LayerDev* L = g.layer[li];
    const int i = bi * 32 + ((int)threadIdx.x >> 5), j = bj * 32 + ((int)threadIdx.x & 31);
    if (i < L->M && j < L->M) L->gram_acc[(int64_t)i * L->M + j] = gram_sum(L, a, li, i, j);
    return;
  }
  const LayerDev* L = g.layer[blockIdx.x];
  const int M = L->M;
  const int S = a.splits[blockIdx.x];
  const bool first = a.first[blockIdx.x] != 0;
  const float inv_rows = 1.0f / (float)rows.v[blockIdx.x];
  const float alpha = L->alpha;
  float phisum = 0.f;
  bool bad = false;
  // A narrow layer leaves most of the block idle while every column walks all S split partials, eight loads at a
  // time: the splits are dealt to KG groups of threads (group kg takes a contiguous range of splits), whose sums
  // are then added in group order -- a fixed order for given (M, S), and a chain of S / (8 KG) load latencies.
  __shared__ float part_s[1024], part_d[1024];
  const int KG = M <= 512 ? min(8, 1024 / M) : 1;
  const int per = (S + KG - 1) / KG;
  const int64_t MM = (int64_t)M * M;
  if (KG > 1) {
    const int kg = threadIdx.x / M, m = threadIdx.x - kg * M;
    if (kg < KG) {
      float s = 0.f, d = 0.f;
      split_sums(L->colsum_part + m, L->gram_part + (int64_t)m * M + m, M, MM, kg * per, min(S, (kg + 1) * per), s, d);
      part_s[threadIdx.x] = s; part_d[threadIdx.x] = d;
    }
    __syncthreads();
  }
  for (int m = threadIdx.x; m < M; m += blockDim.x) {
    const float c = L->shift[m], mu_old = L->mu[m], phi_old = first ? 0.f : L->phi[m];     // under way beside the partial sums
    float s = 0.f, d = 0.f;
    if (KG > 1) {
      for (int kg = 0; kg < KG; ++kg) { s += part_s[kg * M + m]; d += part_d[kg * M + m]; }
    } else {
      split_sums(L->colsum_part + m, L->gram_part + (int64_t)m * M + m, M, MM, 0, S, s, d);
    }
    if (a.corr[blockIdx.x] > 0.f) {
      const float cm = corr_round(L->pmean[m], L->x_dtype == FW_BF16);
      d = fmaf(a.corr[blockIdx.x], cm * cm, d);
    }
    if (a.use_acc[blockIdx.x]) { s += L->colsum_acc[m]; d += L->gram_acc[(int64_t)m * M + m]; }
    const float mh_rel = s * inv_rows;          // batch mean relative to the shift
    const float mhat = c + mh_rel;
    const float mu_new = first ? mhat : fmaf(alpha, mu_old, (1.f - alpha) * mhat);
    L->mu_prev[m] = mu_old;
    L->mu[m] = mu_new;
    // uncentred power (Eq. 37): mean x^2 = mean (x-c)^2 + 2 c mean(x-c) + c^2
    const float ph = fmaf(d, inv_rows, fmaf(2.f * c, mh_rel, c * c));
    const float ph_new = first ? ph : fmaf(alpha, phi_old, (1.f - alpha) * ph);
    L->phi[m] = ph_new;
    phisum += ph_new;
    // per-call scratch in the power-iteration vectors (dead outside a reduction call): batch mean and new
    // mean relative to the shift
    L->pv[0][m] = mh_rel;
    L->pv[1][m] = mu_new - c;
    if (!isfinite(s) || !isfinite(d)) bad = true;
  }
  // Block reduction of phisum, a tree over the threads (t and t + 512, t and t + 256, ... t and t + 1): the upper five levels in
  // the registers of the first warp, the others by shuffles.
  __shared__ float red[1024];
  red[threadIdx.x] = phisum;
  __syncthreads();
  if (threadIdx.x < 32) {
    float v[32];
#pragma unroll
    for (int k = 0; k < 32; ++k) v[k] = red[threadIdx.x + 32 * k];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
      for (int k = 0; k < o; ++k) v[k] += v[k + o];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v[0] += __shfl_down_sync(0xffffffffu, v[0], o);
    if (threadIdx.x == 0) L->scal[SC_LAMBDA_BAR] = v[0] / (float)M;   // Eq. 38
  }
  if (bad) L->iscal[IS_STATUS_NONFINITE] = 1;
}

__device__ __forceinline__ void bias_comp_rows(const LayerDev* L, const float* Wp, float* bp, int blk, int tid);

// One 32 x 32 tile (bi <= bj) of one layer, a thread four entries of a row; the mirror image leaves through shared memory.
// SUMMED: the split partials have been added, into gram_acc.
template <bool V4, bool SUMMED>
__device__ __forceinline__ void moments_tile(const LayerDev* L, const MomentArgs& a, int li, float inv_rows, int bi, int bj,
                                             float (&tile)[32][33]) {
  const int M = L->M, tid = threadIdx.x;
  const bool first = a.first[li] != 0;
  const float alpha = L->alpha;
  const int ii = tid >> 3, qc = 4 * (tid & 7), i = bi * 32 + ii, j = bj * 32 + qc;
  if (i < M && j < M) {
    const int64_t off = (int64_t)i * M + j;
    const float4 old = first ? make_float4(0.f, 0.f, 0.f, 0.f) : load_quad<V4>(L->Phix + off, j, M);
    const float mh_i = L->pv[0][i], nu_i = L->pv[1][i];           // batch mean - shift, new running mean - shift
    const float4 mh_j = load_quad<V4>(L->pv[0] + j, j, M), nu_j = load_quad<V4>(L->pv[1] + j, j, M);
    const float4 s2 = SUMMED ? load_quad<V4>(L->gram_acc + off, j, M) : gram_quad<V4>(L, a, li, i, j);
    // (1/rows) sum (x-mu)(x-mu)^T with x - mu = (x - c) - nu, written symmetrically in i, j so that the result mirrors exactly
    auto entry = [&](float s, float mhj, float nuj, float o) {
      const float cross = __fadd_rn(__fmul_rn(mh_i, nuj), __fmul_rn(nu_i, mhj));
      const float chat = __fadd_rn(__fsub_rn(__fmul_rn(s, inv_rows), cross), __fmul_rn(nu_i, nuj));
      return first ? chat : __fadd_rn(__fmul_rn(alpha, o), __fmul_rn(1.f - alpha, chat));
    };
    const float4 out = make_float4(entry(s2.x, mh_j.x, nu_j.x, old.x), entry(s2.y, mh_j.y, nu_j.y, old.y),
                                   entry(s2.z, mh_j.z, nu_j.z, old.z), entry(s2.w, mh_j.w, nu_j.w, old.w));
    if (bi != bj) store_quad<V4>(L->Phix + off, j, M, out);
    tile[ii][qc] = out.x; tile[ii][qc + 1] = out.y; tile[ii][qc + 2] = out.z; tile[ii][qc + 3] = out.w;
  }
  __syncthreads();
  // element (r, c) of the tile goes to (c, r); in a diagonal tile the entries on and above the diagonal stay where they are
  const int jg = bj * 32 + ii, ig = bi * 32 + qc;
  if (jg < M && ig < M) {
    float v[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) v[e] = (bi == bj && qc + e >= ii) ? tile[ii][qc + e] : tile[qc + e][ii];
    store_quad<V4>(L->Phix + (int64_t)jg * M + ig, ig, M, make_float4(v[0], v[1], v[2], v[3]));
  }
}

// One CTA per 32 x 32 tile of the upper triangle of one layer; the grid is the flat list of these
// tiles over all layers of the group (a grid sized for the largest layer would be mostly empty CTAs when the
// layers differ in size, and handing those out costs more than the work).  Bound by the latency of the split partials where
// layers are small, by HBM where they are large; with a 16-byte access per row and split instead of four rows of 4 bytes one
// after the other, and moments_vec_kernel's sums batched: 368 -> 362 us a step of the
// ResNet-20-shaped set, 5074 -> 5005 of the ResNet-50-shaped set, 342 -> 321 of one with odd sizes.
template <bool SUMMED>
__global__ void __launch_bounds__(256) moments_mat_kernel(const __grid_constant__ GroupDev g,
                                                          const __grid_constant__ Rows64 rows,
                                                          const __grid_constant__ MomentArgs a,
                                                          const __grid_constant__ PtrTable W,
                                                          const __grid_constant__ PtrTable b) {
  dep_sync();
  const int nbias = a.bias_blocks * g.n;
  if ((int)blockIdx.x < nbias) {
    // the first CTAs carry the bias compensation (Eq. 31), which needs the means only: long rows of W start early
    // and the tiles fill in behind them
    const int layer = (int)blockIdx.x / a.bias_blocks, blk = (int)blockIdx.x - layer * a.bias_blocks;
    bias_comp_rows(g.layer[layer], reinterpret_cast<const float*>(W.p[layer]),
                   const_cast<float*>(reinterpret_cast<const float*>(b.p[layer])), blk, threadIdx.x);
    return;
  }
  int bi, bj;
  const int li = find_tile(g, a, (int)blockIdx.x - nbias, bi, bj);
  const LayerDev* L = g.layer[li];
  __shared__ float tile[32][33];
  const float inv_rows = 1.0f / (float)rows.v[li];
  if ((L->M & 3) == 0) moments_tile<true, SUMMED>(L, a, li, inv_rows, bi, bj, tile);
  else moments_tile<false, SUMMED>(L, a, li, inv_rows, bi, bj, tile);
}

// A call that leaves its block open (FW_COV_ACCUMULATE): the split sums of this call are added, in split order,
// to the block's accumulators (or overwrite them on the block's first call).  Same flat grid over the
// upper-triangle 32x32 tiles as moments_mat_kernel; the CTAs of a layer's first tile row also carry the column sums.
__global__ void __launch_bounds__(256) accumulate_kernel(const __grid_constant__ GroupDev g,
                                                         const __grid_constant__ MomentArgs a) {
  dep_sync();
  const int tile_id = (int)blockIdx.x;
  int li = 0;
#pragma unroll 1
  for (int i = 1; i < g.n; ++i)
    if (tile_id >= a.tt.tile0[i]) li = i;
  const LayerDev* L = g.layer[li];
  const int M = L->M;
  int bi, bj;
  tri_decode(tile_id - a.tt.tile0[li], (M + 31) / 32, bi, bj);
  const int S = a.splits[li];
  const bool add = a.use_acc[li] != 0;
  const float corr = a.corr[li];
  const int xbf = L->x_dtype == FW_BF16;
  const int j = bj * 32 + threadIdx.x;
  const float ct_j = (corr > 0.f && j < M) ? corr_round(L->pmean[j], xbf) : 0.f;
  const int64_t MM = (int64_t)M * M;
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const int i = bi * 32 + threadIdx.y + 8 * r;
    if (i < M && j < M) {
      const int64_t off = (int64_t)i * M + j;
      float s2 = 0.f;
      for (int k = 0; k < S; ++k) s2 += L->gram_part[off + (int64_t)k * MM];
      if (corr > 0.f) s2 = fmaf(corr, __fmul_rn(corr_round(L->pmean[i], xbf), ct_j), s2);
      L->gram_acc[off] = add ? L->gram_acc[off] + s2 : s2;
    }
  }
  if (bi == 0 && threadIdx.y == 0 && j < M) {
    float s = 0.f;
    for (int k = 0; k < S; ++k) s += L->colsum_part[(int64_t)k * M + j];
    L->colsum_acc[j] = add ? L->colsum_acc[j] + s : s;
  }
}

// b += W (mu_new - mu_old); one warp per output row, 8 rows per CTA
__device__ __forceinline__ void bias_comp_rows(const LayerDev* L, const float* Wp, float* bp, int blk, int tid) {
  if (!Wp || !bp) return;
  const int M = L->M, N = L->N;
  const int row = blk * 8 + (tid >> 5);
  if (row >= N) return;
  const int lane = tid & 31;
  float acc = 0.f;
  for (int m = lane; m < M; m += 32) acc = fmaf(Wp[(int64_t)row * M + m], L->mu[m] - L->mu_prev[m], acc);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if (lane == 0) bp[row] += acc;
}

// Zero-padded copies of NHWC activations: dst[b][y + 1][x + 1][:] = src[b][y][x][:], one pixel of zeros all round, for
// every layer of a group in one launch.  A warp takes a padded image row at a time, so that its place in the tensors is
// found once per row; all 16-byte loads of four trips are in flight before the first store.
struct PadGroup {
  const float4* src[FW_MAX_GROUP];
  float4* dst[FW_MAX_GROUP];
  int32_t row0[FW_MAX_GROUP + 1];     // first padded row of each layer in the flat list of rows
  int32_t H[FW_MAX_GROUP], W4[FW_MAX_GROUP], C4[FW_MAX_GROUP];   // W4: 16-byte units of an unpadded row
  int32_t tail[FW_MAX_GROUP];         // units past the padded tensor that the last window may read: zeros
  int32_t n;
};
__global__ void __launch_bounds__(256) pad_nhwc_kernel(const __grid_constant__ PadGroup g) {
  dep_sync();
  const int lane = threadIdx.x & 31, nw = gridDim.x * 8, total = g.row0[g.n];
  const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
  for (int w = blockIdx.x * 8 + (threadIdx.x >> 5); w < total; w += nw) {
    int li = 0;
#pragma unroll 1
    for (int i = 1; i < g.n; ++i)
      if (w >= g.row0[i]) li = i;
    const int r = w - g.row0[li], H = g.H[li], W4 = g.W4[li], C4 = g.C4[li];
    const int b = r / (H + 2), y = r - b * (H + 2);
    const int len = W4 + 2 * C4;
    float4* d = g.dst[li] + (int64_t)r * len;
    const bool border = y == 0 || y == H + 1;
    const float4* s = g.src[li] + ((int64_t)b * H + (y - 1)) * W4 - C4;      // unit c of the padded row is s[c] inside
    for (int c0 = lane; c0 < len; c0 += 128) {
      float4 v[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int c = c0 + 32 * u;
        v[u] = !border && c >= C4 && c < len - C4 ? __ldg(s + c) : z;
      }
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (c0 + 32 * u < len) d[c0 + 32 * u] = v[u];
    }
    if (w + 1 == g.row0[li + 1])
      for (int c = lane; c < g.tail[li]; c += 32) d[len + c] = z;
  }
}

__global__ void init_identity_kernel(const LayerDev* L) {
  dep_sync();
  const int M = L->M;
  const int64_t n = (int64_t)M * M;
  const bool alias = (L->Qs == L->Q);
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
    const int i = (int)(e / M), j = (int)(e - (int64_t)i * M);
    const float d = (i == j) ? 1.f : 0.f;
    L->Tt[e] = d;
    if (L->round_t) L->tmp[e] = d;
    L->Q[e] = d;
    if (!alias) L->Qs[e] = d;
    L->Phix[e] = 0.f;
    L->Phiy[e] = 0.f;
  }
  if (blockIdx.x == 0) {
    for (int m = threadIdx.x; m < M; m += blockDim.x) {
      L->mu[m] = 0.f; L->mu_prev[m] = 0.f; L->phi[m] = 0.f; L->shift[m] = 0.f;
    }
    for (int m = threadIdx.x; m < 3 * ((M + 15) & ~15); m += blockDim.x) L->px[m] = 0;     // no exchange has this number
    if (threadIdx.x < SC_COUNT) L->scal[threadIdx.x] = 0.f;
    if (threadIdx.x < IS_COUNT) L->iscal[threadIdx.x] = 0;
  }
}

__global__ void transpose_kernel(const float* __restrict__ src, float* __restrict__ dst, int M) {
  dep_sync();
  __shared__ float tile[32][33];
  const int bi = blockIdx.y * 32, bj = blockIdx.x * 32;
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const int i = bi + threadIdx.y + 8 * r, j = bj + threadIdx.x;
    if (i < M && j < M) tile[threadIdx.y + 8 * r][threadIdx.x] = src[(int64_t)i * M + j];
  }
  __syncthreads();
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const int j = bj + threadIdx.y + 8 * r, i = bi + threadIdx.x;
    if (i < M && j < M) dst[(int64_t)j * M + i] = tile[threadIdx.x][threadIdx.y + 8 * r];
  }
}

// dst <- src, n floats each; the CTAs are dealt to the copies by their sizes.  v4: both 16-byte aligned; what is left
// of a float4 at the end goes float by float (one float a thread throughout took 137 instead of 92 us for M = 8191).
template <int N>                        // 1 or FW_MAX_GROUP: a KB of parameters costs a launch 0.7 us
struct CopyGroup {
  const float* src[N];
  float* dst[N];
  int32_t n[N];                         // floats, at most 8192 x 8192
  int32_t v4[N];
  int32_t first[N + 1];                 // first CTA of each copy
  int32_t copies;
};
// ROUND: the copy is rounded to the TF32 grid (nearest, ties away)
template <int N, bool ROUND>
__global__ void __launch_bounds__(256) copy_kernel(const __grid_constant__ CopyGroup<N> g) {
  dep_sync();
  int c = 0;
#pragma unroll 1
  for (int i = 1; i < g.copies; ++i)
    if ((int)blockIdx.x >= g.first[i]) c = i;
  const float* src = g.src[c];
  float* dst = g.dst[c];
  const int n = g.n[c], step = 256 * (g.first[c + 1] - g.first[c]), i0 = 256 * ((int)blockIdx.x - g.first[c]) + threadIdx.x;
  auto val = [](float x) { return ROUND ? sm100::tf32_rna(x) : x; };
  if (g.v4[c]) {
#pragma unroll 4
    for (int i = i0; i < (n >> 2); i += step) {
      const float4 x = reinterpret_cast<const float4*>(src)[i];
      reinterpret_cast<float4*>(dst)[i] = make_float4(val(x.x), val(x.y), val(x.z), val(x.w));
    }
    if (i0 < (n & 3)) dst[(n & ~3) + i0] = val(src[(n & ~3) + i0]);
  } else {
#pragma unroll 4
    for (int i = i0; i < n; i += step) dst[i] = val(src[i]);
  }
}

// out = A^T x: 32 columns per CTA, the rows dealt to its 32 warps and their sums added in order
__global__ void __launch_bounds__(1024) matT_vec_kernel(const float* __restrict__ A, const float* __restrict__ x,
                                                        float* __restrict__ out, int M) {
  dep_sync();
  __shared__ float sm[32][33];
  const int j = blockIdx.x * 32 + threadIdx.x;
  float acc = 0.f;
  if (j < M) {
#pragma unroll 4
    for (int k = threadIdx.y; k < M; k += 32) acc = fmaf(A[(int64_t)k * M + j], x[k], acc);
  }
  sm[threadIdx.y][threadIdx.x] = acc;
  __syncthreads();
  if (threadIdx.y == 0 && j < M) {
    float t = 0.f;
#pragma unroll
    for (int i = 0; i < 32; ++i) t += sm[i][threadIdx.x];
    out[j] = t;
  }
}

// lam_bar = trace(Phix) / M after a covariance has been injected
__global__ void __launch_bounds__(256) trace_lambda_kernel(const LayerDev* L) {
  dep_sync();
  const int M = L->M;
  float s = 0.f;
  for (int m = threadIdx.x; m < M; m += blockDim.x) s += L->Phix[(int64_t)m * M + m];
  __shared__ float red[256];
  red[threadIdx.x] = s;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) L->scal[SC_LAMBDA_BAR] = red[0] / (float)M;
}

// b <- b - lr g_b for every layer of a group; grid (ceil(max N / 256), layers)
__global__ void sgd_bias_group_kernel(const __grid_constant__ GroupDev g, const __grid_constant__ PtrTable b,
                                      const __grid_constant__ PtrTable gb, float lr) {
  dep_sync();
  const LayerDev* L = g.layer[blockIdx.y];
  float* bp = const_cast<float*>(reinterpret_cast<const float*>(b.p[blockIdx.y]));
  const float* gp = reinterpret_cast<const float*>(gb.p[blockIdx.y]);
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (bp && gp && i < L->N) bp[i] = fmaf(-lr, gp[i], bp[i]);
}

// W <- W - lr G and b <- b - lr g_b (b may be null) in one launch
__global__ void __launch_bounds__(256) sgd_step_kernel(float* __restrict__ W, const float* __restrict__ G, int64_t n,
                                                       float* __restrict__ b, const float* __restrict__ gb, int N, float lr) {
  dep_sync();
  const int64_t first = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, step = (int64_t)gridDim.x * blockDim.x;
  for (int64_t e = first; e < n; e += step) W[e] = fmaf(-lr, G[e], W[e]);
  if (b)
    for (int64_t e = first; e < N; e += step) b[e] = fmaf(-lr, gb[e], b[e]);
}

// v <- momentum v + (G + wd W), W <- W - lr v, and the same without decay for the bias (may be null), in one launch
__device__ __forceinline__ void momentum_entry(float* __restrict__ W, const float* __restrict__ G, float* __restrict__ v,
                                               int64_t e, float lr, float momentum, float wd) {
  const float w = W[e];
  const float vn = fmaf(momentum, v[e], fmaf(wd, w, G[e]));
  v[e] = vn;
  W[e] = fmaf(-lr, vn, w);
}
__global__ void __launch_bounds__(256) momentum_step_kernel(float* __restrict__ W, const float* __restrict__ G,
                                                            float* __restrict__ v, int64_t n, float* __restrict__ b,
                                                            const float* __restrict__ gb, float* __restrict__ vb, int N,
                                                            float lr, float momentum, float wd) {
  dep_sync();
  const int64_t first = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, step = (int64_t)gridDim.x * blockDim.x;
  for (int64_t e = first; e < n; e += step) momentum_entry(W, G, v, e, lr, momentum, wd);
  if (b)
    for (int64_t e = first; e < N; e += step) momentum_entry(b, gb, vb, e, lr, momentum, 0.f);
}

// Eq. 51 over all index pairs.  One CTA; every thread sums its rows in fp64, fixed-order tree over the block.
__global__ void __launch_bounds__(1024) whiteness_kernel(const float* __restrict__ A, int M, float* __restrict__ out) {
  dep_sync();
  double acc = 0.0;
  for (int i = threadIdx.x >> 5; i < M; i += 32) {          // a warp per row
    const double dii = A[(int64_t)i * M + i];
    double r = 0.0;
    for (int j = threadIdx.x & 31; j < M; j += 32) {
      const double a = A[(int64_t)i * M + j];
      r += a * a / (dii * (double)A[(int64_t)j * M + j]);
    }
    acc += r;
  }
  __shared__ double red[1024];
  red[threadIdx.x] = acc;
  __syncthreads();
  for (int o = 512; o > 0; o >>= 1) {
    if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) out[0] = (float)((double)M / red[0]);
}

}  // namespace

static int step_blocks(int64_t n) {
  const int64_t blocks = (n + 255) / 256;
  return (int)(blocks > 2368 ? 2368 : (blocks < 1 ? 1 : blocks));
}

cudaError_t launch_momentum_step(float* W, const float* G, float* v, int64_t n, float* b, const float* gb, float* vb, int N,
                                 float lr, float momentum, float wd, cudaStream_t s) {
  ProfScope ps(FW_PROF_MISC, s);
  return launch_dep(momentum_step_kernel, step_blocks(n), 256, 0, s, W, G, v, n, b, gb, vb, N, lr, momentum, wd);
}

cudaError_t launch_whiteness(const float* A, int M, float* out, cudaStream_t s) {
  ProfScope ps(FW_PROF_MISC, s);
  return launch_dep(whiteness_kernel, 1, 1024, 0, s, A, M, out);
}

cudaError_t launch_pilot_mean(const GroupDev& g, const PtrTable& X, const Rows64& rows, const Rows64& ldx,
                              int in_bf16, int max_M, int to_pmean, cudaStream_t s) {
  dim3 grid((max_M + 31) / 32, g.n), block(32, kPilotTY);
  ProfScope ps(FW_PROF_PILOT, s);
  return launch_dep(pilot_mean_kernel, grid, block, 0, s, g, X, rows, ldx, in_bf16, to_pmean);
}

cudaError_t launch_accumulate(const GroupDev& g, const int32_t* splits, const int32_t* fresh, const float* corr,
                              const int32_t* layer_M, cudaStream_t s) {
  MomentArgs a;
  memset(&a, 0, sizeof(a));
  for (int i = 0; i < g.n; ++i) { a.splits[i] = splits[i]; a.use_acc[i] = fresh[i] ? 0 : 1; a.corr[i] = corr[i]; }
  const int total = fill_tile_table(a.tt, layer_M, g.n);
  ProfScope ps(FW_PROF_MOMENTS, s);
  return launch_dep(accumulate_kernel, total, dim3(32, 8), 0, s, g, a);
}

cudaError_t launch_moments(const GroupDev& g, const Rows64& rows, const int32_t* splits, const int32_t* first,
                           const int32_t* use_acc, const float* corr, const int32_t* layer_M, const PtrTable& W,
                           const PtrTable& b, int max_M, int max_N, bool any_params, cudaStream_t s) {
  (void)max_M;
  MomentArgs a;
  memset(&a, 0, sizeof(a));
  for (int i = 0; i < g.n; ++i) {
    a.splits[i] = splits[i]; a.first[i] = first[i]; a.use_acc[i] = use_acc[i]; a.corr[i] = corr[i];
  }
  const int total = fill_tile_table(a.tt, layer_M, g.n);
  a.bias_blocks = any_params ? (max_N + 7) / 8 : 0;
  // The tiles' split partials are added beside the vectors where the CTAs of both are on the chip at once, two of 1024 threads an SM.
  // fp32 sums, all in moments_mat_kernel and side by side: covariance update of 64 x 128 rows 16.0 and 15.4 us, 147 x 3000 53 and 29,
  // 75 x 7504 49 and 43, 27 x 30000 62 and 51, 402 x 6000 128 and 107, 576 x 6000 109 and 83; tensor cores 64 x 20000 34.7 and
  // 32.7, 700 x 3000 50 and 42.  (1000 x 2000, 530 tiles: 47.4, side by side 43.7, but such a launch is no longer one wave.)  A block of
  // several calls holds its sums in gram_acc, of which moments_vec_kernel reads the diagonal.
  bool side = g.n + total <= 2 * sm_count();
  for (int i = 0; i < g.n; ++i) side = side && !use_acc[i];
  a.sum_blocks = side ? total : 0;
  cudaError_t e;
  { ProfScope ps(FW_PROF_MOMENTS, s); e = launch_dep(moments_vec_kernel, g.n + a.sum_blocks, 1024, 0, s, g, rows, a); }
  if (e != cudaSuccess) return e;
  ProfScope ps(FW_PROF_MOMENTS, s);
  return launch_dep(side ? moments_mat_kernel<true> : moments_mat_kernel<false>, total + a.bias_blocks * g.n, 256, 0, s, g, rows, a, W, b);
}

cudaError_t launch_pad_nhwc(int n, const float* const* src, float* const* dst, const int* B, const int* H, const int* W,
                            const int* C, const int64_t* dst_floats, cudaStream_t s) {
  // dst_floats covers the padded tensor plus the slack the last window may read past it: all of it is written
  PadGroup g;
  memset(&g, 0, sizeof(g));
  int rows = 0;
  for (int i = 0; i < n; ++i) {
    g.src[i] = reinterpret_cast<const float4*>(src[i]); g.dst[i] = reinterpret_cast<float4*>(dst[i]);
    g.H[i] = H[i]; g.C4[i] = C[i] / 4; g.W4[i] = W[i] * (C[i] / 4);
    g.tail[i] = (int)(dst_floats[i] / 4 - (int64_t)B[i] * (H[i] + 2) * (g.W4[i] + 2 * g.C4[i]));
    g.row0[i] = rows;
    rows += B[i] * (H[i] + 2);
  }
  g.row0[n] = rows;
  g.n = n;
  int blocks = (rows + 7) / 8;
  if (blocks > 148 * 8) blocks = 148 * 8;
  ProfScope ps(FW_PROF_PILOT, s);
  return launch_dep(pad_nhwc_kernel, blocks, 256, 0, s, g);
}

cudaError_t launch_init_identity(const LayerDev* dev, int M, cudaStream_t s) {
  int64_t n = (int64_t)M * M;
  int blocks = (int)((n + 255) / 256);
  if (blocks > 1184) blocks = 1184;
  ProfScope ps(FW_PROF_MISC, s);
  return launch_dep(init_identity_kernel, blocks, 256, 0, s, dev);
}

cudaError_t launch_transpose(const float* src, float* dst, int M, cudaStream_t s) {
  const int t = (M + 31) / 32;
  ProfScope ps(FW_PROF_MISC, s);
  return launch_dep(transpose_kernel, dim3(t, t), dim3(32, 8), 0, s, src, dst, M);
}

template <int N, bool ROUND>
static cudaError_t launch_copies_of(int n, const float* const* src, float* const* dst, const int64_t* floats, cudaStream_t s) {
  CopyGroup<N> g;
  memset(&g, 0, sizeof(g));
  int64_t total = 0;
  for (int i = 0; i < n; ++i) total += floats[i];
  // a 16-byte access a thread, or more where that would be more CTAs than run together
  const int64_t per_cta = std::max<int64_t>(1024, (total + 8 * sm_count() - 1) / (8 * sm_count()));
  g.copies = n;
  for (int i = 0; i < n; ++i) {
    g.src[i] = src[i]; g.dst[i] = dst[i]; g.n[i] = (int32_t)floats[i];
    g.v4[i] = ((reinterpret_cast<uintptr_t>(src[i]) | reinterpret_cast<uintptr_t>(dst[i])) & 15) == 0;
    g.first[i + 1] = g.first[i] + (int)((floats[i] + per_cta - 1) / per_cta);
  }
  ProfScope ps(ROUND ? FW_PROF_RESYNC : FW_PROF_MISC, s);
  return launch_dep(copy_kernel<N, ROUND>, g.first[n], 256, 0, s, g);
}
cudaError_t launch_copies(int n, const float* const* src, float* const* dst, const int64_t* floats, cudaStream_t s) {
  return n == 1 ? launch_copies_of<1, false>(n, src, dst, floats, s) : launch_copies_of<FW_MAX_GROUP, false>(n, src, dst, floats, s);
}
cudaError_t launch_round(int n, const float* const* src, float* const* dst, const int64_t* floats, cudaStream_t s) {
  return n == 1 ? launch_copies_of<1, true>(n, src, dst, floats, s) : launch_copies_of<FW_MAX_GROUP, true>(n, src, dst, floats, s);
}

cudaError_t launch_matT_vec(const float* A, const float* x, float* out, int M, cudaStream_t s) {
  ProfScope ps(FW_PROF_MISC, s);
  return launch_dep(matT_vec_kernel, (M + 31) / 32, dim3(32, 32), 0, s, A, x, out, M);
}

cudaError_t launch_trace_lambda(const LayerDev* dev, int M, cudaStream_t s) {
  (void)M;
  ProfScope ps(FW_PROF_MISC, s);
  return launch_dep(trace_lambda_kernel, 1, 256, 0, s, dev);
}

cudaError_t launch_sgd_bias_group(const GroupDev& g, const PtrTable& b, const PtrTable& gb, float lr, int max_N,
                                  cudaStream_t s) {
  ProfScope ps(FW_PROF_MISC, s);
  return launch_dep(sgd_bias_group_kernel, dim3((max_N + 255) / 256, g.n), 256, 0, s, g, b, gb, lr);
}

cudaError_t launch_sgd_step(float* W, const float* G, int64_t n, float* b, const float* gb, int N, float lr, cudaStream_t s) {
  ProfScope ps(FW_PROF_MISC, s);
  return launch_dep(sgd_step_kernel, step_blocks(n), 256, 0, s, W, G, n, b, gb, N, lr);
}

}  // namespace fw
