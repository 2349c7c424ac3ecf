// Whitening from the eigenvalue decomposition (Sec. 2, Eqs. 7-10; practical gains Eqs. 32 and 34): the method the
// recursion of Sec. 4 is measured against.  Phi = V Lambda V^T is computed by one-sided block Jacobi rotations in fp64:
// Phi = R^T R (Cholesky), and the columns of W = R^T Z, starting from Z = I, are rotated until all are orthogonal; then they
// are V Lambda^(1/2): the normalised columns are the eigenvectors and their squared lengths the eigenvalues, and Z is never
// carried along.  Where Phi is not (safely) positive definite, W starts from Phi itself and ends as V Lambda, which takes
// more sweeps: 13 instead of 10 for the covariances of M = 576 here (340 to 351 rounds), 15 instead of 9 at condition 1e3.
// Columns are stored as rows, fp64 throughout: T = Phi^(-1/2) carries the rounding of the
// decomposition times cond(Phi) / 2, which fp32 cannot afford.
//
// A CTA takes a pair of blocks of 16 columns: their products (tensor-core fp64, the columns staged in shared memory), one
// sweep of 2 x 2 rotations on that 32 x 32 matrix in shared memory, accumulated into U, and W <- U^T W on the 32
// rows.  The block pairs of a round (round-robin tournament) are disjoint, so a layer's CTAs meet
// once per round, M / 16 - 1 rounds a sweep, instead of once per round of column pairs (M - 1 rounds).  The first round of a
// sweep rotates all pairs of a visit's 32 columns, the others those of different blocks (visit).  All layers of a
// group share the launch, each with CTAs and barriers of its own.  What bounds a round at M = 576 (17.8 us) is a chain, in
// clocks: staging 3500, products 4000, 16 inner rounds 9500 (592 each), update 11700 (9200 at the rate of the fp64 tensor
// cores), barrier 5000 to 7700; a round that rotates nothing takes 13000.  An inner round is a chain too: load 71, rotation 255,
// the 2 x 2 products 164, barrier and waiting for the slowest warp 100.  15 layers of the ResNet-20-shaped set: 12.5 ms from
// Phi, 9.3 from the factor (0.35 of it the factorisation), 6.7 with cross visits and inner rounds of this shape (1014 clocks
// with 256 threads on all of the matrix and as many on U, 553 with an fp32 copy of the products, which the angles alone allow).
// One-sided rotations are those of Hestenes (1958), the start from the Cholesky factor that of Veselic and
// Hari (1989), the tournament of block pairs that of Brent and Luk (1985).
//
// Then T = V diag(sqrt g) V^T (Eq. 9), Q = T^T T = V diag(g) V^T and Phi_y = T Phi T^T = V diag(g lambda) V^T come
// out of one pass over V.
#include <algorithm>
#include <cstring>

#include "fw_internal.h"
#include "fw_lanes.cuh"
#include "fw_sm100.cuh"

namespace fw {
namespace {

constexpr int ET = 512;               // threads per CTA of the rotation kernel
constexpr int EW = ET / 32;
constexpr int EB = 16;                // columns per block
constexpr int EP = 2 * EB;            // columns of a block pair
constexpr int kChunk = 640;           // entries of a column staged at a time (rows of up to this length stay for both products)
constexpr int kMaxSweeps = 60;       // (30000 rounds at the largest M: the barrier packs their number into 16 bits)
constexpr uint32_t kEvdSpin = 1u << 22;
constexpr int kSlots = 64;            // of kWords 4-byte words at the start of a layer's scratch
constexpr int kWords = 256;
constexpr double kOrthTol = 1e-14;    // |w_p . w_q| <= tol |w_p| |w_q|: the pair is left alone
// Below kFloor max_i Phi_ii a column is rounding (lambda_max is at least that diagonal entry): repeated features, for one,
// leave columns that are parallel to another one at any length.  Such columns are not rotated, and eigenvalues below
// kNull lambda_max have no direction of their own: together they span what the other eigenvectors leave.
constexpr double kFloor = 1e-14, kNull = 1e-13;

// shared-memory row stride in doubles: 4 mod 16, so that the fragments of both products read without conflicts
__host__ __device__ inline int evd_stride(int cols) { return ((cols + 15) & ~15) + 4; }
__host__ __device__ inline int evd_ld(int M) { return (M + 7) & ~7; }
constexpr int kULd = EP + 1;          // leading dimensions of the 32 x 32 matrices in shared memory: U, read along a row,
constexpr int kGLd = EP + 2;          // and the products, read along wrapped diagonals (row + column, or row - column, fixed)
constexpr int kTri = 10;              // 8 x 8 blocks of the upper triangle of a 32 x 32 matrix
constexpr int kCross = 4 * 64 + EP;    // partial sums of a warp of a cross visit: four 8 x 8 blocks and 32 squared lengths
constexpr int kPartDoubles = EW / 2 * kTri * 64;
static_assert(EW * kCross <= kPartDoubles, "partial sums of cross visits");

struct EvdLayer {
  const float* A;    // M x M symmetric input (fp32, row-major)
  double* W;         // M rows of evd_ld(M): row m is column m of Phi V
  int32_t* words;    // [0] W came from a factor of Phi, [1] abort, [kSlots + c] barriers CTA c has reached and the last round
                     // it rotated in (zeroed before the launch)
  int32_t* status;   // time-out word of the layer
  int32_t M;
  int32_t nb;        // blocks of 16 columns, rounded up to even (the tournament's players)
  int32_t cta0, n;   // its CTAs
};

struct EvdArgs {
  EvdLayer l[FW_MAX_GROUP];
  int32_t nl;
};

// maximum over the block of values that are not negative
__device__ double evd_block_max(float x) {
  __shared__ uint32_t m;
  if (threadIdx.x == 0) m = 0;
  __syncthreads();
  atomicMax(&m, __float_as_uint(x));
  __syncthreads();
  const double r = (double)__uint_as_float(m);
  __syncthreads();
  return r;
}

// D (8 x 8) += A (8 x 4) B (4 x 8): lane holds A[lane / 4][lane % 4], B[lane % 4][lane / 4], D[lane / 4][2 (lane % 4) + {0, 1}]
__device__ __forceinline__ void mma_f64(double (&d)[2], double a, double b) {
  asm("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0, %1}, {%2}, {%3}, {%0, %1};" : "+d"(d[0]), "+d"(d[1]) : "d"(a), "d"(b));
}

// Barrier number idx (from 1) of a layer's CTAs; false once the layer is aborted.  Every CTA raises its own slot and the
// first warp polls all of them: no chain of atomic additions.  The wait is bounded.  A slot also carries the last round its
// CTA rotated in, and *s_last is the latest of them: the same in every CTA, since none goes on to barrier idx + 1 unless
// what it saw at idx was recent enough to go on (and the numbers only grow).
__device__ bool evd_barrier(const EvdLayer& L, int sub, int idx, int last, int* s_abort, int* s_last) {
  __syncthreads();
  if (threadIdx.x < 32 && *s_abort == 0) {
    volatile int* slots = L.words + kSlots;
    volatile int* ab = L.words + 1;
    if (threadIdx.x == 0) {
      __threadfence();
      slots[sub] = (idx << 16) | last;
    }
    bool ok = false;
    int latest = 0;
    for (uint32_t i = 0; i < kEvdSpin && !ok; ++i) {
      bool here = true;
      latest = 0;
      for (int c = threadIdx.x; c < L.n; c += 32) {
        const int v = slots[c];
        here = here && (v >> 16) >= idx;
        latest = max(latest, v & 0xffff);
      }
      ok = __all_sync(0xffffffffu, here);
      if (!ok && (i & 63u) == 63u && *ab != 0) break;
    }
    latest = __reduce_max_sync(0xffffffffu, latest);
    if (threadIdx.x == 0) {
      if (!ok) {
        *ab = 1;
        atomicExch(L.status, 601);
        *s_abort = 1;
      }
      *s_last = latest;
      __threadfence();
    }
  }
  __syncthreads();
  return *s_abort == 0;
}

// A wait for copies gave up: report, and let the layer's other CTAs leave at their next barrier.
__device__ void evd_give_up(const EvdLayer& L) {
  if (threadIdx.x == 0) {
    atomicExch(L.status, 601);
    *(volatile int*)(L.words + 1) = 1;
  }
}

// players of pair k in inner round q: a tournament of all 32, or (CROSS) of the 16 of one block against those of the other
template <bool CROSS>
__device__ __forceinline__ void evd_players(int k, int q, int& p, int& r) {
  if (CROSS) {
    p = k;
    r = EB + ((k + q) & (EB - 1));
    return;
  }
  p = q + k; r = q - k;
  if (p >= EP - 1) p -= EP - 1;
  if (r < 0) r += EP - 1;
  if (k == 0) p = EP - 1;
}

// dynamic shared memory: [32 rows of a chunk][partial Gram blocks of the warps, later U and the second Gram buffer][Gram]
extern __shared__ __align__(16) double esm[];

// Rows of the block pair (I, J): row r of the pair is column I * 16 + r or J * 16 + r - 16 of the layer.
__device__ __forceinline__ int pair_row(int I, int J, int r) { return r < EB ? I * EB + r : J * EB + r - EB; }

// Entries [k0, k0 + nk) of the first nrows rows of the pair (I, J) into shared memory at dst, one bulk copy per row; rows past
// the matrix and entries past ld are zero.
__device__ __forceinline__ void stage_issue(const EvdLayer& L, double* dst, int I, int J, int nrows, int k0, int nk, int stride,
                                            uint32_t bar) {
  const int ld = evd_ld(L.M), have = min(nk, ld - k0);
  const int rows = max(0, min(EB, L.M - I * EB)) + (nrows > EB ? max(0, min(EB, L.M - J * EB)) : 0);
  const int tid = threadIdx.x;
  if (tid < 32) {
    asm volatile("fence.proxy.async;" ::: "memory");       // the rows were last written and read by ordinary accesses
    if (tid == 0) sm100::mbar_expect_tx(bar, (uint32_t)rows * (uint32_t)have * 8u);
    __syncwarp();
    const int row = pair_row(I, J, tid);
    if (tid < nrows && row < L.M)
      asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                   ::"r"(sm100::smem_u32(dst + tid * stride)), "l"(L.W + (int64_t)row * ld + k0), "r"((uint32_t)have * 8u), "r"(bar)
                   : "memory");
  }
  if (rows < nrows || have < nk) {
    for (int i = tid; i < nrows * nk; i += ET) {
      const int r = i / nk, c = i - r * nk;
      if (pair_row(I, J, r) >= L.M || c >= have) dst[r * stride + c] = 0.0;
    }
  }
}
// Waits for the copies (parity: of their mbarrier) and for the block; false when the bounded wait gave up.
__device__ __forceinline__ bool stage_wait(uint32_t bar, uint32_t parity) {
  bool ok = false;
  for (uint32_t i = 0; i < sm100::kSpinLimit && !ok; ++i) ok = sm100::mbar_try_wait(bar, parity);
  return __syncthreads_and(ok) != 0;
}
__device__ __forceinline__ bool stage_rows(const EvdLayer& L, int I, int J, int k0, int nk, int stride, uint32_t bar, uint32_t parity) {
  stage_issue(L, esm, I, J, EP, k0, nk, stride, bar);
  return stage_wait(bar, parity);
}

__device__ __forceinline__ float rsqrt_approx(float x) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
// x 2^(127 - e) as fp32, truncated, for e the (biased) fp64 exponent of a number at least as large; 0 when too small
__device__ __forceinline__ float to_float_scaled(double x, int e) {
  const int hi = __double2hiint(x), lo = __double2loint(x);
  const int ex = ((hi >> 20) & 0x7ff) - e + 127;
  const uint32_t bits = (uint32_t)(hi & 0x80000000) | ((uint32_t)ex << 23) | (__funnelshift_l((uint32_t)lo, (uint32_t)hi, 3) & 0x007fffffu);
  return ex > 0 ? __uint_as_float(bits) : 0.f;
}
// The fp32 number as fp64, without the conversion unit (8 clocks a warp); 0 becomes 6e-39.
__device__ __forceinline__ double to_double(float x) {
  const uint32_t b = __float_as_uint(x);
  return __hiloint2double((int)((b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + 0x38000000u)), (int)(b << 29));
}

// Are columns with squared lengths al, be and product ga to be rotated?  floor2: squared length of a null column.  The one rule for
// whether a visit has anything to rotate and whether a pair is: what the first finds the second has to rotate, or every
// sweep would find it again.
__device__ __forceinline__ bool to_rotate(double al, double be, double ga, double floor2) {
  return ga * ga > kOrthTol * kOrthTol * (al * be) && fmin(al, be) > floor2;
}

// The rotation (c, s) that makes columns p, q orthogonal (the smaller of the two angles phi, tan 2 phi = 2 ga / (be - al)); (1, 0)
// when it is not needed.  The angle comes from fp32 arithmetic (what it misses, 1e-7 of the product, the next visit sees);
// then (c, s) is brought to unit length in fp64, 1 / sqrt(1 + x) = 1 - x / 2 + 3 x^2 / 8 with x below 1e-6, so the
// rotation is orthonormal in fp64 whatever its angle.  This is the chain of an inner round: seven dependent fp64 operations and
// four of the 2 x 2 update, no fp64 division or root.
__device__ __forceinline__ void rotation(double al, double be, double ga, double floor2, double& c, double& s) {
  const double d = be - al;
  const int e = max((__double2hiint(d) >> 20) & 0x7ff, (__double2hiint(ga) >> 20) & 0x7ff);
  const float df = fabsf(to_float_scaled(d, e)), gf = to_float_scaled(ga, e), g2 = gf + gf;
  const float ir = rsqrt_approx(fmaf(df, df, g2 * g2));            // 1 / R
  const float c2 = fmaf(0.5f * df, ir, 0.5f);                      // cos^2 phi
  const float ic = rsqrt_approx(c2);
  const double cd = to_double(c2 * ic), sd = to_double((d < 0.0 ? -gf : gf) * ir * ic);
  const double x = fma(cd, cd, fma(sd, sd, -1.0)), y = fma(0.375, x, -0.5);
  const bool rot = to_rotate(al, be, ga, floor2);
  c = rot ? fma(cd * x, y, cd) : 1.0;
  s = rot ? fma(sd * x, y, sd) : 0.0;
}

// ---- Phi = R^T R (R upper triangular), in place in W ----
// The rows of R are columns of a factor of Phi as the rows of Phi V are of Phi Phi^T = Phi^2: rotated until they are
// orthogonal they are the eigenvectors too, with lengths sqrt(lambda).  They start closer to orthogonal (the factor's Gram
// matrix R R^T is one step of the LR iteration on from Phi, and its condition is that of Phi, not of Phi^2).
constexpr int kRLd = EB + 1;
constexpr int kOwn = 8;               // block rows of a CTA updated per staging where rows come in chunks
constexpr double kPivot = 1e-12;      // of max_i Phi_ii: with a pivot below it, Phi is taken as it is

struct Factor {
  double* R;         // [2][16][kRLd] triangular factors of the diagonal blocks, then [2][16] reciprocals of their diagonals
  double* P;         // [kOwn][16][kRLd] blocks of the current block row of R
};

// x <- R_kk^-T x, a column of the block row
__device__ __forceinline__ void solve_column(double (&x)[EB], const double* R, const double* inv) {
#pragma unroll
  for (int j = 0; j < EB; ++j) {
    x[j] *= inv[j];
#pragma unroll
    for (int p = j + 1; p < EB; ++p) x[p] = fma(-R[j * kRLd + p], x[j], x[p]);
  }
}
// columns [c0, c1) of the staged block row
__device__ __forceinline__ void solve_staged(double* row, int stride, int c0, int c1, const double* R, const double* inv) {
  for (int c = c0 + (int)threadIdx.x; c < c1; c += ET) {
    double x[EB];
#pragma unroll
    for (int p = 0; p < EB; ++p) x[p] = row[p * stride + c];
    solve_column(x, R, inv);
#pragma unroll
    for (int p = 0; p < EB; ++p) row[p * stride + c] = x[p];
  }
}
// The 16 x 16 diagonal block k <- its triangular factor, one warp, a column per lane; false with a pivot that is too small.
__device__ __forceinline__ bool factor_diagonal(const EvdLayer& L, int k, double pivot, double* R, double* inv) {
  const int lane = threadIdx.x & 31, c = lane & (EB - 1), M = L.M, ld = evd_ld(M);
  double a[EB];
#pragma unroll
  for (int r = 0; r < EB; ++r)
    a[r] = (k * EB + r < M && k * EB + c < M) ? __ldcg(L.W + (int64_t)(k * EB + r) * ld + k * EB + c) : 0.0;
  bool ok = true;
#pragma unroll
  for (int j = 0; j < EB; ++j) {
    double d = __shfl_sync(0xffffffffu, a[j], j);
    if (k * EB + j >= M) d = 1.0;
    else ok = ok && d > pivot && d <= 1e300;
    const double q = ok ? rsqrt(d) : 1.0;
    a[j] *= q;
#pragma unroll
    for (int i = j + 1; i < EB; ++i) a[i] = fma(-__shfl_sync(0xffffffffu, a[j], i), a[j], a[i]);
    if (lane < EB) R[j * kRLd + c] = c >= j ? a[j] : 0.0;
    if (lane == 0) inv[j] = q;
  }
  return ok;
}
// W_i -= R_ki^T (block row k of R), columns [c0, c1) of the layer; row: entry c0 of the first staged row; P: R_ki, prow apart.
__device__ __forceinline__ void update_block_row(const EvdLayer& L, int i, int c0, int c1, const double* row, int stride,
                                                 const double* P, int prow) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, M = L.M, ld = evd_ld(M);
  double af[2][4];
#pragma unroll
  for (int t = 0; t < 2; ++t)
#pragma unroll
    for (int q = 0; q < 4; ++q) af[t][q] = -P[(4 * q + (lane & 3)) * prow + 8 * t + (lane >> 2)];
  const int r0 = i * EB + (lane >> 2);
#pragma unroll 2
  for (int c = max(c0, i * EB) + 8 * warp; c < c1; c += 8 * EW) {
    double2 d[2];
#pragma unroll
    for (int t = 0; t < 2; ++t)
      d[t] = r0 + 8 * t < M ? __ldcg(reinterpret_cast<const double2*>(L.W + (int64_t)(r0 + 8 * t) * ld + c + 2 * (lane & 3)))
                            : make_double2(0.0, 0.0);
    double acc[2][2] = {{d[0].x, d[0].y}, {d[1].x, d[1].y}};
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const double b = row[(4 * q + (lane & 3)) * stride + c - c0 + (lane >> 2)];
      mma_f64(acc[0], af[0][q], b);
      mma_f64(acc[1], af[1][q], b);
    }
#pragma unroll
    for (int t = 0; t < 2; ++t)
      if (r0 + 8 * t < M)
        __stcg(reinterpret_cast<double2*>(L.W + (int64_t)(r0 + 8 * t) * ld + c + 2 * (lane & 3)), make_double2(acc[t][0], acc[t][1]));
  }
}
// columns [c0, c1) of the finished rows of block k: zeros, the diagonal factor, the solved columns (row: entry c0)
__device__ __forceinline__ void write_block_row(const EvdLayer& L, int k, int c0, int c1, const double* row, int stride, const double* R) {
  const int ld = evd_ld(L.M), half = (c1 - c0) >> 1;
  for (int i = threadIdx.x; i < EB * half; i += ET) {
    const int r = i / half, c = c0 + 2 * (i - r * half);
    if (k * EB + r >= L.M) continue;
    double2 v = make_double2(0.0, 0.0);
    if (c >= (k + 1) * EB) v = make_double2(row[r * stride + c - c0], row[r * stride + c - c0 + 1]);
    else if (c >= k * EB) v = make_double2(R[r * kRLd + c - k * EB], R[r * kRLd + c - k * EB + 1]);
    __stcg(reinterpret_cast<double2*>(L.W + (int64_t)(k * EB + r) * ld + c), v);
  }
}

// Block row k of a step is finished by every CTA for itself (its 16 x 16 factor, then a column per thread) and subtracted
// from the block rows i > k with i mod n = sub, which are the CTA's own; one barrier a step.  Its owner writes it one step later,
// when nobody reads the unfinished row any more.  All CTAs see the same pivots and give up at the same step.
// 1: done; 0: not positive definite (W is spoilt); -1: a wait gave up.
__device__ __noinline__ int evd_factor(const EvdLayer& L, int sub, double pivot, int nk, int stride, const Factor& f, uint32_t bar,
                                       uint32_t& parity, int& bidx, int* s_abort, int* s_last) {
  __shared__ int s_bad;
  const int M = L.M, ld = evd_ld(M), nblk = (M + EB - 1) / EB, tid = threadIdx.x;
  const bool whole = ld <= nk;
  if (tid == 0) s_bad = 0;
  __syncthreads();
  for (int k = 0; k <= nblk; ++k) {
    double* row = esm + (k & 1) * EB * stride;
    double* R = f.R + (k & 1) * EB * kRLd;
    double* inv = f.R + 2 * EB * kRLd + (k & 1) * EB;
    const int i0 = k + 1 + (sub + L.n - (k + 1) % L.n) % L.n;      // my first block row after k
    const bool any = i0 < nblk, owner = k < nblk && k % L.n == sub;
    const int c0 = k * EB;
    if (whole && (any || owner)) stage_issue(L, row, k, k, EB, c0, ld - c0, stride, bar);
    if (k < nblk && tid >= 32 && tid < 64) {
      const bool ok = factor_diagonal(L, k, pivot, R, inv);
      if (!ok && tid == 32) s_bad = 1;
    }
    if (whole && (any || owner)) {
      if (!stage_wait(bar, parity)) { evd_give_up(L); return -1; }
      parity ^= 1;
    } else {
      __syncthreads();
    }
    if (s_bad) return evd_barrier(L, sub, ++bidx, 0, s_abort, s_last) ? 0 : -1;
    if (whole) {
      if (any || owner) solve_staged(row, stride, owner ? EB : (i0 - k) * EB, ld - c0, R, inv);
      __syncthreads();
      for (int i = i0; i < nblk; i += L.n) update_block_row(L, i, c0, ld, row, stride, row + (i - k) * EB, stride);
    } else {
      for (int i = i0; i < nblk; i += kOwn * L.n) {
        const int g = tid >> 4, r = tid & (EB - 1), ig = i + g * L.n;
        if (g < kOwn && ig < nblk) {
          double x[EB];
#pragma unroll
          for (int p = 0; p < EB; ++p) x[p] = ig * EB + r < M ? __ldcg(L.W + (int64_t)(c0 + p) * ld + ig * EB + r) : 0.0;
          solve_column(x, R, inv);
#pragma unroll
          for (int p = 0; p < EB; ++p) f.P[(g * EB + p) * kRLd + r] = x[p];
        }
        for (int c = i * EB; c < ld; c += nk) {
          __syncthreads();                                         // P is written, the chunk before has been read
          stage_issue(L, row, k, k, EB, c, nk, stride, bar);
          if (!stage_wait(bar, parity)) { evd_give_up(L); return -1; }
          parity ^= 1;
          solve_staged(row, stride, 0, nk, R, inv);
          __syncthreads();
          for (int h = 0; h < kOwn && i + h * L.n < nblk; ++h)
            update_block_row(L, i + h * L.n, c, min(c + nk, ld), row, stride, f.P + h * EB * kRLd, kRLd);
        }
        __syncthreads();
      }
    }
    // the block row before, when it is mine: nobody reads it as it was any more
    if (k > 0 && (k - 1) % L.n == sub) {
      double* row1 = esm + ((k - 1) & 1) * EB * stride;
      double* R1 = f.R + ((k - 1) & 1) * EB * kRLd;
      const double* inv1 = f.R + 2 * EB * kRLd + ((k - 1) & 1) * EB;
      if (whole) {
        write_block_row(L, k - 1, 0, c0 - EB, row1, stride, R1);
        write_block_row(L, k - 1, c0 - EB, ld, row1, stride, R1);
      } else {
        for (int c = 0; c < ld; c += nk) {
          if (c + nk > c0) {
            __syncthreads();
            stage_issue(L, row1, k - 1, k - 1, EB, c, nk, stride, bar);
            if (!stage_wait(bar, parity)) { evd_give_up(L); return -1; }
            parity ^= 1;
            solve_staged(row1, stride, max(0, c0 - c), nk, R1, inv1);
            __syncthreads();
          }
          write_block_row(L, k - 1, c, min(c + nk, ld), row1, stride, R1);
        }
      }
    }
    if (!evd_barrier(L, sub, ++bidx, 0, s_abort, s_last)) return -1;
  }
  return 1;
}

// W = Phi, padded with zeros to whole rows of ld
__device__ __forceinline__ void evd_load(const EvdLayer& L, int sub) {
  const int M = L.M, ld = evd_ld(M);
  for (int64_t i = (int64_t)sub * ET + threadIdx.x; i < (int64_t)M * ld; i += (int64_t)L.n * ET) {
    const int r = (int)(i / ld), c = (int)(i - (int64_t)r * ld);
    __stcg(L.W + i, c < M ? (double)L.A[(int64_t)r * M + c] : 0.0);
  }
}

// The 2 x 2 block of products of pairs a (rows i) and b (columns), pair a's rotation in lane a, b's (cb, sb): both applied.
// Where two entries hold one product, both are written, except in cross visits, where a pair's first column is always of the
// first block: an entry is then met again in the same place, if products of the two blocks are always taken from the upper
// right quarter (only those of opposite pairs, a = b + 8, of the second block change places: mirror).
struct Block2 { int i[2]; double g[2][2]; };
template <bool CROSS>
__device__ __forceinline__ Block2 load_block(const double* src, int a, int q, int jp, int jq) {
  Block2 r;
  evd_players<CROSS>(a, q, r.i[0], r.i[1]);
  r.g[0][0] = src[r.i[0] * kGLd + jp]; r.g[0][1] = src[r.i[0] * kGLd + jq];
  r.g[1][0] = CROSS ? src[jp * kGLd + r.i[1]] : src[r.i[1] * kGLd + jp];
  r.g[1][1] = src[r.i[1] * kGLd + jq];
  return r;
}
template <bool CROSS>
__device__ __forceinline__ void rotate_block(double* dst, const Block2& r, int a, int jp, int jq, double cb, double sb, bool mine,
                                             bool mirror) {
  const double ca = __shfl_sync(0xffffffffu, cb, a), sa = __shfl_sync(0xffffffffu, sb, a);
  const double h00 = cb * r.g[0][0] - sb * r.g[0][1], h01 = sb * r.g[0][0] + cb * r.g[0][1];
  const double h10 = cb * r.g[1][0] - sb * r.g[1][1], h11 = sb * r.g[1][0] + cb * r.g[1][1];
  const double v00 = ca * h00 - sa * h10, v01 = ca * h01 - sa * h11;
  const double v10 = sa * h00 + ca * h10, v11 = sa * h01 + ca * h11;
  if (!mine) return;
  dst[r.i[0] * kGLd + jp] = v00; dst[r.i[0] * kGLd + jq] = v01;
  dst[jp * kGLd + r.i[1]] = v10; dst[r.i[1] * kGLd + jq] = v11;
  if (!CROSS || mirror) dst[jq * kGLd + r.i[1]] = v11;
  if (CROSS) return;
  dst[jp * kGLd + r.i[0]] = v00; dst[jq * kGLd + r.i[0]] = v01; dst[r.i[1] * kGLd + jp] = v10;
}

// A visit to the block pair (I, J).  CROSS: rotations between columns of different blocks only, with the products within a
// block taken as zero (all but the squared lengths): they were rotated in the sweep's first round, and what they have become
// since enters only at second order.  That is 4 of 10 blocks of the Gram matrix and 16 of 31 inner rounds, for half a sweep
// more.  1: rotated; 0: nothing to rotate; -1: a wait gave up.
template <bool CROSS>
__device__ __forceinline__ int visit(const EvdLayer& L, int I, int J, int nk, int chunks, int stride, double floor2, double2 (*rots)[EB],
                                     uint32_t bar, uint32_t& parity) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, M = L.M, ld = evd_ld(M);
  double* part = esm + EP * stride;                               // kPartDoubles
  double* G0 = part + kPartDoubles;
  double* U = part;                                               // these two reuse the partial blocks
  double* G1 = part + EP * kULd;
  // ---- G = (rows)(rows)^T: each warp a sixteenth of the entries, all blocks that are wanted ----
  constexpr int NB = CROSS ? 4 : kTri;
  double acc[NB][2], n2[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
  for (int b = 0; b < NB; ++b) acc[b][0] = acc[b][1] = 0.0;
  for (int ch = 0; ch < chunks; ++ch) {
    if (ch) __syncthreads();                                // the chunk before has been read
    if (!stage_rows(L, I, J, ch * kChunk, nk, stride, bar, parity)) return -1;
    parity ^= 1;
    const double* w = esm + (lane >> 2) * stride + (lane & 3);
#pragma unroll 2
    for (int st = warp; st < nk / 4; st += EW) {
      double f[4];
#pragma unroll
      for (int b = 0; b < 4; ++b) f[b] = w[8 * b * stride + 4 * st];
      if (CROSS) {
#pragma unroll
        for (int b = 0; b < 4; ++b) {
          mma_f64(acc[b], f[b >> 1], f[2 + (b & 1)]);
          n2[b] = fma(f[b], f[b], n2[b]);
        }
      } else {
        int t = 0;
#pragma unroll
        for (int b = 0; b < 4; ++b)
#pragma unroll
          for (int c = b; c < 4; ++c) mma_f64(acc[t++], f[b], f[c]);
      }
    }
  }
  if (CROSS) {
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      *reinterpret_cast<double2*>(part + warp * kCross + b * 64 + 2 * lane) = make_double2(acc[b][0], acc[b][1]);
      n2[b] += __shfl_xor_sync(0xffffffffu, n2[b], 1);
      n2[b] += __shfl_xor_sync(0xffffffffu, n2[b], 2);
      if ((lane & 3) == 0) part[warp * kCross + 256 + 8 * b + (lane >> 2)] = n2[b];
    }
    __syncthreads();
    if (tid < kCross) {
      double x = 0.0, y = 0.0;
#pragma unroll
      for (int w = 0; w < EW; w += 2) { x += part[w * kCross + tid]; y += part[(w + 1) * kCross + tid]; }
      x += y;
      const int b = tid >> 6, e = tid & 63;
      if (b < 4) {
        const int gi = 8 * (b >> 1) + (e >> 3), gj = EB + 8 * (b & 1) + (e & 7);
        G0[gi * kGLd + gj] = x; G0[gj * kGLd + gi] = x;
      } else {
        G0[e * kGLd + e] = x;
      }
    }
    const int p = tid >> 4, q = (p & EB) + (tid & (EB - 1));         // ET = 32 x 16: a thread for each entry within the blocks
    if (p != q) G0[p * kGLd + q] = 0.0;
  } else {
    // the second half of the warps hand their sums to the first half, which add to them
    if (warp >= EW / 2) {
#pragma unroll
      for (int b = 0; b < NB; ++b)
        *reinterpret_cast<double2*>(part + ((warp - EW / 2) * kTri + b) * 64 + 2 * lane) = make_double2(acc[b][0], acc[b][1]);
    }
    __syncthreads();
    if (warp < EW / 2) {
#pragma unroll
      for (int b = 0; b < NB; ++b) {
        double2* q = reinterpret_cast<double2*>(part + (warp * kTri + b) * 64 + 2 * lane);
        const double2 o = *q;
        *q = make_double2(acc[b][0] + o.x, acc[b][1] + o.y);
      }
    }
    __syncthreads();
    for (int i = tid; i < kTri * 64; i += ET) {
      double x = 0.0;
#pragma unroll
      for (int w = 0; w < EW / 2; ++w) x += part[w * kTri * 64 + i];
      const int b = i >> 6, e = i & 63;
      const int rb = b < 4 ? 0 : (b < 7 ? 1 : (b < 9 ? 2 : 3)), cb = b - (b < 4 ? 0 : (b < 7 ? 3 : (b < 9 ? 5 : 6)));
      const int gi = 8 * rb + (e >> 3), gj = 8 * cb + (e & 7);
      if (rb != cb || gj >= gi) { G0[gi * kGLd + gj] = x; G0[gj * kGLd + gi] = x; }
    }
  }
  __syncthreads();
  // ---- anything to rotate? ----
  bool act = false;
  for (int i = tid; i < EP * EP; i += ET) {
    const int p = i >> 5, q = i & 31;
    U[p * kULd + q] = p == q ? 1.0 : 0.0;
    act |= p < q && to_rotate(G0[p * kGLd + p], G0[q * kGLd + q], G0[p * kGLd + q], floor2);
  }
  if (!__syncthreads_or(act)) return 0;
  // ---- one sweep of 2 x 2 rotations on G.  A half-warp of the first five warps owns the 2 x 2 blocks of pairs (b + k, b), b its
  //      lane: k = 0 ... 7 and, for half of the b, 8.  Six more warps apply each round's rotations to U one round later, off
  //      the chain (not warp 8: two of the five share its scheduler). ----
  if (warp < 12 && warp != 8) {
    const int pb = tid & 15;
    constexpr int kRounds = CROSS ? EB : EP - 1;
    if (warp < 5) {
      const int k = min(tid >> 4, 8), pa = (pb + k) & 15;
      const bool mine = k < 8 || tid < 8 * EB + 8;
      double* src = G0;
      double* dst = G1;
      int jp, jq;
      evd_players<CROSS>(pb, 0, jp, jq);
      for (int q = 0; q <= kRounds; ++q) {
        if (q < kRounds) {
          const double al = src[jp * kGLd + jp], be = src[jq * kGLd + jq], ga = src[jp * kGLd + jq];
          const Block2 g = load_block<CROSS>(src, pa, q, jp, jq);
          double cb, sb;
          rotation(al, be, ga, floor2, cb, sb);
          rotate_block<CROSS>(dst, g, pa, jp, jq, cb, sb, mine, k == 8);
          if (tid >= 9 * EB) rots[q & 1][pb] = make_double2(cb, sb);
          double* z = src; src = dst; dst = z;
          evd_players<CROSS>(pb, q + 1, jp, jq);
        }
        asm volatile("bar.sync 1, 352;" ::: "memory");
      }
    } else {
      const int row0 = 2 * (warp - (warp > 8 ? 6 : 5)) + (lane >> 4);    // and 12, 24 more
      for (int q = 0; q <= kRounds; ++q) {
        if (q > 0) {
          int jp, jq;
          evd_players<CROSS>(pb, q - 1, jp, jq);
          const double2 r = rots[(q - 1) & 1][pb];
#pragma unroll
          for (int i = 0; i < 3; ++i) {
            double* u = U + (row0 + 12 * i) * kULd;
            if (i == 2 && row0 >= 8) break;
            const double x0 = u[jp], x1 = u[jq];
            u[jp] = r.x * x0 - r.y * x1;
            u[jq] = r.y * x0 + r.x * x1;
          }
        }
        asm volatile("bar.sync 1, 352;" ::: "memory");
      }
    }
  }
  __syncthreads();
  // ---- rows <- U^T rows, in place chunk by chunk (a single chunk is still staged) ----
  // the first half of the warps computes the first 16 rows, the second half the others
  double uf[2][8];
  const int half = warp / (EW / 2), wcol = warp - half * (EW / 2);
#pragma unroll
  for (int cb = 0; cb < 2; ++cb)
#pragma unroll
    for (int kb = 0; kb < 8; ++kb) uf[cb][kb] = U[(4 * kb + (lane & 3)) * kULd + 16 * half + 8 * cb + (lane >> 2)];
  for (int ch = 0; ch < chunks; ++ch) {
    if (chunks > 1) {
      __syncthreads();
      if (!stage_rows(L, I, J, ch * kChunk, nk, stride, bar, parity)) return -1;
      parity ^= 1;
    }
#pragma unroll 3
    for (int b = wcol; b < nk / 8; b += EW / 2) {
      double bf[8];
#pragma unroll
      for (int kb = 0; kb < 8; ++kb) bf[kb] = esm[(4 * kb + (lane & 3)) * stride + 8 * b + (lane >> 2)];
      const int col = ch * kChunk + 8 * b + 2 * (lane & 3);
#pragma unroll
      for (int cb = 0; cb < 2; ++cb) {
        double d[2] = {0.0, 0.0};
#pragma unroll
        for (int kb = 0; kb < 8; ++kb) mma_f64(d, uf[cb][kb], bf[kb]);
        const int row = pair_row(I, J, 16 * half + 8 * cb + (lane >> 2));
        if (row < M && col < ld) __stcg(reinterpret_cast<double2*>(L.W + (int64_t)row * ld + col), make_double2(d[0], d[1]));
      }
    }
  }
  return 1;
}

// the words of every layer, a CTA each
__global__ void __launch_bounds__(kWords) evd_clear_kernel(const __grid_constant__ EvdArgs a) {
  dep_sync();
  a.l[blockIdx.x].words[threadIdx.x] = 0;
}

__global__ void __launch_bounds__(ET, 1) jacobi_kernel(const __grid_constant__ EvdArgs a) {
  __shared__ int s_abort, s_last;
  __shared__ __align__(8) uint64_t s_bar;
  __shared__ double2 rots[2][EB];
  const int tid = threadIdx.x;
  int li = -1;
#pragma unroll 1
  for (int i = 0; i < a.nl; ++i)
    if ((int)blockIdx.x >= a.l[i].cta0 && (int)blockIdx.x < a.l[i].cta0 + a.l[i].n) li = i;
  if (li < 0) return;
  const EvdLayer L = a.l[li];
  const int M = L.M, ld = evd_ld(M), sub = (int)blockIdx.x - L.cta0;
  const uint32_t bar = sm100::smem_u32(&s_bar);
  uint32_t parity = 0;
  if (tid == 0) {
    s_abort = 0;
    sm100::mbar_init(bar, 1);
    sm100::mbar_fence_init();
  }
  float dmax = 0.f;
  for (int i = tid; i < M; i += ET) dmax = fmaxf(dmax, fabsf(L.A[(int64_t)i * M + i]));
  const double top = evd_block_max(dmax);
  evd_load(L, sub);
  const int chunks = (ld + kChunk - 1) / kChunk;
  const int nk = chunks == 1 ? ld : kChunk;                       // entries per chunk
  const int stride = evd_stride(nk);
  double* part = esm + EP * stride;                               // kPartDoubles
  int bidx = 0;
  if (!evd_barrier(L, sub, ++bidx, 0, &s_abort, &s_last)) return;
  const Factor f{part, part + 2 * EB * (kRLd + 1)};
  const int fac = evd_factor(L, sub, kPivot * top, nk, stride, f, bar, parity, bidx, &s_abort, &s_last);
  if (fac < 0) return;
  if (fac == 0) {
    evd_load(L, sub);
    if (!evd_barrier(L, sub, ++bidx, 0, &s_abort, &s_last)) return;
  } else if (sub == 0 && tid == 0) {
    L.words[0] = 1;
  }
  // squared length of a column that is rounding
  const double floor2 = fac ? kFloor * top : kFloor * top * (kFloor * top);
  const int np = L.nb / 2, n1 = L.nb - 1;
  // rounds until a sweep's worth of them in a row has rotated nothing
  int last = 0;
  for (int round = 1, r = 0; round <= kMaxSweeps * n1; ++round, r = r + 1 == n1 ? 0 : r + 1) {
    for (int k = sub; k < np; k += L.n) {
      int I, J;
      if (k == 0) { I = n1; J = r; }
      else { I = (r + k) % n1; J = (r - k + n1) % n1; }
      if (I > J) { const int x = I; I = J; J = x; }
      if (I * EB >= M) continue;                                  // both blocks past the matrix
      const int v = r == 0 ? visit<false>(L, I, J, nk, chunks, stride, floor2, rots, bar, parity)
                           : visit<true>(L, I, J, nk, chunks, stride, floor2, rots, bar, parity);
      if (v < 0) { evd_give_up(L); return; }
      if (v > 0) last = round;
      __syncthreads();                                            // the staged rows are free for the next pair
    }
    if (!evd_barrier(L, sub, ++bidx, last, &s_abort, &s_last)) return;
    if (round - s_last >= n1) break;                              // every pair is orthogonal
  }
}

struct FinishArgs {
  EvdLayer l[FW_MAX_GROUP];
  double* lam[FW_MAX_GROUP];       // M eigenvalues, in the order of the rows of W
  double* dvec[FW_MAX_GROUP];      // 3 M weights of the rows' outer products, then kBase values (null: eigenvalues only)
  float* lam_sorted[FW_MAX_GROUP]; // optional output: eigenvalues in decreasing order
  float* kappa[FW_MAX_GROUP];      // optional output: rank estimate / M
  float eps[FW_MAX_GROUP];
  int32_t block0[FW_MAX_GROUP + 1];   // first CTA of each layer in the grid of norm_kernel (a warp per column)
  int32_t nl;
  float g_max;                     // <= 0: g = 1 / max(lambda, eps) (Eq. 10); > 0: the gains of Eq. 34
};
constexpr int kBase = 4;           // weights of the identity in the three outputs; 1.0 when Phi = 0

// lambda_m = |w_m|, with the sign of the Rayleigh quotient (one row of Phi suffices: w_m is parallel to v_m) where the
// eigenvectors are wanted; a warp per column
__global__ void __launch_bounds__(256) norm_kernel(const __grid_constant__ FinishArgs a) {
  dep_sync();
  int li = 0;
#pragma unroll 1
  for (int i = 1; i < a.nl; ++i)
    if ((int)blockIdx.x >= a.block0[i]) li = i;
  const EvdLayer L = a.l[li];
  const int M = L.M, lane = threadIdx.x & 31;
  const int m = ((int)blockIdx.x - a.block0[li]) * 8 + (threadIdx.x >> 5);
  if (m >= M) return;
  const double* w = L.W + (int64_t)m * evd_ld(M);
  double acc = 0.0, best = -1.0;
  int bi = 0;
  for (int i = lane; i < M; i += 32) {
    const double x = w[i];
    acc = fma(x, x, acc);
    if (fabs(x) > best) { best = fabs(x); bi = i; }
  }
  acc = warp_sum(acc);
  const bool factored = L.words[0] != 0;                         // lambda_m = |w_m|^2 > 0
  if (!factored) acc = sqrt(acc);
  if (a.dvec[li] && !factored) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const double xo = __shfl_xor_sync(0xffffffffu, best, o);
      const int io = __shfl_xor_sync(0xffffffffu, bi, o);
      if (xo > best || (xo == best && io < bi)) { best = xo; bi = io; }
    }
    double dot = 0.0;
    for (int i = lane; i < M; i += 32) dot = fma((double)L.A[(int64_t)bi * M + i], w[i], dot);
    dot = warp_sum(dot);
    if (dot * w[bi] < 0.0) acc = -acc;
  }
  if (lane == 0) a.lam[li][m] = acc;
}

// sum over the block in a fixed order
__device__ double block_sum_d(double x, double* red) {
  x = warp_sum(x);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = x;
  __syncthreads();
  x = threadIdx.x < 32 ? red[threadIdx.x] : 0.0;
  if (threadIdx.x < 32) {
    x = warp_sum(x);
    if (threadIdx.x == 0) red[0] = x;
  }
  __syncthreads();
  return red[0];
}

// One CTA per layer: ranks of the eigenvalues, the rank estimate (Eq. 32 read as exp(-sum lbar log lbar)) and the gains.
// The sums decide an integer (the rank): their order does not depend on the launch.
__global__ void __launch_bounds__(1024) evd_finish_kernel(const __grid_constant__ FinishArgs a) {
  dep_sync();
  __shared__ double red[32];
  const EvdLayer L = a.l[blockIdx.x];
  const int M = L.M;
  const double* lam = a.lam[blockIdx.x];
  const bool factored = L.words[0] != 0;
  double x = 0.0;
  for (int m = threadIdx.x; m < M; m += 1024) x += fmax(lam[m], 0.0);
  const double S = block_sum_d(x, red);
  x = 0.0;
  for (int m = threadIdx.x; m < M; m += 1024) {
    const double lb = S > 0.0 ? fmax(lam[m], 0.0) / S : 0.0;
    if (lb > 0.0) x -= lb * log(lb);
  }
  const double ms_hat = exp(block_sum_d(x, red));
  const int Ms = min(max((int)rint(ms_hat), 1), M);
  if (threadIdx.x == 0 && a.kappa[blockIdx.x]) *a.kappa[blockIdx.x] = (float)(ms_hat / (double)M);
  double* dv = a.dvec[blockIdx.x];
  const double eps = (double)a.eps[blockIdx.x], g_max = (double)a.g_max;
  auto gain = [&](double lm, int rank) {
    if (a.g_max <= 0.f) return 1.0 / fmax(lm, eps);                                        // Eq. 10
    const double lb = S > 0.0 ? fmax(lm, 0.0) / S : 0.0;
    return rank < Ms ? fmin(1.0 / fmax((double)M * lb, 1e-300), g_max) : 1.0;              // Eq. 34
  };
  float top = 0.f;
  for (int m = threadIdx.x; m < M; m += 1024) top = fmaxf(top, (float)fabs(lam[m]));
  const double null = kNull * evd_block_max(top);
  int nulls = 0;
  for (int m = threadIdx.x; m < M; m += 1024) nulls += fabs(lam[m]) <= null ? 1 : 0;
  nulls = (int)(block_sum_d((double)nulls, red) + 0.5);
  // Null columns span what the others leave: with their common gain g0 they contribute g0 (I - sum v v^T).  When Phi = 0
  // every column is its own unit vector.
  const bool zero = nulls == M, some = nulls > 0 && !zero;
  const double g0 = gain(0.0, M - 1), b0 = some ? sqrt(g0) : 0.0, b1 = some ? g0 : 0.0;
  for (int m = threadIdx.x; m < M; m += 1024) {
    const double lm = lam[m];
    int rank = 0;                                   // position of lambda_m in decreasing order
#pragma unroll 8
    for (int j = 0; j < M; ++j) {
      const double lj = lam[j];
      rank += (lj > lm || (lj == lm && j < m)) ? 1 : 0;
    }
    if (a.lam_sorted[blockIdx.x]) a.lam_sorted[blockIdx.x][rank] = (float)lm;
    if (dv) {
      const double g = gain(lm, rank);
      // rows of W are lambda_m v_m, or sqrt(lambda_m) v_m where Phi was factored
      const double n2 = zero ? 1.0 : (fabs(lm) <= null ? 0.0 : 1.0 / (factored ? lm : lm * lm));
      dv[m] = (sqrt(g) - b0) * n2;
      dv[M + m] = (g - b1) * n2;
      dv[2 * M + m] = g * lm * n2;
    }
  }
  if (dv && threadIdx.x == 0) { dv[3 * M] = b0; dv[3 * M + 1] = b1; dv[3 * M + 2] = 0.0; dv[3 * M + 3] = zero ? 1.0 : 0.0; }
}

struct VdvArgs {
  EvdLayer l[FW_MAX_GROUP];
  const double* dvec[FW_MAX_GROUP];
  float* T[FW_MAX_GROUP];
  float* Q[FW_MAX_GROUP];
  float* Y[FW_MAX_GROUP];
  int32_t tile0[FW_MAX_GROUP + 1];   // flat grid over the upper-triangle 64 x 64 tiles of all layers
  int32_t nl;
};

// out_ij = sum_m d_m w_mi w_mj for the three weight vectors at once, on the fp64 tensor cores; a CTA computes a tile of
// the upper triangle and writes its mirror image too, so the outputs are exactly symmetric.  A warp takes 16 x 32.
// Bound by the fp64 tensor cores (24 products of 8 x 8 x 4 a warp and step); the next two slices of 16 rows are on their way
// meanwhile.  15 layers of the ResNet-20-shaped set: 202 us, 290 with a slice loaded between two barriers, 109 at the tensor cores' rate.
constexpr int VT = 64, VK = 16, kVs = VT + 4, VS = 3;
struct VdvStage { double a[VK][kVs], b[VK][kVs], d[3][VK]; };
__global__ void __launch_bounds__(256) vdv_kernel(const __grid_constant__ VdvArgs a) {
  dep_sync();
  int li = 0;
#pragma unroll 1
  for (int i = 1; i < a.nl; ++i)
    if ((int)blockIdx.x >= a.tile0[i]) li = i;
  const EvdLayer L = a.l[li];
  const int M = L.M, ld = evd_ld(M);
  int bi, bj;
  tri_decode((int)blockIdx.x - a.tile0[li], (M + VT - 1) / VT, bi, bj);
  VdvStage* st = reinterpret_cast<VdvStage*>(esm);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int wi = (warp >> 1) * 16, wj = (warp & 1) * 32;         // 4 x 2 warps
  const double* dv = a.dvec[li];
  double acc[3][2][4][2];
#pragma unroll
  for (int o = 0; o < 3; ++o)
#pragma unroll
    for (int r = 0; r < 2; ++r)
#pragma unroll
      for (int c = 0; c < 4; ++c) acc[o][r][c][0] = acc[o][r][c][1] = 0.0;
  const bool unit = dv[3 * M + 3] != 0.0;                          // Phi = 0: unit vectors
  const int slices = unit ? 0 : (M + VK - 1) / VK;
  // slice s into its stage; rows and columns past the matrix as zeros (an entry past M and below ld is a zero of W)
  auto load = [&](int s) {
    if (s < slices) {
      VdvStage& d = st[s % VS];
      const int m0 = s * VK;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int i = tid + 256 * h, mm = i >> 5, c = 2 * (i & 31);
        const double* w = L.W + (int64_t)min(m0 + mm, M - 1) * ld;
        const int ca = bi * VT + c, cb = bj * VT + c;
        const int na = m0 + mm < M && ca < ld ? 16 : 0, nb = m0 + mm < M && cb < ld ? 16 : 0;
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(sm100::smem_u32(&d.a[mm][c])), "l"(w + min(ca, ld - 2)), "r"(na) : "memory");
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(sm100::smem_u32(&d.b[mm][c])), "l"(w + min(cb, ld - 2)), "r"(nb) : "memory");
      }
      if (tid < 3 * VK) {
        const int o = tid / VK, mm = tid - o * VK, n = m0 + mm < M ? 8 : 0;
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(sm100::smem_u32(&d.d[o][mm])), "l"(dv + o * M + min(m0 + mm, M - 1)), "r"(n) : "memory");
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  load(0);
  load(1);
  for (int s = 0; s < slices; ++s) {
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    __syncthreads();                                               // slice s is here, slice s - 1 has been used
    load(s + 2);
    const VdvStage& t = st[s % VS];
#pragma unroll
    for (int k = 0; k < VK / 4; ++k) {
      const int mm = 4 * k + (lane & 3);
      double af[2], bf[4];
#pragma unroll
      for (int r = 0; r < 2; ++r) af[r] = t.a[mm][wi + 8 * r + (lane >> 2)];
#pragma unroll
      for (int c = 0; c < 4; ++c) bf[c] = t.b[mm][wj + 8 * c + (lane >> 2)];
#pragma unroll
      for (int o = 0; o < 3; ++o) {
        const double d = t.d[o][mm];
#pragma unroll
        for (int r = 0; r < 2; ++r) {
          const double ad = af[r] * d;
#pragma unroll
          for (int c = 0; c < 4; ++c) mma_f64(acc[o][r][c], ad, bf[c]);
        }
      }
    }
  }
  float* out[3] = {a.T[li], a.Q[li], a.Y[li]};
#pragma unroll
  for (int o = 0; o < 3; ++o) {
    const double base = dv[3 * M + o];
#pragma unroll
    for (int r = 0; r < 2; ++r)
#pragma unroll
      for (int c = 0; c < 4; ++c)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int i = bi * VT + wi + 8 * r + (lane >> 2), j = bj * VT + wj + 8 * c + 2 * (lane & 3) + h;
          if (i < M && j < M && j >= i) {
            double x = acc[o][r][c][h];
            if (i == j) x += unit ? dv[o * M + i] : base;
            out[o][(int64_t)i * M + j] = (float)x;
            out[o][(int64_t)j * M + i] = (float)x;
          }
        }
  }
}

}  // namespace

// Scratch of one layer: barrier words, W (fp64), eigenvalues, the three weight vectors and the identity's weights.  The
// size callers have been told is that of two M x M matrices; small M need more for the padding of the rows.
size_t evd_scratch_bytes(int M) {
  const size_t m = (size_t)M;
  return std::max(m * evd_ld(M), 2 * m * m) * sizeof(double) + (4 * m + kBase) * sizeof(double) + kWords * 4;
}

// Decomposes src[i] (M x M fp32 symmetric) of every layer.  with_v: T, Q, Phi_y are written to the three outputs (T is
// symmetric: it is its own transpose).  lam_out / kappa_out: optional per-layer outputs.
cudaError_t launch_evd(int n, const float* const* src, const int* layer_M, void* const* scratch,
                       int32_t* const* status, const float* eps, bool with_v, float g_max, float* const* T_out,
                       float* const* Q_out, float* const* Y_out, float* const* lam_out, float* const* kappa_out,
                       cudaStream_t s) {
  static SmemAttrCache attr;
  const int sms = sm_count();
  cudaError_t e = cudaSuccess;
  EvdArgs a;
  FinishArgs f;
  VdvArgs v;
  memset(&a, 0, sizeof(a)); memset(&f, 0, sizeof(f)); memset(&v, 0, sizeof(v));
  int tiles = 0, blocks = 0, stride = 0;
  for (int i = 0; i < n; ++i) {
    const int M = layer_M[i];
    char* base = reinterpret_cast<char*>(scratch[i]);
    EvdLayer& l = a.l[i];
    l.A = src[i];
    l.words = reinterpret_cast<int32_t*>(base);
    l.W = reinterpret_cast<double*>(base + kWords * 4);
    l.status = status[i];
    l.M = M;
    l.nb = ((M + EB - 1) / EB + 1) & ~1;
    l.n = 1;
    f.lam[i] = l.W + (size_t)M * evd_ld(M);
    f.dvec[i] = with_v ? f.lam[i] + M : nullptr;
    f.lam_sorted[i] = lam_out ? lam_out[i] : nullptr;
    f.kappa[i] = kappa_out ? kappa_out[i] : nullptr;
    f.eps[i] = eps[i];
    f.block0[i] = blocks;
    blocks += (M + 7) / 8;
    v.dvec[i] = f.dvec[i];
    if (with_v) { v.T[i] = T_out[i]; v.Q[i] = Q_out[i]; v.Y[i] = Y_out[i]; }
    v.tile0[i] = tiles;
    const int t = (M + VT - 1) / VT;
    tiles += t * (t + 1) / 2;
    stride = std::max(stride, evd_stride(std::min(evd_ld(M), kChunk)));
  }
  f.block0[n] = blocks; v.tile0[n] = tiles;
  a.nl = n; f.nl = n; v.nl = n;
  f.g_max = g_max;
  // CTAs: one per layer, then one more to the layer that takes longest, as long as it helps it.  A round costs a fixed
  // part (inner rotations, barrier) and a part in proportion to the columns' length; a CTA takes its pairs in turn.
  auto cost = [&](const EvdLayer& l, int ctas) {
    const int np = l.nb / 2;
    return (double)(l.nb - 1) * ((np + ctas - 1) / ctas) * (600.0 + l.M);
  };
  for (int used = n; used < sms; ) {
    int w = 0;
    for (int i = 1; i < n; ++i)
      if (cost(a.l[i], a.l[i].n) > cost(a.l[w], a.l[w].n)) w = i;
    const int np = a.l[w].nb / 2;
    const int turns = (np + a.l[w].n - 1) / a.l[w].n;
    if (turns == 1) break;
    const int need = (np + turns - 2) / (turns - 1);             // CTAs for one turn less
    if (used + need - a.l[w].n > sms) break;
    used += need - a.l[w].n;
    a.l[w].n = need;
  }
  int ctas = 0;
  for (int i = 0; i < n; ++i) { a.l[i].cta0 = ctas; ctas += a.l[i].n; f.l[i] = a.l[i]; v.l[i] = a.l[i]; }
  const size_t smem = ((size_t)EP * stride + kPartDoubles + EP * kGLd) * sizeof(double);
  e = ensure_dyn_smem(jacobi_kernel, smem, attr);
  if (e != cudaSuccess) return e;
  {
    ProfScope ps(FW_PROF_MISC, s);
    e = launch_dep(evd_clear_kernel, n, kWords, 0, s, a);
    if (e != cudaSuccess) return e;
  }
  {
    void* args[] = {&a};
    ProfScope ps(FW_PROF_MISC, s);
    e = cudaLaunchCooperativeKernel((void*)jacobi_kernel, dim3(ctas), dim3(ET), args, smem, s);
    if (e != cudaSuccess) return e;
  }
  {
    ProfScope ps(FW_PROF_MISC, s);
    e = launch_dep(norm_kernel, blocks, 256, 0, s, f);
    if (e != cudaSuccess) return e;
  }
  {
    ProfScope ps(FW_PROF_MISC, s);
    e = launch_dep(evd_finish_kernel, n, 1024, 0, s, f);
    if (e != cudaSuccess) return e;
  }
  if (with_v) {
    ProfScope ps(FW_PROF_MISC, s);
    static SmemAttrCache vattr;
    e = ensure_dyn_smem(vdv_kernel, VS * sizeof(VdvStage), vattr);
    if (e != cudaSuccess) return e;
    e = launch_dep(vdv_kernel, tiles, 256, VS * sizeof(VdvStage), s, v);
  }
  return e;
}

}  // namespace fw
