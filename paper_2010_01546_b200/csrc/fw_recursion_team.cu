// Recursive condition-number reduction (Sec. 4) for layers too large for one
// cluster, all steps of a launch in one cooperative launch.  A layer is given a
// team of CTAs (one CTA per SM) that holds all rows of Phi_y in shared memory, as
// many as fit, for all its steps; the layers of a group run side by side on
// disjoint teams and, where the chip cannot hold them together, in waves.  T and
// Q are not needed by a step: its v_e and a_e are recorded and applied afterwards
// (fw_recursion_apply.cu).  So a step moves no matrix through HBM, and what bounds
// it is the chain of P + 5 dependent passes:
//   - the products themselves: 32 matrix elements per clock and SM, both by
//     shared-memory bandwidth and by the four operations an element costs (below);
//     rows that do not fit are streamed from L2 / HBM instead;
//   - one exchange per pass through L2.  A result is stored as one 8-byte packet
//     {value, exchange number}; every CTA of the team polls the packets it needs
//     until they carry the number it waits for.  No flag, no fence, no barrier
//     counter: the exchange costs one store and one load latency.
//
// Two packet slots alternate: a CTA sends exchange e + 1 only after it has received
// all of e, so nobody still reads e - 1 when its slot is written again.  The row
// norms have a slot of their own, read again when the coherent set is formed.
//
// Precision of the products.  Alignment weights 1 / c_m (Eq. 49) amplify the error
// of c_m by up to 1 / c_rel, so the products are summed in more than fp32.  fp64
// would be bound by the conversions (16 per clock and SM).  Instead the sum is held
// as s + l in two fp32 numbers: s starts at C = 1.5 * 2^k, at least four times the
// bound ||row|| ||x|| on every partial sum, so fma(a, x, s) rounds each product to a
// multiple of ulp(C) without leaving the binade; the part rounded off is exactly
// fma(a, x, s_old - s_new) to fp32, and l collects it.  The total is (s - C) + l with
// an error near 2^-42 ||row|| ||x||.
//
// Every wait is bounded: a thread that gives up raises its CTA's flag, after which
// the CTA waits for nothing, runs to the end and reports FW_ERR_TIMEOUT.
#include <algorithm>
#include <cstring>
#include <vector>

#include "fw_fixsum.cuh"
#include "fw_internal.h"
#include "fw_lanes.cuh"

namespace fw {
namespace {

constexpr int PT = 512;              // threads per CTA
constexpr int PW = PT / 32;          // warps
constexpr int kMaxRows = 96;         // rows of a layer per CTA, at most
constexpr uint32_t kPollLimit = 1u << 19;
constexpr size_t kSmem = 227 * 1024 - 1280;   // dynamic; the static variables take the rest (48 rows of M = 1152 fit)

struct TeamArgs {
  GroupDev g;
  PtrTable traces;
  int32_t wave[FW_MAX_GROUP];        // when a layer runs
  int32_t first[FW_MAX_GROUP];       // its first CTA
  int32_t n[FW_MAX_GROUP];           // its CTAs
  uint32_t epoch[FW_MAX_GROUP];      // number of the layer's last exchange before this launch
  int32_t k0, K, P, nwaves;
  int32_t last;                      // this launch ends the call
};

// packets of a slot, whole 128-byte lines
__host__ __device__ inline int packet_stride(int M) { return (M + 15) & ~15; }

__device__ __forceinline__ void put(u64* p, float v, uint32_t epoch) {
  const u64 w = ((u64)epoch << 32) | __float_as_uint(v);
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(w) : "memory");
}
__device__ __forceinline__ u64 peek(const u64* p) {
  u64 w;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(w) : "l"(p) : "memory");
  return w;
}
__device__ __forceinline__ float value_of(u64 w) { return __uint_as_float((uint32_t)w); }

// (d + l) scale, rounded once
__device__ __forceinline__ float scaled(float2 a, float scale) {
  const float p = __fmul_rn(a.x, scale);
  return __fadd_rn(p, fmaf(a.y, scale, fmaf(a.x, scale, -p)));
}
// sums of four such values over the warp; lane 8 r holds the r-th
__device__ __forceinline__ float2 warp_sum4(float2 y0, float2 y1, float2 y2, float2 y3) {
  const int lane = threadIdx.x & 31;
  const bool hi = (lane & 16) != 0, mid = (lane & 8) != 0;
  const float2 u0 = add2(hi ? y2 : y0, shfl_xor2(hi ? y0 : y2, 16));
  const float2 u1 = add2(hi ? y3 : y1, shfl_xor2(hi ? y1 : y3, 16));
  float2 z = add2(mid ? u1 : u0, shfl_xor2(mid ? u0 : u1, 8));
  z = add2(z, shfl_xor2(z, 4));
  z = add2(z, shfl_xor2(z, 2));
  return add2(z, shfl_xor2(z, 1));
}

// dynamic shared memory: [two vectors of Mp floats][partial results][cached rows, Mp floats each].  Vectors and rows are
// addressed by their offset from here, so that the compiler knows them to be in shared memory.
extern __shared__ __align__(16) float psm[];

// One layer as its CTA sees it.
struct Team {
  const LayerDev* L;
  int rows;           // offset of the cached rows, Mp apart
  int part;           // offset of the partial results (float2) of the warps that share a row, kPartRows apart
  float* phiy;        // my rows in global memory
  u64* slot;          // two alternating packet slots, Me (M rounded up to even) apart
  u64* xi;            // packet slot of the squared row norms
  int M, Mp;
  int row0, nrows;    // my rows
  int ncached;        // leading rows kept in shared memory (all of them or a multiple of four)
  int cg_log;         // warps that share a group of four rows, each a part of the columns: 1, 2 or 4 (its logarithm)
  int sub, n;
};

constexpr int kPartRows = 32;   // rows per CTA up to which the columns of a row are split over warps

struct Shared {
  Team t;
  int layer, fail;
  float red[2][PW][2];
  uint32_t key[PW], idx[PW];
  float xi2[kMaxRows], xn[kMaxRows];   // squared norms and norms of my rows
};

// four consecutive entries c4, M of a row in global memory (rows of odd length are not 16-byte aligned)
__device__ __forceinline__ float4 load4(const float* row, int c, int M, bool v4) {
  if (v4) return *(reinterpret_cast<const float4*>(row) + c);
  float4 r = make_float4(0.f, 0.f, 0.f, 0.f);
  if (4 * c < M) r.x = row[4 * c];
  if (4 * c + 1 < M) r.y = row[4 * c + 1];
  if (4 * c + 2 < M) r.z = row[4 * c + 2];
  if (4 * c + 3 < M) r.w = row[4 * c + 3];
  return r;
}
__device__ __forceinline__ void store4(float* row, int c, int M, bool v4, float4 r) {
  if (v4) { reinterpret_cast<float4*>(row)[c] = r; return; }
  if (4 * c < M) row[4 * c] = r.x;
  if (4 * c + 1 < M) row[4 * c + 1] = r.y;
  if (4 * c + 2 < M) row[4 * c + 2] = r.z;
  if (4 * c + 3 < M) row[4 * c + 3] = r.w;
}

// Pairs of packets a thread takes in one go (M = 2304 in one): pair p holds packets 2 p, 2 p + 1.  16-byte loads halve the requests
// that all CTAs of a team aim at the same lines (1.0 us an exchange instead of 1.2 at M = 1152, 1.35 instead of 1.9 at
// M = 2304 on 144 CTAs).
constexpr int kPairs = 3;
__device__ __forceinline__ void peek2(const u64* p, u64& a, u64& b) {
  asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "l"(p) : "memory");
}
// Polls pairs p0, p0 + PT, ... of `slot` until their packets carry `epoch`; v: the values, 0 past the vector.  p0 differs
// by lane only: the warp polls as one (lanes past the vector repeat its last pair), since a warp whose lanes leave the
// loop one by one took 0.4 us longer an exchange.
__device__ __forceinline__ void poll(const u64* slot, int p0, int M, uint32_t epoch, Shared& sh, float2 (&v)[kPairs]) {
  u64 a[kPairs], b[kPairs];
  const int last = (M - 1) >> 1;
  uint32_t i = 0;
  for (;;) {
    bool ok = true;
#pragma unroll
    for (int j = 0; j < kPairs; ++j)
      if (2 * (p0 - (int)(threadIdx.x & 31) + j * PT) < M) peek2(slot + 2 * min(p0 + j * PT, last), a[j], b[j]);
#pragma unroll
    for (int j = 0; j < kPairs; ++j) {
      if (2 * (p0 - (int)(threadIdx.x & 31) + j * PT) < M) {
        const bool two = 2 * min(p0 + j * PT, last) + 1 < M;
        ok = ok && (uint32_t)(a[j] >> 32) == epoch && (!two || (uint32_t)(b[j] >> 32) == epoch);
      }
    }
    if (__all_sync(0xffffffffu, ok)) break;
    if ((++i & 255u) == 0 && (i >= kPollLimit || *(volatile int*)&sh.fail)) { *(volatile int*)&sh.fail = 1; break; }
  }
#pragma unroll
  for (int j = 0; j < kPairs; ++j) {
    const int m = 2 * (p0 + j * PT);
    v[j].x = m < M ? value_of(a[j]) : 0.f;
    v[j].y = m + 1 < M ? value_of(b[j]) : 0.f;
  }
}

// block sums of two values; one barrier.  Calls alternate between two sets of slots (flip).
__device__ __forceinline__ void block_sum2(float& a, float& b, Shared& sh, int flip) {
  a = warp_sum(a); b = warp_sum(b);
  float(*red)[2] = sh.red[flip & 1];
  if ((threadIdx.x & 31) == 0) { red[threadIdx.x >> 5][0] = a; red[threadIdx.x >> 5][1] = b; }
  __syncthreads();
  a = b = 0.f;
#pragma unroll
  for (int w = 0; w < PW; ++w) { a += red[w][0]; b += red[w][1]; }
}

// The vector at offset `dst` <- the vector of exchange `epoch`; returns its squared norm and, where dot >= 0, its product
// with the vector at `dot` in d
__device__ __forceinline__ float receive(const u64* slot, int M, uint32_t epoch, int dst, Shared& sh, int flip, int dot,
                                         float& d) {
  float sq = 0.f, dt = 0.f;
  for (int p0 = threadIdx.x; 2 * (p0 & ~31) < M; p0 += kPairs * PT) {
    float2 v[kPairs];
    poll(slot, p0, M, epoch, sh, v);
#pragma unroll
    for (int j = 0; j < kPairs; ++j) {
      const int p = p0 + j * PT;
      if (2 * p < M) {
        reinterpret_cast<float2*>(psm + dst)[p] = v[j];
        sq = fmaf(v[j].x, v[j].x, sq); sq = fmaf(v[j].y, v[j].y, sq);
        if (dot >= 0) {
          const float2 q = reinterpret_cast<const float2*>(psm + dot)[p];
          dt = fmaf(v[j].x, q.x, dt); dt = fmaf(v[j].y, q.y, dt);
        }
      }
    }
  }
  block_sum2(sq, dt, sh, flip);
  d = dt;
  return sq;
}

// Four rows times the vector at offset xo, columns c0, c0 + stride, ... of it; lane 8 r returns the r-th row's sum.
// CACHED: the rows are in shared memory, Mp apart; else in global memory, M apart, nrows of them.
template <bool CACHED>
__device__ __forceinline__ float2 group_product(const float* grow, int row, int nrows, int M, int Mp, int xo, float xnorm,
                                                const float* xn, int c0, int stride) {
  u64 s[4], l[4];
  float C[4];
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    C[r] = anchor(xn[r] * xnorm);
    s[r] = pack2(C[r], C[r]);
    l[r] = 0;
  }
  const bool v4 = (M & 3) == 0;
#pragma unroll 2
  for (int c = 4 * c0; c < Mp; c += 4 * stride) {
    const ulonglong2 xv = *reinterpret_cast<const ulonglong2*>(psm + xo + c);
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      ulonglong2 av;
      if (CACHED) av = *reinterpret_cast<const ulonglong2*>(psm + row + r * Mp + c);
      else { const float4 q = load4(grow + (size_t)min(r, nrows - 1) * M, c >> 2, M, v4); av.x = pack2(q.x, q.y); av.y = pack2(q.z, q.w); }
      fix_add(s[r], l[r], av.x, xv.x);
      fix_add(s[r], l[r], av.y, xv.y);
    }
  }
  float2 y[4];
#pragma unroll
  for (int r = 0; r < 4; ++r) y[r] = fix_value(s[r], l[r], C[r]);
  return warp_sum4(y[0], y[1], y[2], y[3]);
}
// y = scale (my rows) x, sent into `slot` as exchange `epoch`; x at offset xo, xnorm: ||x||.  One group of four rows at a
// time per warp (or per cg warps, which split the columns).  STREAM: some rows are in global memory.
template <bool STREAM>
__device__ __forceinline__ void product(const Shared& sh, int xo, float xnorm, float scale, u64* slot, uint32_t epoch) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int M = sh.t.M, Mp = sh.t.Mp, nrows = sh.t.nrows, shift = sh.t.cg_log, rows = sh.t.rows;
  const int groups = (nrows + 3) >> 2, cached = STREAM ? sh.t.ncached >> 2 : groups;
  const int part = warp & ((1 << shift) - 1), step = PW >> shift;
  float2* parts = reinterpret_cast<float2*>(psm + sh.t.part);
  slot += sh.t.row0;
  xnorm *= 1.01f;
  for (int g = warp >> shift; g < groups; g += step) {
    const int c0 = part * 32 + lane, stride = 32 << shift;
    float2 y;
    if (!STREAM || g < cached) y = group_product<true>(nullptr, rows + 4 * g * Mp, 4, M, Mp, xo, xnorm, sh.xn + 4 * g, c0, stride);
    else y = group_product<false>(sh.t.phiy + (size_t)4 * g * M, 0, nrows - 4 * g, M, Mp, xo, xnorm, sh.xn + 4 * g, c0, stride);
    const int lr = 4 * g + (lane >> 3);
    if ((lane & 7) == 0 && lr < nrows) {
      if (shift == 0) put(slot + lr, scaled(y, scale), epoch);
      else parts[part * kPartRows + lr] = y;
    }
  }
  if (shift) {
    __syncthreads();
    if ((int)threadIdx.x < nrows) {
      float2 y = parts[threadIdx.x];
      for (int p = 1; p < (1 << shift); ++p) y = add2(y, parts[p * kPartRows + threadIdx.x]);
      put(slot + threadIdx.x, scaled(y, scale), epoch);
    }
  }
}

// n passes y = scale Phi_y x with the vectors exchanged between them: the first with (xnorm, scale) as given, the others
// with x normalised; x at offset xo, the results alternate between the two vectors.  A function of its own with nothing
// else in it, so that no register of the loop lives in memory: what is left of the L1 cache beside 226 KB of shared
// memory does not hold the spilled registers of 512 threads (measured: 5.7 us a pass instead of 2.9 at M = 1152).
struct PassOut { float x2, y2, xy; };    // of the last pass: ||x||^2, ||y||^2, x.y
template <bool STREAM>
__device__ __noinline__ PassOut passes(Shared& sh, int n, int xo, int yo, float xnorm, float scale, uint32_t epoch, int flip) {
  const int M = sh.t.M;
  u64* const slot = sh.t.slot;
  const int Me = packet_stride(M);
  float x2 = 0.f, n2 = 0.f, dot = 0.f;
#pragma unroll 1
  for (int i = 0; i < n; ++i) {
    u64* s = slot + ((epoch & 1u) ? Me : 0);
    product<STREAM>(sh, xo, xnorm, scale, s, epoch);
    x2 = n2;
    if (sh.t.cg_log == 0) __syncthreads();
    n2 = receive(s, M, epoch, yo, sh, flip, i + 1 == n ? xo : -1, dot);
    xnorm = sqrtf(n2);
    scale = inv_norm(n2);
    const int z = xo; xo = yo; yo = z;
    ++epoch;
    flip ^= 1;
  }
  return PassOut{x2, n2, dot};
}

// block maximum of (key, lowest index); one barrier before the result is read
__device__ __forceinline__ int block_argmax(uint32_t key, uint32_t idx, Shared& sh, int M) {
  const uint32_t top = __reduce_max_sync(0xffffffffu, key);
  const uint32_t at = __reduce_min_sync(0xffffffffu, key == top ? idx : 0xffffffffu);
  if ((threadIdx.x & 31) == 0) { sh.key[threadIdx.x >> 5] = top; sh.idx[threadIdx.x >> 5] = at; }
  __syncthreads();
  uint32_t k = sh.key[threadIdx.x & (PW - 1)], i = sh.idx[threadIdx.x & (PW - 1)];
  const uint32_t best = __reduce_max_sync(0xffffffffu, k);
  const uint32_t b = __reduce_min_sync(0xffffffffu, k == best ? i : 0xffffffffu);
  return best == 0 || b >= (uint32_t)M ? 0 : (int)b;
}

// Squared norms of my rows as they are, sent as exchange `epoch` (later steps get them from the update).
__device__ __noinline__ void row_norms(Shared& sh, uint32_t epoch) {
  const Team& t = sh.t;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int M = t.M, Mp = t.Mp, M4 = Mp >> 2;
  const bool v4 = (M & 3) == 0;
  for (int r = warp; r < t.nrows; r += PW) {
    double acc = 0.0;
    for (int c = lane; c < M4; c += 32) {
      const float4 q = r < t.ncached ? *reinterpret_cast<const float4*>(psm + t.rows + r * Mp + 4 * c)
                                     : load4(t.phiy + (size_t)r * M, c, M, v4);
      acc = fma((double)q.x, (double)q.x, acc); acc = fma((double)q.y, (double)q.y, acc);
      acc = fma((double)q.z, (double)q.z, acc); acc = fma((double)q.w, (double)q.w, acc);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) { sh.xi2[r] = (float)acc; sh.xn[r] = sqrtf((float)acc); put(t.xi + t.row0 + r, (float)acc, epoch); }
  }
}

// m' = argmax xi, lowest index on ties (Eqs. 45-46), of exchange `epoch`
__device__ __noinline__ int receive_argmax(Shared& sh, uint32_t epoch) {
  const int M = sh.t.M;
  uint32_t key = 0, idx = 0;
  for (int p0 = threadIdx.x; 2 * (p0 & ~31) < M; p0 += kPairs * PT) {
    float2 v[kPairs];
    poll(sh.t.xi, p0, M, epoch, sh, v);
#pragma unroll
    for (int j = 0; j < kPairs; ++j) {
      const int m = 2 * (p0 + j * PT);
      const uint32_t k0 = v[j].x >= 0.f && m < M ? __float_as_uint(v[j].x) + 1u : 0u;       // a NaN never wins
      const uint32_t k1 = v[j].y >= 0.f && m + 1 < M ? __float_as_uint(v[j].y) + 1u : 0u;
      if (k0 > key) { key = k0; idx = m; }
      if (k1 > key) { key = k1; idx = m + 1; }
    }
  }
  return block_argmax(key, idx, sh, M);
}

// Row m' from its owner into the vector at xo (exchange `epoch`), c = Phi_y (Phi_y e_m') (Eq. 47, exchange `epoch` + 1),
// and the weights of the coherent set (Eqs. 48-49) into the vector at yo; returns the size of the set, and ||w||^2 in w2.
template <bool STREAM>
__device__ __noinline__ float2 correlate(Shared& sh, int mp, int xo, int yo, uint32_t epoch, int flip, bool keep) {
  const Team& t = sh.t;
  const LayerDev* L = t.L;
  const int tid = threadIdx.x, M = t.M;
  const int Me = packet_stride(M);
  u64* s = t.slot + ((epoch & 1u) ? Me : 0);
  if (mp >= t.row0 && mp < t.row0 + t.nrows) {
    const int r = mp - t.row0;
    if (r < t.ncached) for (int m = tid; m < M; m += PT) put(s + m, psm[t.rows + r * t.Mp + m], epoch);
    else for (int m = tid; m < M; m += PT) put(s + m, t.phiy[(size_t)r * M + m], epoch);
  }
  float unused;
  const float xi_mp = sqrtf(receive(s, M, epoch, xo, sh, flip, -1, unused));
  ++epoch;
  s = t.slot + ((epoch & 1u) ? Me : 0);
  product<STREAM>(sh, xo, xi_mp, 1.f, s, epoch);
  float cnt = 0.f, w2 = 0.f;
  if (L->init == FW_INIT_MAXCOL) {
    for (int m = tid; m < M; m += PT) psm[yo + m] = (m == mp) ? 1.f : 0.f;
    for (int p0 = tid; 2 * (p0 & ~31) < M; p0 += kPairs * PT) {       // received all the same: the slots alternate on that
      float2 v[kPairs];
      poll(s, p0, M, epoch, sh, v);
    }
    __syncthreads();
    return make_float2(1.f, 1.f);
  }
  const float c_rel = L->c_rel, c_abs = L->c_abs;
  const float xi_mx = sqrtf(value_of(peek(t.xi + mp)));
  for (int p0 = tid; 2 * (p0 & ~31) < M; p0 += kPairs * PT) {
    float2 v[kPairs];
    poll(s, p0, M, epoch, sh, v);
#pragma unroll
    for (int j = 0; j < kPairs; ++j) {
      const int m = 2 * (p0 + j * PT);
      if (m >= M) continue;
      u64 xa, xb;
      peek2(t.xi + m, xa, xb);
#define FW_WEIGHT(X, xi, i)                                                          \
      if ((i) < M) {                                                                 \
        const float thr = fmaxf(c_rel * xi_mx * sqrtf(value_of(xi)), c_abs);         \
        const bool in = fabsf(v[j].X) >= thr;          /* false for NaN */           \
        const float q = in ? 1.f / v[j].X : 0.f;                                     \
        psm[yo + (i)] = q;                                                           \
        cnt += in ? 1.f : 0.f;                                                       \
        w2 = fmaf(q, q, w2);                                                         \
        if (keep) L->wvec[i] = q;                                                    \
      }
      FW_WEIGHT(x, xa, m)
      FW_WEIGHT(y, xb, m + 1)
#undef FW_WEIGHT
    }
  }
  block_sum2(cnt, w2, sh, flip ^ 1);
  return make_float2(cnt, w2);
}

// Phi_y += a (v u^T + u v^T) + a^2 lambda_e v v^T = v w^T + w v^T with w = a u + (a^2 lambda_e / 2) v on my rows, exactly
// symmetric; v = inv x.  Squared norms of the new rows, sent as exchange `epoch` if `send`.
__device__ __noinline__ void update_rows(Shared& sh, int xo, int yo, float inv, float aa, float lam_e, float u2, bool send, uint32_t epoch) {
  const Team& t = sh.t;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int M = t.M, Mp = t.Mp, M4 = Mp >> 2, nrows = t.nrows, ncached = t.ncached, row0 = t.row0, rows = t.rows;
  const bool v4 = (M & 3) == 0;
  float* phiy = t.phiy;
  const float hl = 0.5f * aa * aa * lam_e;
  // ||w|| and with it a bound on the new rows' norms, which anchors their sums
  const float wn = 1.01f * (fabsf(aa) * sqrtf(u2) + fabsf(hl));
  for (int r = warp; r < nrows; r += PW) {
    const float vi = psm[xo + row0 + r] * inv;
    const float wi = __fadd_rn(__fmul_rn(aa, psm[yo + row0 + r]), __fmul_rn(hl, vi));
    const float bound = 1.01f * (sh.xn[r] + fabsf(vi) * wn + fabsf(wi));
    const float C = anchor(bound * bound);
    u64 s = pack2(C, C), l = 0;
    const bool cached = r < ncached;
#pragma unroll 2
    for (int c = lane; c < M4; c += 32) {
      float4 p = cached ? *reinterpret_cast<const float4*>(psm + rows + r * Mp + 4 * c) : load4(phiy + (size_t)r * M, c, M, v4);
      const float4 xv = *reinterpret_cast<const float4*>(psm + xo + 4 * c), uv = *reinterpret_cast<const float4*>(psm + yo + 4 * c);
#define FW_UPD(X)                                                                                  \
      {                                                                                            \
        const float vj = xv.X * inv;                                                               \
        const float wj = __fadd_rn(__fmul_rn(aa, uv.X), __fmul_rn(hl, vj));                         \
        p.X = __fadd_rn(p.X, __fadd_rn(__fmul_rn(vi, wj), __fmul_rn(wi, vj)));                      \
      }
      FW_UPD(x) FW_UPD(y) FW_UPD(z) FW_UPD(w)
#undef FW_UPD
      if (cached) *reinterpret_cast<float4*>(psm + rows + r * Mp + 4 * c) = p;
      else store4(phiy + (size_t)r * M, c, M, v4, p);
      const u64 p0 = pack2(p.x, p.y), p1 = pack2(p.z, p.w);
      fix_add(s, l, p0, p0);
      fix_add(s, l, p1, p1);
    }
    float2 acc = fix_value(s, l, C);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc = add2(acc, shfl_xor2(acc, o));
    if (lane == 0) {
      const float n2r = acc.x + acc.y;
      sh.xi2[r] = n2r; sh.xn[r] = sqrtf(n2r);
      if (send) put(t.xi + row0 + r, n2r, epoch);
    }
  }
}

// All steps of one layer by its team.
__device__ __noinline__ void run_layer(const TeamArgs& a, Shared& sh, int li) {
  const Team& t = sh.t;
  const int tid = threadIdx.x;
  uint32_t e = a.epoch[li];
  int flip = 0;
  {
    // ---- the cached rows into shared memory, zero rows up to whole groups of four ----
    const int M = t.M, Mp = t.Mp, M4 = Mp >> 2, padded = min((t.ncached + 3) & ~3, (t.nrows + 3) & ~3);
    const bool v4 = (M & 3) == 0;
    for (int i = tid; i < padded * M4; i += PT) {
      const int r = i / M4, c = i - r * M4;
      *reinterpret_cast<float4*>(psm + t.rows + r * Mp + 4 * c) =
          r < t.ncached ? load4(t.phiy + (size_t)r * M, c, M, v4) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    for (int i = tid; i < 2 * Mp; i += PT) psm[i] = 0.f;
    for (int i = tid; i < kMaxRows; i += PT) sh.xi2[i] = sh.xn[i] = 0.f;
  }
  __syncthreads();
  row_norms(sh, ++e);
  bool updated = false;
#pragma unroll 1
  for (int step = 0; step < a.K; ++step) {
    const int mp = receive_argmax(sh, e);
    const int Mp = t.Mp, M = t.M, P = a.P;
    const bool stream = t.ncached < t.nrows;
    const bool keep = a.last && step + 1 == a.K && t.sub == 0;
    const float2 cw = stream ? correlate<true>(sh, mp, 0, Mp, e + 1, flip, keep)
                             : correlate<false>(sh, mp, 0, Mp, e + 1, flip, keep);
    const int cnt = (int)(cw.x + 0.5f);
    // aligned average, P power iterations y = Phi_y (x / ||x||), then u = Phi_y v with v = x / ||x|| (Eqs. 49-50)
    const float inv_cnt = cnt > 0 ? 1.f / (float)cnt : 0.f;
    const PassOut o = stream ? passes<true>(sh, P + 2, Mp, 0, sqrtf(cw.y), inv_cnt, e + 3, flip)
                             : passes<false>(sh, P + 2, Mp, 0, sqrtf(cw.y), inv_cnt, e + 3, flip);
    flip ^= P & 1;
    e += (uint32_t)P + 4u;
    const int xo = (P & 1) ? Mp : 0, yo = Mp - xo;               // x and u of the last pass
    const float inv = inv_norm(o.x2), lam_e = o.xy * inv;          // Eq. 36
    // ---- g_e, a_e (Eqs. 40-41) ----
    const LayerDev* L = t.L;
    const bool ok = cnt > 0 && o.x2 > 0.f && isfinite(o.x2) && isfinite(lam_e);
    float g_e = 1.f, aa = 0.f;
    if (ok) {
      g_e = L->delta * L->scal[SC_LAMBDA_BAR] / fmaxf(lam_e, L->eps);
      aa = sqrtf(g_e) - 1.f;
    }
    if (t.sub == 0) {
      float* vh = L->vh + (size_t)step * M;
      for (int m = tid; m < M; m += PT) vh[m] = psm[xo + m] * inv;
      if (tid == 0) {
        L->ah[step] = aa;
        L->scal[SC_LAMBDA_E] = lam_e; L->scal[SC_G_E] = g_e; L->scal[SC_A_E] = aa;
        L->iscal[IS_MPRIME] = mp; L->iscal[IS_SETSIZE] = cnt;
        if (!ok) L->iscal[IS_STATUS_NOSUB] = 1;
        if (!isfinite(o.x2) || !isfinite(lam_e)) L->iscal[IS_STATUS_NONFINITE] = 1;
        float* tr = const_cast<float*>(reinterpret_cast<const float*>(a.traces.p[li]));
        if (tr) {
          tr += 4 * (a.k0 + step);
          tr[0] = lam_e; tr[1] = g_e; tr[2] = (float)cnt; tr[3] = (float)mp;
        }
      }
    }
    // ---- rank update, norms for the next step ----
    const bool more = step + 1 < a.K;
    if (more) ++e;
    if (aa != 0.f) {
      updated = true;
      update_rows(sh, xo, yo, inv, aa, lam_e, o.y2, more, e);
    } else if (more) {
      for (int r = tid; r < t.nrows; r += PT) put(t.xi + t.row0 + r, sh.xi2[r], e);
    }
    __syncthreads();           // rows, norms and both vectors are free for the next step
  }
  if (updated) {
    const int M = t.M, Mp = t.Mp, M4 = Mp >> 2;
    for (int i = tid; i < t.ncached * M4; i += PT) {
      const int r = i / M4, c = i - r * M4;
      store4(t.phiy + (size_t)r * M, c, M, (M & 3) == 0, *reinterpret_cast<const float4*>(psm + t.rows + r * Mp + 4 * c));
    }
  }
  if (tid == 0 && *(volatile int*)&sh.fail) atomicExch(t.L->iscal + IS_STATUS_TIMEOUT, 501);
}

__host__ __device__ inline int team_rows(int M, int n) { return (M + n - 1) / n; }
// rows that fit beside the two vectors and the partial results, whole groups of four; R: rows per CTA
constexpr int kPartFloats = 4 * kPartRows * 2;   // float2 each
__host__ __device__ inline int team_cache(int M, int R) {
  const int Mp = (M + 3) & ~3;
  return (((int)(kSmem / sizeof(float)) - 2 * Mp - (R <= kPartRows ? kPartFloats : 0)) / Mp) & ~3;
}

__global__ void __launch_bounds__(PT, 1) recursion_team_kernel(const __grid_constant__ TeamArgs a) {
  dep_sync();
  __shared__ Shared sh;
  if (threadIdx.x == 0) sh.fail = 0;
  for (int w = 0; w < a.nwaves; ++w) {
    __syncthreads();
    if (threadIdx.x == 0) {
      int li = -1;
#pragma unroll 1
      for (int l = 0; l < a.g.n; ++l)
        if (a.wave[l] == w && (int)blockIdx.x >= a.first[l] && (int)blockIdx.x < a.first[l] + a.n[l]) li = l;
      sh.layer = li;
      if (li >= 0) {
        const LayerDev* L = a.g.layer[li];
        const int M = L->M, R = team_rows(M, a.n[li]);
        Team& t = sh.t;
        t.L = L; t.M = M; t.Mp = (M + 3) & ~3;
        t.n = a.n[li]; t.sub = (int)blockIdx.x - a.first[li];
        t.row0 = min(M, t.sub * R);
        t.nrows = min(M, t.row0 + R) - t.row0;
        t.phiy = L->Phiy + (size_t)t.row0 * M;
        const int fit = team_cache(M, R);
        t.ncached = min(t.nrows, fit);
        t.part = 2 * t.Mp;
        t.rows = 2 * t.Mp + (R <= kPartRows ? kPartFloats : 0);
        t.slot = L->px; t.xi = L->px + 2 * packet_stride(M);
        const int groups = (R + 3) / 4;
        t.cg_log = groups <= 4 ? 2 : (R <= kPartRows ? 1 : 0);
      }
    }
    __syncthreads();
    if (sh.layer >= 0) run_layer(a, sh, sh.layer);
  }
}

// Waves and teams.  Largest layers first; a wave takes layers while the CTAs that hold their rows fit, then its spare
// CTAs go to the layer whose passes cost most.
struct TeamPlan {
  int dev = -1, n = 0, waves = 0;
  int dims[FW_MAX_GROUP];
  int32_t wave[FW_MAX_GROUP], first[FW_MAX_GROUP], cnt[FW_MAX_GROUP];
};

// clocks of a pass on n CTAs: rows in shared memory at 32 elements per clock, streamed rows at about 12
double team_cost(int M, int n) {
  const int R = team_rows(M, n), fit = team_cache(M, R), cached = std::min(R, fit);
  return ((double)cached / 32 + (double)(R - cached) / 12) * M;
}

void make_plan(TeamPlan& p, const int* M, int n, int ctas) {
  std::vector<int> order(n);
  for (int i = 0; i < n; ++i) order[i] = i;
  std::stable_sort(order.begin(), order.end(), [&](int x, int y) { return M[x] > M[y]; });
  std::vector<bool> done(n, false);
  int left = n, w = 0;
  while (left) {
    std::vector<int> in;
    int used = 0;
    for (int oi = 0; oi < n; ++oi) {
      const int i = order[oi];
      if (done[i]) continue;
      const int fit = std::min(team_cache(M[i], kMaxRows), kMaxRows);
      int need = (M[i] + fit - 1) / fit;
      if (need > ctas) need = ctas;
      // half the chip is enough for a layer that nearly fits it: two such layers side by side stream a row or two each
      if (need > ctas / 2 && need <= ctas / 2 + 4) need = ctas / 2;
      if (used + need > ctas) continue;
      in.push_back(i); p.cnt[i] = need; p.wave[i] = w; used += need; done[i] = true; --left;
    }
    for (;;) {
      int worst = in[0];
      for (int i : in) if (team_cost(M[i], p.cnt[i]) > team_cost(M[worst], p.cnt[worst])) worst = i;
      // one more row less per CTA, while the wave has the CTAs and eight rows a CTA are left
      const int R = team_rows(M[worst], p.cnt[worst]);
      if (R <= 8) break;
      const int next = (M[worst] + R - 2) / (R - 1);
      if (used + next - p.cnt[worst] > ctas) break;
      used += next - p.cnt[worst];
      p.cnt[worst] = next;
    }
    int at = 0;
    for (int i : in) { p.first[i] = at; at += p.cnt[i]; }
    ++w;
  }
  p.waves = w; p.n = n;
  memcpy(p.dims, M, n * sizeof(int));
}

}  // namespace

int team_exchanges(int K, int P) { return K * (P + 5); }

cudaError_t launch_recursion_team(const GroupDev& g, const PtrTable& traces, const int* layer_M, const uint32_t* epoch,
                                  int k0, int K, int P, bool last, cudaStream_t s) {
  static int n_sm[64] = {0};
  static SmemAttrCache attr;
  thread_local TeamPlan plan;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) dev = 0;
  if (n_sm[dev] == 0) {
    int v = 0;
    e = cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    n_sm[dev] = v;
  }
  e = ensure_dyn_smem(recursion_team_kernel, kSmem, attr);
  if (e != cudaSuccess) return e;
  if (plan.dev != dev || plan.n != g.n || memcmp(plan.dims, layer_M, g.n * sizeof(int)) != 0) {
    make_plan(plan, layer_M, g.n, n_sm[dev]);
    plan.dev = dev;
  }
  TeamArgs a;
  memset(&a, 0, sizeof(a));
  a.g = g; a.traces = traces; a.k0 = k0; a.K = K; a.P = P; a.nwaves = plan.waves; a.last = last ? 1 : 0;
  int ctas = 0;
  for (int i = 0; i < g.n; ++i) {
    a.wave[i] = plan.wave[i]; a.first[i] = plan.first[i]; a.n[i] = plan.cnt[i]; a.epoch[i] = epoch[i];
    ctas = std::max(ctas, plan.first[i] + plan.cnt[i]);
  }
  void* args[] = {&a};
  ProfScope ps(FW_PROF_RECUR_MV, s);
  return cudaLaunchCooperativeKernel((void*)recursion_team_kernel, dim3(ctas), dim3(PT), args, kSmem, s);
}

}  // namespace fw
