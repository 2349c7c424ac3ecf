// Recursive condition-number reduction (Sec. 4) for layers too large for one
// cluster, all steps of a launch in one cooperative launch.  A layer is given a
// team of CTAs (one CTA per SM) that holds all rows of Phi_y in shared memory, as
// many as fit, for all its steps; the layers of a group run side by side on
// disjoint teams and, where the chip cannot hold them together, in waves.  T and
// Q are not needed by a step: its v_e and a_e are recorded and applied afterwards
// (fw_recursion_apply.cu).  So a step moves no matrix through HBM, and what bounds
// it is the chain of P + 5 dependent passes:
//   - the products: 5 bytes of shared memory an element (four rows share a load of the
//     vector), so at most 26 matrix elements per clock and SM; rows that do not fit are
//     streamed from L2 / HBM instead;
//   - one exchange per pass through L2.  A result is stored as one 8-byte packet
//     {value, exchange number}; every CTA of the team polls the packets it needs
//     until they carry the number it waits for.  No flag, no fence, no barrier
//     counter: the exchange costs one store and one load latency.
// Clocks of a pass (clock64 in one CTA; six layers of M = 1152, 48 rows a CTA / one of
// M = 2304, 16 rows): product 4740 / 3830, block barrier 100 / 110, polling 1500 / 1900,
// norm and scale 950 / 1300: 7290 = 3.7 us / 7140 = 3.6 us.  The product is about 1800
// clocks from the first load to the last packet whatever its size, and 108 per four rows
// by 128 columns and SM partition, where shared memory alone would take 80.
//
// Two packet slots alternate: a CTA sends exchange e + 1 only after it has received
// all of e, so nobody still reads e - 1 when its slot is written again.  The row
// norms have a slot of their own, read again when the coherent set is formed.  The
// numbers go on from launch to launch (a layer's IS_EXCHANGE, in device memory: a
// launch replayed from a captured graph counts on as well).
//
// Rounding.  The set of Eq. 48 is a comparison per column and step, and at condition 1e4 a start vector with one column
// more or less leads to another transform; so every operation is rounded in one stated way, whatever the team:
//   - a product is the fp64 sum of its row in one order (exact_row below) rounded to fp32;
//   - vectors are normalised in fp32, entry by entry, before they are multiplied;
//   - norms and v.u are fp32 sums in the order given at block_sum();
//   - the rank update has one rounding per operation (rank2).
//
// Every wait is bounded: a thread that gives up raises its CTA's flag, after which
// the CTA waits for nothing, runs to the end and reports FW_ERR_TIMEOUT.
#include <algorithm>
#include <cstring>
#include <vector>

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

// Sums over the warp of four values per lane; lane 8 r holds the r-th.
__device__ __forceinline__ double warp_sum4(double y0, double y1, double y2, double y3) {
  const int lane = threadIdx.x & 31;
  const bool hi = (lane & 16) != 0, mid = (lane & 8) != 0;
  const double u0 = (hi ? y2 : y0) + __shfl_xor_sync(0xffffffffu, hi ? y0 : y2, 16);
  const double u1 = (hi ? y3 : y1) + __shfl_xor_sync(0xffffffffu, hi ? y1 : y3, 16);
  double z = (mid ? u1 : u0) + __shfl_xor_sync(0xffffffffu, mid ? u0 : u1, 8);
  z += __shfl_xor_sync(0xffffffffu, z, 4);
  z += __shfl_xor_sync(0xffffffffu, z, 2);
  return z + __shfl_xor_sync(0xffffffffu, z, 1);
}

// dynamic shared memory: [two vectors of Mp floats][partial sums][cached rows, Mp floats each].  All are addressed by their offset from here, so that the compiler knows them to be in shared memory.
extern __shared__ __align__(16) float psm[];

// One layer as its CTA sees it.
struct Team {
  const LayerDev* L;
  int rows;           // offset of the cached rows, Mp apart
  int part;           // offset of the partial sums: fp64 of warps that share rows, fp32 of a norm (pair_partial)
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
  float negz;            // -0
  __align__(16) float red[2][2 * PW];
  uint32_t key[PW], idx[PW];
  float xi2[kMaxRows];   // squared norms of my rows
  float win[kMaxRows];   // what two orders of a row's product with a unit vector may differ by
};

// four consecutive entries c4, M of a row in global memory (rows that are not whole float4s are not 16-byte aligned)
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

// Sum over the block of two values per thread, those of pairs of neighbouring entries.  Entry m belongs to (virtual) thread
// m mod 1024, which adds its entries in ascending order; 32 neighbouring threads are added as a butterfly from 16 to 1 and
// their 32 sums in ascending order.  Two neighbouring entries are a thread here, so the butterfly of 32 runs over 16 lanes and
// ends within the thread.  One barrier; calls alternate between two sets of slots (flip).
__device__ __forceinline__ float block_sum(float x, float y, Shared& sh, int flip) {
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) { x += __shfl_xor_sync(0xffffffffu, x, o); y += __shfl_xor_sync(0xffffffffu, y, o); }
  float* red = sh.red[flip & 1];
  if ((threadIdx.x & 15) == 0) red[threadIdx.x >> 4] = x + y;
  __syncthreads();
  float t = 0.f;
#pragma unroll
  for (int w = 0; w < 2 * PW / 4; ++w) {
    const float4 r = reinterpret_cast<const float4*>(red)[w];
    t += r.x; t += r.y; t += r.z; t += r.w;
  }
  return t;
}
// The same for vectors that are not whole float4s, in another order: pairs of entries, eight pairs in ascending order
// (partial sums in `part`), partial b to thread b mod 256, a butterfly over 32 threads, their eight sums in ascending order.
// q: sum of the thread's pair p.
__device__ __forceinline__ void pair_partial(float q, int p, float* part) {
  float s = 0.f;
#pragma unroll
  for (int w = 0; w < 8; ++w) s += __shfl_sync(0xffffffffu, q, (threadIdx.x & 24) + w);
  if ((threadIdx.x & 7) == 0) part[p >> 3] = s;
}
__device__ __forceinline__ float partial_sum(const float* part, int n, Shared& sh, int flip) {
  __syncthreads();
  float s = 0.f;
  if (threadIdx.x < 256) {
    for (int b = threadIdx.x; b < n; b += 256) s += part[b];
    s = warp_sum(s);
    if ((threadIdx.x & 31) == 0) sh.red[flip & 1][threadIdx.x >> 5] = s;
  }
  __syncthreads();
  s = 0.f;
#pragma unroll
  for (int w = 0; w < 8; ++w) s += sh.red[flip & 1][w];
  return s;
}
// The vector at offset `dst` <- the vector of exchange `epoch`.
enum { SUM_NONE, SUM_SQUARES, SUM_DOT };
// Returns its squared norm or, SUM_DOT, its product with xs times the vector at `dot`.
template <bool V4>
__device__ __forceinline__ float receive(const u64* slot, int M, uint32_t epoch, int dst, Shared& sh, int flip, int what,
                                         int dot, float xs) {
  float sx = 0.f, sy = 0.f;
  float* part = psm + sh.t.part;
  for (int p0 = threadIdx.x; 2 * (p0 & ~31) < M; p0 += kPairs * PT) {
    float2 v[kPairs];
    poll(slot, p0, M, epoch, sh, v);
#pragma unroll
    for (int j = 0; j < kPairs; ++j) {
      const int p = p0 + j * PT;
      if (2 * (p & ~31) >= M) continue;                // uniform in the warp
      float2 q = v[j];                                 // 0 past the vector
      if (2 * p < M) {
        reinterpret_cast<float2*>(psm + dst)[p] = q;
        if (what == SUM_DOT) {
          q = reinterpret_cast<const float2*>(psm + dot)[p];
          q.x *= xs; q.y *= xs;
        }
      }
      if (what == SUM_NONE) continue;
      if (V4) { sx = fmaf(q.x, v[j].x, sx); sy = fmaf(q.y, v[j].y, sy); }
      else pair_partial(fmaf(q.y, v[j].y, __fmul_rn(q.x, v[j].x)), p, part);
    }
  }
  if (what == SUM_NONE) { __syncthreads(); return 0.f; }
  if (V4) return block_sum(sx, sy, sh, flip);
  return partial_sum(part, (((M + 1) >> 1) + 7) >> 3, sh, flip);
}

// Row r of mine times xs x (x at offset xo), the sum of record: in fp64, a lane takes the entries of every 32nd float4 (rows
// that are not whole float4s: every 32nd entry) in ascending order, the lanes are added as a butterfly from 16 to 1.
__device__ __noinline__ double exact_row(const Shared& sh, int r, int xo, float xs) {
  const int lane = threadIdx.x & 31;
  const int M = sh.t.M;
  const float* row = r < sh.t.ncached ? psm + sh.t.rows + r * sh.t.Mp : sh.t.phiy + (size_t)r * M;
  double acc = 0.0;
  if ((M & 3) == 0) {
    constexpr int B = 9;                           // loads in flight
    for (int c0 = lane; c0 < (M >> 2); c0 += 32 * B) {
      float4 a[B];
#pragma unroll
      for (int h = 0; h < B; ++h) a[h] = reinterpret_cast<const float4*>(row)[min(c0 + 32 * h, (M >> 2) - 1)];
#pragma unroll
      for (int h = 0; h < B; ++h) {
        const int c = c0 + 32 * h;
        if (c >= (M >> 2)) break;
        const float4 x = *reinterpret_cast<const float4*>(psm + xo + 4 * c);
        acc = fma((double)a[h].x, (double)(x.x * xs), acc); acc = fma((double)a[h].y, (double)(x.y * xs), acc);
        acc = fma((double)a[h].z, (double)(x.z * xs), acc); acc = fma((double)a[h].w, (double)(x.w * xs), acc);
      }
    }
  } else {
#pragma unroll 4
    for (int c = lane; c < M; c += 32) acc = fma((double)row[c], (double)(psm[xo + c] * xs), acc);
  }
  return warp_sum(acc);
}

// Four rows times xs x, x the vector at offset xo, entries (float4s where V4) c0, c0 + stride, ... of them; lane 8 r returns
// the r-th row's sum.  CACHED: the rows are in shared memory, Mp apart; else in global memory, M apart, nrows of them.
// An SM converts 16 numbers per clock to fp64; so three entries in four of a row are widened by integer operations, beside
// the conversions of the fourth and of x (clocks of a product, six layers of M = 1152: 4750; 5790 with conversions alone,
// 4930 with all four widened).
template <bool CACHED, bool V4, int SHIFT>
__device__ __forceinline__ double group_product(const float* grow, int row, int nrows, int M, int Mp, int xo, float xs, int c0) {
  constexpr int stride = 32 << SHIFT;
  double acc[4] = {0.0, 0.0, 0.0, 0.0};
  if (V4) {
#pragma unroll 2
    for (int c = c0; c < (M >> 2); c += stride) {
      const float4 x = *reinterpret_cast<const float4*>(psm + xo + 4 * c);
      const double x0 = (double)(x.x * xs) * kWiden, x1 = (double)(x.y * xs) * kWiden, x2 = (double)(x.z * xs) * kWiden,
                   x3 = (double)(x.w * xs);
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const float4 a = CACHED ? *reinterpret_cast<const float4*>(psm + row + r * Mp + 4 * c)
                                : *(reinterpret_cast<const float4*>(grow + (size_t)min(r, nrows - 1) * M) + c);
        acc[r] = fma(widen(a.x), x0, acc[r]); acc[r] = fma(widen(a.y), x1, acc[r]);
        acc[r] = fma(widen(a.z), x2, acc[r]); acc[r] = fma((double)a.w, x3, acc[r]);
      }
    }
  } else {
#pragma unroll 4
    for (int c = c0; c < M; c += stride) {
      const double x = (double)(psm[xo + c] * xs) * kWiden;
#pragma unroll
      for (int r = 0; r < 4; ++r)
        acc[r] = fma(widen(CACHED ? psm[row + r * Mp + c] : grow[(size_t)min(r, nrows - 1) * M + c]), x, acc[r]);
    }
  }
  return warp_sum4(acc[0], acc[1], acc[2], acc[3]);
}

// Whether the fp64 sum y of my row lr, formed in another order, may round to another fp32 number than the sum of record
// (about one row in 1e5).  sh.win[lr] xnorm: what the two sums may differ by; infinite for a row that is not finite.
__device__ __forceinline__ bool open_rounding(const Shared& sh, double y, int lr, float xnorm) {
  const double w = (double)(sh.win[lr] * xnorm);
  return (float)(y - w) != (float)(y + w);
}
// y = scale (my rows) (xs x), sent into `slot` as exchange `epoch`; x at offset xo, xnorm: a bound on ||xs x||.  One group of
// four rows at a time per warp (or per cg warps, which split the columns).  STREAM: some rows are in global memory.
template <bool STREAM, bool V4, int SHIFT>
__device__ __forceinline__ void product_split(const Shared& sh, int xo, float xs, float xnorm, float scale, u64* slot, uint32_t epoch) {
  constexpr int shift = SHIFT;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int M = sh.t.M, Mp = sh.t.Mp, nrows = sh.t.nrows, rows = sh.t.rows;
  slot += sh.t.row0;
  const int groups = (nrows + 3) >> 2, cached = STREAM ? sh.t.ncached >> 2 : groups;
  const int part = warp & ((1 << shift) - 1), step = PW >> shift;
  double* parts = reinterpret_cast<double*>(psm + sh.t.part);
  uint32_t open = 0;                                 // rows to be summed in the order of record: bit 8 r + i, row r of my i-th group
  int i = 0;
  for (int g = warp >> shift; g < groups; g += step, ++i) {
    const int c0 = part * 32 + lane;
    double y;
    if (!STREAM || g < cached) y = group_product<true, V4, SHIFT>(nullptr, rows + 4 * g * Mp, 4, M, Mp, xo, xs, c0);
    else y = group_product<false, V4, SHIFT>(sh.t.phiy + (size_t)4 * g * M, 0, nrows - 4 * g, M, Mp, xo, xs, c0);
    const int lr = 4 * g + (lane >> 3);
    const bool mine = (lane & 7) == 0 && lr < nrows;
    if (shift == 0) {
      const bool o = mine && open_rounding(sh, y, lr, xnorm);
      if (mine && !o) put(slot + lr, __fmul_rn((float)y, scale), epoch);
      open |= __ballot_sync(0xffffffffu, o) << i;
    } else if (mine) {
      parts[part * kPartRows + lr] = y;
    }
  }
  if (shift) {
    __syncthreads();
    if (warp == 0) {
      double y = 0.0;
      if (lane < nrows)
        for (int p = 0; p < (1 << shift); ++p) y += parts[p * kPartRows + lane];
      const bool o = lane < nrows && open_rounding(sh, y, lane, xnorm);
      if (lane < nrows && !o) put(slot + lane, __fmul_rn((float)y, scale), epoch);
      open = __ballot_sync(0xffffffffu, o);
    }
  }
  while (open) {
    const int l = __ffs(open) - 1, lr = shift ? l : 4 * (warp + (l & 7) * PW) + (l >> 3);
    open &= open - 1;
    const double y = exact_row(sh, lr, xo, xs);
    if (lane == 0) put(slot + lr, __fmul_rn((float)y, scale), epoch);
  }
}

template <bool STREAM, bool V4>
__device__ __forceinline__ void product(const Shared& sh, int xo, float xs, float xnorm, float scale, u64* slot, uint32_t epoch) {
  const int shift = sh.t.cg_log;
  if (shift == 0) product_split<STREAM, V4, 0>(sh, xo, xs, xnorm, scale, slot, epoch);
  else if (shift == 1) product_split<STREAM, V4, 1>(sh, xo, xs, xnorm, scale, slot, epoch);
  else product_split<STREAM, V4, 2>(sh, xo, xs, xnorm, scale, slot, epoch);
}

// n >= 2 passes with the vectors exchanged between them: y = scale Phi_y x, then y = Phi_y (x / ||x||); x at offset xo,
// xnorm a bound on the first one's length, the results alternate between the two vectors.  A function of its own with nothing else in it, so that no register of the loop
// lives in memory: what is left of the L1 cache beside 226 KB of shared memory does not hold the spilled registers of 512
// threads (measured: 5.7 us a pass instead of 2.9 at M = 1152).
struct PassOut { float x2, lam; };    // of the last pass: ||x||^2, y.x / ||x||
template <bool STREAM, bool V4>
__device__ __noinline__ PassOut passes(Shared& sh, int n, int xo, int yo, float xnorm, float scale, uint32_t epoch, int flip) {
  const int M = sh.t.M;
  u64* const slot = sh.t.slot;
  const int Me = packet_stride(M);
  float xs = 1.f, x2 = 0.f, sum = 0.f;
#pragma unroll 1
  for (int i = 0; i < n; ++i) {
    u64* s = slot + ((epoch & 1u) ? Me : 0);
    product<STREAM, V4>(sh, xo, xs, xnorm, scale, s, epoch);
    scale = 1.f; xnorm = 1.001f;
    x2 = sum;
    if (!V4 || sh.t.cg_log == 0) __syncthreads();
    sum = receive<V4>(s, M, epoch, yo, sh, flip, i + 1 == n ? SUM_DOT : SUM_SQUARES, xo, xs);
    xs = inv_norm(sum);
    const int z = xo; xo = yo; yo = z;
    ++epoch;
    flip ^= 1;
  }
  return PassOut{x2, sum};
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

// squared norm of my row r; sent as exchange `epoch` if `send`.  In fp64 it is finite exactly where the row is.
__device__ __forceinline__ void new_norm(Shared& sh, int r, double n2, bool send, uint32_t epoch) {
  if ((threadIdx.x & 31) != 0) return;
  sh.xi2[r] = (float)n2;
  sh.win[r] = n2 == 0.0 ? 0.f : isfinite(n2) ? fmaxf(sqrtf((float)n2), 1e-19f) * kOrderWindow : INFINITY;
  if (send) put(sh.t.xi + sh.t.row0 + r, (float)n2, epoch);
}

// Squared norms of my rows as they are, sent as exchange `epoch` (later steps get them from the update).
__device__ __noinline__ void row_norms(Shared& sh, uint32_t epoch) {
  const Team& t = sh.t;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int M = t.M, Mp = t.Mp;
  for (int r = warp; r < t.nrows; r += PW) {
    const float* row = r < t.ncached ? psm + t.rows + r * Mp : t.phiy + (size_t)r * M;
    double acc = 0.0;
    if ((M & 3) == 0) {
      for (int c = lane; c < (M >> 2); c += 32) {
        const float4 q = reinterpret_cast<const float4*>(row)[c];
        acc = fma((double)q.x, (double)q.x, acc); acc = fma((double)q.y, (double)q.y, acc);
        acc = fma((double)q.z, (double)q.z, acc); acc = fma((double)q.w, (double)q.w, acc);
      }
    } else {
      for (int c = lane; c < M; c += 32) acc = fma((double)row[c], (double)row[c], acc);
    }
    new_norm(sh, r, warp_sum(acc), true, epoch);
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
// and the weights of the coherent set (Eqs. 48-49) into the vector at yo; returns the size of the set and a bound on ||w||.
struct Aligned { int cnt; float wnorm; };
template <bool STREAM, bool V4>
__device__ __noinline__ Aligned correlate(Shared& sh, int mp, int xo, int yo, uint32_t epoch, bool keep) {
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
  receive<V4>(s, M, epoch, xo, sh, 0, SUM_NONE, 0, 0.f);
  ++epoch;
  s = t.slot + ((epoch & 1u) ? Me : 0);
  const float xi_mx = sqrtf(value_of(peek(t.xi + mp)));
  product<STREAM, V4>(sh, xo, 1.f, 1.001f * xi_mx, 1.f, s, epoch);
  if (L->init == FW_INIT_MAXCOL) {
    for (int m = tid; m < M; m += PT) psm[yo + m] = (m == mp) ? 1.f : 0.f;
    for (int p0 = tid; 2 * (p0 & ~31) < M; p0 += kPairs * PT) {       // received all the same: the slots alternate on that
      float2 v[kPairs];
      poll(s, p0, M, epoch, sh, v);
    }
    __syncthreads();
    return Aligned{1, 1.f};
  }
  const float c_rel = L->c_rel, c_abs = L->c_abs;
  int cnt = 0;
  float w2 = 0.f;
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
        cnt += in ? 1 : 0;                                                           \
        w2 = fmaf(q, q, w2);                                                         \
        if (keep) L->wvec[i] = q;                                                    \
      }
      FW_WEIGHT(x, xa, m)
      FW_WEIGHT(y, xb, m + 1)
#undef FW_WEIGHT
    }
  }
  cnt = __reduce_add_sync(0xffffffffu, cnt);
  w2 = warp_sum(w2);
  if ((tid & 31) == 0) { sh.key[tid >> 5] = (uint32_t)cnt; sh.idx[tid >> 5] = __float_as_uint(w2); }
  __syncthreads();
  cnt = (int)__reduce_add_sync(0xffffffffu, (tid & 31) < PW ? sh.key[tid & 31] : 0u);
  w2 = warp_sum((tid & 31) < PW ? __uint_as_float(sh.idx[tid & 31]) : 0.f);
  return Aligned{cnt, 1.001f * sqrtf(w2)};
}

// Phi_y += a (v u^T + u v^T) + a^2 lambda_e v v^T on my rows, one rounding per operation and symmetric; v = inv x, x at
// offset xo, u at yo.  Squared norms of the new rows, sent as exchange `epoch` if `send`.
__device__ __noinline__ void update_rows(Shared& sh, int xo, int yo, float inv, float aa, float lam_e, bool send, uint32_t epoch) {
  const Team& t = sh.t;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int M = t.M, Mp = t.Mp, nrows = t.nrows, row0 = t.row0;
  const float a2l = aa * aa * lam_e;
  for (int r = warp; r < nrows; r += PW) {
    const float vi = psm[xo + row0 + r] * inv, ui = psm[yo + row0 + r];
    float* row = r < t.ncached ? psm + t.rows + r * Mp : t.phiy + (size_t)r * M;
    double acc = 0.0;
    if ((M & 3) == 0) {
      const u64 z = pack2(sh.negz, sh.negz), a2 = pack2(aa, aa), l2 = pack2(a2l, a2l), vi2 = pack2(vi, vi), ui2 = pack2(ui, ui);
#pragma unroll 2
      for (int c = lane; c < (M >> 2); c += 32) {
        float4 p = reinterpret_cast<const float4*>(row)[c];
        float4 v = *reinterpret_cast<const float4*>(psm + xo + 4 * c);
        const float4 u = *reinterpret_cast<const float4*>(psm + yo + 4 * c);
        v.x *= inv; v.y *= inv; v.z *= inv; v.w *= inv;
        p = rank2(p, vi2, ui2, pack2(v.x, v.y), pack2(v.z, v.w), pack2(u.x, u.y), pack2(u.z, u.w), a2, l2, z);
        reinterpret_cast<float4*>(row)[c] = p;
        acc = fma((double)p.x, (double)p.x, acc); acc = fma((double)p.y, (double)p.y, acc);
        acc = fma((double)p.z, (double)p.z, acc); acc = fma((double)p.w, (double)p.w, acc);
      }
    } else {
      for (int c = lane; c < M; c += 32) {
        const float vj = psm[xo + c] * inv, uj = psm[yo + c];
        const float p = __fadd_rn(row[c], __fadd_rn(__fmul_rn(aa, __fadd_rn(__fmul_rn(vi, uj), __fmul_rn(ui, vj))),
                                                    __fmul_rn(a2l, __fmul_rn(vi, vj))));
        row[c] = p;
        acc = fma((double)p, (double)p, acc);
      }
    }
    new_norm(sh, r, warp_sum(acc), send, epoch);
  }
}

// All steps of one layer by its team.
__device__ __noinline__ void run_layer(const TeamArgs& a, Shared& sh, int li) {
  const Team& t = sh.t;
  const int tid = threadIdx.x;
  uint32_t e = (uint32_t)t.L->iscal[IS_EXCHANGE];              // the layer's last exchange
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
  }
  __syncthreads();
  row_norms(sh, ++e);
  bool updated = false;
#pragma unroll 1
  for (int step = 0; step < a.K; ++step) {
    const int mp = receive_argmax(sh, e);
    const int Mp = t.Mp, M = t.M, P = a.P;
    const bool stream = t.ncached < t.nrows, v4 = (M & 3) == 0;
    const bool keep = a.last && step + 1 == a.K && t.sub == 0;
    const Aligned al = stream ? (v4 ? correlate<true, true>(sh, mp, 0, Mp, e + 1, keep) : correlate<true, false>(sh, mp, 0, Mp, e + 1, keep))
                           : (v4 ? correlate<false, true>(sh, mp, 0, Mp, e + 1, keep) : correlate<false, false>(sh, mp, 0, Mp, e + 1, keep));
    // aligned average, P power iterations y = Phi_y (x / ||x||), then u = Phi_y v with v = x / ||x|| (Eqs. 49-50)
    const int cnt = al.cnt;
    const float inv_cnt = cnt > 0 ? 1.f / (float)cnt : 0.f;
    const PassOut o = stream ? (v4 ? passes<true, true>(sh, P + 2, Mp, 0, al.wnorm, inv_cnt, e + 3, flip) : passes<true, false>(sh, P + 2, Mp, 0, al.wnorm, inv_cnt, e + 3, flip))
                             : (v4 ? passes<false, true>(sh, P + 2, Mp, 0, al.wnorm, inv_cnt, e + 3, flip) : passes<false, false>(sh, P + 2, Mp, 0, al.wnorm, inv_cnt, e + 3, flip));
    flip ^= P & 1;
    e += (uint32_t)P + 4u;
    const int xo = (P & 1) ? Mp : 0, yo = Mp - xo;               // x and u of the last pass
    const float inv = inv_norm(o.x2), lam_e = o.lam;              // Eq. 36
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
      update_rows(sh, xo, yo, inv, aa, lam_e, more, e);
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
// floats of the partial sums; R: rows per CTA.  Pairs of M <= 8192 entries, eight to a partial sum of a norm.
__host__ __device__ inline int team_part(int M, int R) { return (M & 3) ? 512 : (R <= kPartRows ? 2 * 4 * kPartRows : 0); }
// rows that fit beside the two vectors and the partial sums, whole groups of four
__host__ __device__ inline int team_cache(int M, int R) {
  const int Mp = (M + 3) & ~3;
  return (((int)(kSmem / sizeof(float)) - 2 * Mp - team_part(M, R)) / Mp) & ~3;
}

__global__ void __launch_bounds__(PT, 1) recursion_team_kernel(const __grid_constant__ TeamArgs a) {
  dep_sync();
  __shared__ Shared sh;
  if (threadIdx.x == 0) { sh.fail = 0; sh.negz = -0.f; }
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
        t.ncached = min(t.nrows, team_cache(M, R));
        t.part = 2 * t.Mp;
        t.rows = t.part + team_part(M, R);
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

// what a pass costs on n CTAs, to compare splits: a row from L2 or HBM takes about 2.7 times one in shared memory
double team_cost(int M, int n) {
  const int R = team_rows(M, n), fit = team_cache(M, R), cached = std::min(R, fit);
  return (cached + 2.7 * (R - cached)) * M;
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

cudaError_t launch_recursion_team(const GroupDev& g, const PtrTable& traces, const int* layer_M, int k0, int K, int P,
                                  bool last, cudaStream_t s) {
  static SmemAttrCache attr;
  thread_local TeamPlan plan;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) dev = 0;
  e = ensure_dyn_smem(recursion_team_kernel, kSmem, attr);
  if (e != cudaSuccess) return e;
  if (plan.dev != dev || plan.n != g.n || memcmp(plan.dims, layer_M, g.n * sizeof(int)) != 0) {
    make_plan(plan, layer_M, g.n, sm_count());
    plan.dev = dev;
  }
  for (int i = 0; i < g.n; ++i)      // the tables of a CTA's rows (86 SMs are enough for the largest M)
    if (team_rows(layer_M[i], plan.cnt[i]) > kMaxRows) return cudaErrorInvalidConfiguration;
  TeamArgs a;
  memset(&a, 0, sizeof(a));
  a.g = g; a.traces = traces; a.k0 = k0; a.K = K; a.P = P; a.nwaves = plan.waves; a.last = last ? 1 : 0;
  int ctas = 0;
  for (int i = 0; i < g.n; ++i) {
    a.wave[i] = plan.wave[i]; a.first[i] = plan.first[i]; a.n[i] = plan.cnt[i];
    ctas = std::max(ctas, plan.first[i] + plan.cnt[i]);
  }
  void* args[] = {&a};
  ProfScope ps(FW_PROF_RECUR_MV, s);
  return cudaLaunchCooperativeKernel((void*)recursion_team_kernel, dim3(ctas), dim3(PT), args, kSmem, s);
}

}  // namespace fw
