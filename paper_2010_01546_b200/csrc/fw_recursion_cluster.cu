// On-chip recursion for small layers (Sec. 4): a layer's whitened covariance Phi_y
// stays on chip for all steps of a launch, each warp's rows in its registers (row m'
// of a step is sent round as column m', four entries a warp).  The launch uses
// thread-block clusters; a layer takes n = 1 ... 16 consecutive CTAs of one
// cluster (at least as many as its rows need; more while the clusters of one wave
// allow and the layer is the launch's slowest).  CTA `sub` of a layer owns a slab
// of rows; every pass of a step is a slab-times-vector product.  The passes are
// chained as a dataflow: each warp pushes its slice of a result straight into all
// CTAs' copies of the vector with asynchronous remote stores that count bytes on
// the receiver's mbarrier, and every warp waits on its own CTA's barrier -- no
// block or cluster barrier separates the power iterations.  T and Q are not
// needed by a step, so a step only records its v_e and a_e; after the last one
// each warp loads its rows of T^T, forms t = T^T v_e step by step (t goes round on a
// barrier of its own), and T and Q take the rank-one terms in step order (Eqs. 42, 44).
//
// What bounds it: the chain of P + 5 dependent exchanges per step.  A pass reads
// only the vector from shared memory (rows in registers: at M = 576 the slab's 83
// KB per pass alone would take 0.35 us of shared-memory bandwidth), so what is
// left is the latency of the reduction, the remote store and the wait.
//
// Buffer reuse is safe without further synchronisation: a CTA can send exchange
// e + 1 only after it received every warp's slice of exchange e, and a warp sends
// its slice after its last read of the pass's input; vectors alternate and the
// barriers are double-buffered.  Warps that own no rows take no part in the steps.
//
// Dot products are accumulated in fp32 (rows are at most 624 long and split over
// two accumulators per lane); rank updates are evaluated symmetrically.
#include <cooperative_groups.h>
#include <algorithm>
#include <cstring>
#include <mutex>

#include "fw_internal.h"
#include "fw_lanes.cuh"
#include "fw_sm100.cuh"

namespace cg = cooperative_groups;

namespace fw {
namespace {

using sm100::smem_u32;

constexpr int CLMAX = 16;          // largest cluster (beyond 8: non-portable size)
constexpr int CT = 512;            // threads per CTA
constexpr int CW = CT / 32;        // warps per CTA
constexpr int kMaxIt = 5;          // float4 columns per lane, at most
constexpr int kMaxM = 624;         // longest row whose products are summed in fp32; longer ones take teams of CTAs and fp64 sums
constexpr int kSolo = 64;          // largest layer that takes one CTA and eight lanes a row
constexpr int KH = 8;              // steps that T and Q take together
constexpr size_t kSmemLimit = 64 * 1024;   // the vectors of the longest row: 22 of 16 slabs of at most 43 entries

// A warp owns one group of four rows (up to kMaxIt float4 columns per lane: 80 registers) or, for rows of at most 256
// entries, two (64 registers).
__host__ __device__ constexpr int max_groups(int it) { return it <= 2 ? 2 : 1; }

struct ClusterArgs {
  GroupDev g;
  PtrTable traces;
  int32_t first_cta[FW_MAX_GROUP];   // first CTA of each layer (a layer never straddles a cluster)
  int32_t ncta[FW_MAX_GROUP];        // CTAs of each layer: 1 ... cluster size
  int32_t k0, K, P;                  // first step of the call in this launch, steps, power iterations
  int32_t last;                      // this launch ends the call
};

// shared-memory address of the same variable in CTA `rank` of the cluster
__device__ __forceinline__ uint32_t map_cluster(uint32_t saddr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(saddr), "r"(rank));
  return r;
}
// asynchronous 16-byte store into a CTA's shared memory; its mbarrier counts the bytes.  One message carries four
// results: the receiver's barrier takes a few clocks per message, so the count of messages, not their size, is what
// an exchange costs.
__device__ __forceinline__ void st_async_v4(uint32_t raddr, float4 v, uint32_t rbar) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];"
               ::"r"(raddr), "r"(__float_as_uint(v.x)), "r"(__float_as_uint(v.y)), "r"(__float_as_uint(v.z)),
                 "r"(__float_as_uint(v.w)), "r"(rbar) : "memory");
}

// dynamic shared memory: [xi2][cvec][wvec][two power-iteration vectors][uvec][vh: KH][th: KH], vectors
// of Mv floats: what n slices of R results fill, and at least whole trips of a warp over the columns
extern __shared__ __align__(16) float csm[];

// What a CTA knows about its layer; lives in shared memory (the threads' registers hold matrix rows).
struct Slab {
  // offsets into the dynamic shared memory (not pointers: the compiler then knows which memory they point to)
  int xi2, cvec, wvec, buf0, uvec;   // vectors of Mv floats; buf0: two, Mv apart
  int vh, th;     // v_e and t of the steps, KH vectors each
  int M, Mp;      // matrix size, padded row length
  int Mv;         // vector length in shared memory
  int R;          // rows per CTA, a multiple of four (rows past the matrix are zero rows)
  int row0;       // my first row
  int n;          // CTAs of this layer
  int sub;        // my index among them
  uint32_t tx;    // bytes of one exchanged vector
  int maxcol;     // start vector: largest column instead of the alignment
  float c_rel, c_abs, delta, eps, lam_bar;
  float ah[KH];   // a_e of the steps
  float negz;     // -0
  int fail;       // set once a bounded wait of this CTA gave up
};
// The parts of it every pass needs, in registers.
struct Link {
  uint32_t rdelta;  // lane p < n: cluster address of CTA p's shared memory minus this CTA's own
  uint32_t bar0;    // two exchange barriers and the one of all steps' t, 8 bytes apart
  int n;
  int active;       // threads of the warps that own rows; the others take no part in the steps
};

// barriers among the warps that own rows
__device__ __forceinline__ void rows_sync(const Link& l) { asm volatile("bar.sync 1, %0;" ::"r"(l.active) : "memory"); }

// Arms the barrier of exchange e (one thread) ahead of the pass, off the chain.
__device__ __forceinline__ void arm(const Link& l, uint32_t e, uint32_t bytes) {
  if (l.n > 1 && threadIdx.x == 0) sm100::mbar_expect_tx(l.bar0 + ((e & 1) << 3), bytes);
}
// Bounded wait for exchange e.  Every warp waits for itself.  Once a wait has given up no later wait of the CTA
// blocks: the CTA runs on with stale data to the end of the call, so that its block barriers and its peers stay in
// step, and reports the time-out there.  A layer on one CTA exchanges through its own shared memory.
__device__ __forceinline__ void wait_bar(uint32_t bar, uint32_t parity, int* fail) {
  if (sm100::mbar_try_wait(bar, parity)) return;
  if (*(volatile int*)fail) return;
  for (uint32_t i = 0; i < sm100::kSpinLimit; ++i)
    if (sm100::mbar_try_wait(bar, parity)) return;
  *(volatile int*)fail = 1;
}
__device__ __forceinline__ void wait_exchange(const Link& l, uint32_t e, int* fail) {
  if (l.n == 1) rows_sync(l);
  else wait_bar(l.bar0 + ((e & 1) << 3), (e >> 1) & 1, fail);
}
// four results of a group into `tgt` of every CTA of the layer
__device__ __forceinline__ void send4(const Link& l, float* tgt, float4 v, uint32_t e) {
  const int lane = threadIdx.x & 31;
  if (l.n == 1) {
    if (lane == 0) *reinterpret_cast<float4*>(tgt) = v;
  } else if (lane < l.n) {
    st_async_v4(smem_u32(tgt) + l.rdelta, v, l.bar0 + ((e & 1) << 3) + l.rdelta);
  }
}

// One pass: y = (my rows) x, sent to `dst` (the slot of the warp's first group in the result vector) of every CTA of the
// layer.  SCALE: y times `scale`.  NORM and UNIT take x as it was sent times `scale`: a power iteration's y = Phi_y x / ||x|| is
// sent without the 1 / ||x||, which a receiver applies to the entries it loads.  NORM returns ||scale x||^2, reduced once y has gone,
// so that the norm's reduction and root run beside the exchange.  UNIT: the rows times scale x / ||scale x||, the norm first;
// returns its square.  SELF: squared norms of the rows themselves.  Sums are packed pairs: half the instructions, every
// product and sum rounded as before.  Recursion of the ResNet-20-shaped set (K = 4, P = 16): 124 us with scalar sums, 107
// packed; 64 layers of M = 256, K = 8, P = 32: 292 and 262.  One warp's norm for the whole CTA, arming the exchange's barrier
// when it is there, took 114 and 296.
enum { PASS_SELF, PASS_SCALE, PASS_NORM, PASS_UNIT };
template <int MODE, int NG, int IT>
__device__ __forceinline__ float pass(const Quad (&a)[4 * NG][IT], const float* x, float scale, const Link& l,
                                      float* dst, uint32_t e) {
  const int lane = threadIdx.x & 31;
  const float4* x4 = reinterpret_cast<const float4*>(x);
  u64 acc[4 * NG], nn = pack2(0.f, 0.f);
#pragma unroll
  for (int q = 0; q < 4 * NG; ++q) acc[q] = pack2(0.f, 0.f);
  const u64 sc = pack2(scale, scale);
  float n2 = 0.f;
  u64 inv = 0;
  if (MODE == PASS_UNIT) {
#pragma unroll
    for (int k = 0; k < IT; ++k) {
      const float4 b = x4[lane + 32 * k];
      const u64 lo = times2(pack2(b.x, b.y), sc), hi = times2(pack2(b.z, b.w), sc);
      nn = fmadd2(hi, hi, fmadd2(lo, lo, nn));
    }
    float n0, n1;
    unpack2(nn, n0, n1);
    n2 = warp_sum(n0 + n1);
    const float i = inv_norm(n2);
    inv = pack2(i, i);
  }
#pragma unroll
  for (int k = 0; k < IT; ++k) {
    u64 lo = 0, hi = 0;
    if (MODE != PASS_SELF) {
      const float4 b = x4[lane + 32 * k];
      lo = pack2(b.x, b.y); hi = pack2(b.z, b.w);
    }
    if (MODE == PASS_NORM || MODE == PASS_UNIT) { lo = times2(lo, sc); hi = times2(hi, sc); }
    if (MODE == PASS_UNIT) { lo = times2(lo, inv); hi = times2(hi, inv); }
    if (MODE == PASS_NORM) nn = fmadd2(hi, hi, fmadd2(lo, lo, nn));
#pragma unroll
    for (int q = 0; q < 4 * NG; ++q) {
      const Quad v = a[q][k];
      acc[q] = fmadd2(v.hi, MODE == PASS_SELF ? v.hi : hi, fmadd2(v.lo, MODE == PASS_SELF ? v.lo : lo, acc[q]));
    }
  }
#pragma unroll
  for (int g = 0; g < NG; ++g) {
    float y[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      float y0, y1;
      unpack2(acc[4 * g + q], y0, y1);
      y[q] = y0 + y1;
    }
    float4 v = warp_sum4(y[0], y[1], y[2], y[3]);
    if (MODE == PASS_SCALE) { v.x *= scale; v.y *= scale; v.z *= scale; v.w *= scale; }
    send4(l, dst + 4 * CW * g, v, e);
  }
  if (MODE == PASS_NORM) {
    float n0, n1;
    unpack2(nn, n0, n1);
    n2 = warp_sum(n0 + n1);
  }
  return n2;
}

// m' = argmax xi, lowest index on ties (Eq. 46).  Every warp finds it for itself: squared norms are not negative, so
// their bit patterns are ordered; a NaN never wins.
__device__ __forceinline__ int argmax_xi(const Slab& s) {
  const int lane = threadIdx.x & 31;
  uint32_t best = 0, bi = 0;
  for (int c = lane; c < (s.Mp >> 2); c += 32) {
    const float4 x = reinterpret_cast<const float4*>(csm + s.xi2)[c];
#define FW_CAND(X, o)                                                                                     \
    {                                                                                                     \
      const uint32_t k = (X) >= 0.f && 4 * c + (o) < s.M ? __float_as_uint(X) + 1u : 0u;                   \
      if (k > best) { best = k; bi = 4 * c + (o); }                                                       \
    }
    FW_CAND(x.x, 0) FW_CAND(x.y, 1) FW_CAND(x.z, 2) FW_CAND(x.w, 3)
#undef FW_CAND
  }
  const uint32_t top = __reduce_max_sync(0xffffffffu, best);
  bi = __reduce_min_sync(0xffffffffu, best == top ? bi : 0xffffffffu);
  return top == 0 || bi >= (uint32_t)s.M ? 0 : (int)bi;
}

// Row m' of Phi_y into wvec of every CTA of the layer (exchange e).  Phi_y is exactly symmetric, so every warp sends the entries of
// its rows in column m': a message of four entries a warp like any other exchange, where the owner of row m' sending it to
// all alone took 4900 clocks (M = 576 on 12 CTAs: 1728 messages of one SM).
template <int NG, int IT>
__device__ __forceinline__ void send_column(const Quad (&a)[4 * NG][IT], int mp, const Link& l, float* dst, uint32_t e) {
  const int k0 = mp >> 7, from = (mp >> 2) & 31, c = mp & 3;
#pragma unroll
  for (int g = 0; g < NG; ++g) {
    float y[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      float x = 0.f;
#pragma unroll
      for (int k = 0; k < IT; ++k) {
        if (k == k0) {
          float even, odd;
          unpack2(c < 2 ? a[4 * g + q][k].lo : a[4 * g + q][k].hi, even, odd);
          x = c & 1 ? odd : even;
        }
      }
      y[q] = __shfl_sync(0xffffffffu, x, from);
    }
    send4(l, dst + 4 * CW * g, make_float4(y[0], y[1], y[2], y[3]), e);
  }
}

// Weights of the coherent set into wvec (Eqs. 48-49); returns the size of the set
__device__ __forceinline__ int align_weights(Slab& s, const Link& l, int mp) {
  if (s.maxcol) {
    rows_sync(l);                     // wvec may still be read by a slower warp
    for (int m = threadIdx.x; m < s.Mp; m += l.active) csm[s.wvec + m] = (m == mp) ? 1.f : 0.f;
    rows_sync(l);
    return 1;
  }
  const float xi_mp = sqrtf(csm[s.xi2 + mp]), c_rel = s.c_rel, c_abs = s.c_abs;
  int cnt = 0;
  for (int base = 0; base < s.Mp; base += l.active) {
    const int m = base + (int)threadIdx.x;
    int in = 0;
    if (m < s.Mp) {
      float wv = 0.f;
      if (m < s.M) {
        const float c = csm[s.cvec + m];
        const float thr = fmaxf(c_rel * xi_mp * sqrtf(csm[s.xi2 + m]), c_abs);
        in = fabsf(c) >= thr;       // false for NaN
        wv = in ? (1.f / c) : 0.f;
      }
      csm[s.wvec + m] = wv;
    }
    int n;
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.s32 p, %1, 0;\n\tbarrier.cta.red.popc.aligned.u32 %0, 1, %2, p;\n\t}"
                 : "=r"(n) : "r"(in), "r"(l.active) : "memory");
    cnt += n;
  }
  return cnt;
}

// rows of a row-major matrix in global memory <-> the registers of the warp that owns them; V4: rows of whole float4s
template <int NG, int IT, bool V4>
__device__ __forceinline__ void load_rows(Quad (&a)[4 * NG][IT], const float* G, const Slab& s) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int M = s.M;
#pragma unroll
  for (int q = 0; q < 4 * NG; ++q) {
    const int i = s.row0 + 4 * (warp + CW * (q >> 2)) + (q & 3);
    const float* row = G + (size_t)i * M;
#pragma unroll
    for (int k = 0; k < IT; ++k) {
      const int c = lane + 32 * k;
      float4 r = make_float4(0.f, 0.f, 0.f, 0.f);
      if (i < M) {
        if (V4) {
          if (4 * c < M) r = reinterpret_cast<const float4*>(row)[c];
        } else {
          if (4 * c < M) r.x = row[4 * c];
          if (4 * c + 1 < M) r.y = row[4 * c + 1];
          if (4 * c + 2 < M) r.z = row[4 * c + 2];
          if (4 * c + 3 < M) r.w = row[4 * c + 3];
        }
      }
      a[q][k].lo = pack2(r.x, r.y); a[q][k].hi = pack2(r.z, r.w);
    }
  }
}
// ROUND: rounded to the TF32 grid
template <int NG, int IT, bool V4, bool ROUND = false>
__device__ __forceinline__ void store_rows(const Quad (&a)[4 * NG][IT], float* G, const Slab& s) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int M = s.M;
#pragma unroll
  for (int q = 0; q < 4 * NG; ++q) {
    const int i = s.row0 + 4 * (warp + CW * (q >> 2)) + (q & 3);
    if (i >= M) continue;
    float* row = G + (size_t)i * M;
#pragma unroll
    for (int k = 0; k < IT; ++k) {
      const int c = lane + 32 * k;
      float4 r;
      unpack2(a[q][k].lo, r.x, r.y);
      unpack2(a[q][k].hi, r.z, r.w);
      if (ROUND) r = make_float4(sm100::tf32_rna(r.x), sm100::tf32_rna(r.y), sm100::tf32_rna(r.z), sm100::tf32_rna(r.w));
      if (V4) {
        if (4 * c < M) reinterpret_cast<float4*>(row)[c] = r;
      } else {
        if (4 * c < M) row[4 * c] = r.x;
        if (4 * c + 1 < M) row[4 * c + 1] = r.y;
        if (4 * c + 2 < M) row[4 * c + 2] = r.z;
        if (4 * c + 3 < M) row[4 * c + 3] = r.w;
      }
    }
  }
}

// The K recorded steps in T and Q: T first (t of step k comes from T after step k - 1), then Q, with the operations on every
// element in step order; smooth: Qs <- beta Qs + (1 - beta) Q (Eq. 35).
template <int NG, int IT, bool V4>
__device__ __forceinline__ void apply_steps(Slab& s, const Link& l, const LayerDev* L, int K, bool smooth) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, M = s.M;
  int live = 0;
#pragma unroll 1
  for (int k = 0; k < K; ++k) live += s.ah[k] != 0.f ? 1 : 0;
  if (!live && !smooth) return;
  Quad a[4 * NG][IT];
  if (live) {
    load_rows<NG, IT, V4>(a, L->Tt, s);
#pragma unroll 1
    for (int k = 0; k < K; ++k) {
      const float ak = s.ah[k];
      if (ak == 0.f) continue;
      const float4* v4 = reinterpret_cast<const float4*>(csm + s.vh + k * s.Mv);
      u64 acc[4 * NG];
#pragma unroll
      for (int q = 0; q < 4 * NG; ++q) acc[q] = pack2(0.f, 0.f);
#pragma unroll
      for (int it = 0; it < IT; ++it) {
        const float4 b = v4[lane + 32 * it];
        const u64 lo = pack2(b.x, b.y), hi = pack2(b.z, b.w);
#pragma unroll
        for (int q = 0; q < 4 * NG; ++q) acc[q] = fmadd2(a[q][it].hi, hi, fmadd2(a[q][it].lo, lo, acc[q]));
      }
      u64 at[4 * NG];
#pragma unroll
      for (int g = 0; g < NG; ++g) {
        float y[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          float y0, y1;
          unpack2(acc[4 * g + q], y0, y1);
          y[q] = y0 + y1;
        }
        const float4 t = warp_sum4(y[0], y[1], y[2], y[3]);
        float* tgt = csm + s.th + k * s.Mv + s.row0 + 4 * (warp + CW * g);
        if (l.n == 1) {
          if (lane == 0) *reinterpret_cast<float4*>(tgt) = t;
        } else if (lane < l.n) {
          st_async_v4(smem_u32(tgt) + l.rdelta, t, l.bar0 + 16 + l.rdelta);
        }
        at[4 * g] = pack2(ak * t.x, ak * t.x); at[4 * g + 1] = pack2(ak * t.y, ak * t.y);
        at[4 * g + 2] = pack2(ak * t.z, ak * t.z); at[4 * g + 3] = pack2(ak * t.w, ak * t.w);
      }
#pragma unroll
      for (int it = 0; it < IT; ++it) {
        const float4 b = v4[lane + 32 * it];
        const u64 lo = pack2(b.x, b.y), hi = pack2(b.z, b.w);
#pragma unroll
        for (int q = 0; q < 4 * NG; ++q) { a[q][it].lo = fmadd2(at[q], lo, a[q][it].lo); a[q][it].hi = fmadd2(at[q], hi, a[q][it].hi); }
      }
    }
    store_rows<NG, IT, V4>(a, L->Tt, s);
    if (V4 && L->round_t) store_rows<NG, IT, true, true>(a, L->tmp, s);
  }
  load_rows<NG, IT, V4>(a, L->Q, s);
  if (live) {
    if (l.n == 1) {
      rows_sync(l);
    } else {
      if (threadIdx.x == 0) sm100::mbar_expect_tx(l.bar0 + 16, (uint32_t)live * s.tx);
      wait_bar(l.bar0 + 16, 0, &s.fail);
    }
    const u64 z = pack2(s.negz, s.negz);
#pragma unroll 1
    for (int k = 0; k < K; ++k) {
      const float ak = s.ah[k];
      if (ak == 0.f) continue;
      const float aq = ak * (ak + 2.f);
      const u64 aq2 = pack2(aq, aq);
      const float* tk = csm + s.th + k * s.Mv;
      u64 ti[4 * NG];
#pragma unroll
      for (int q = 0; q < 4 * NG; ++q) {
        const float t = tk[s.row0 + 4 * (warp + CW * (q >> 2)) + (q & 3)];
        ti[q] = pack2(t, t);
      }
#pragma unroll
      for (int it = 0; it < IT; ++it) {
        const float4 b = reinterpret_cast<const float4*>(tk)[lane + 32 * it];
        const u64 lo = pack2(b.x, b.y), hi = pack2(b.z, b.w);
#pragma unroll
        for (int q = 0; q < 4 * NG; ++q) {
          a[q][it].lo = add2(a[q][it].lo, mul2(aq2, mul2(ti[q], lo, z), z));
          a[q][it].hi = add2(a[q][it].hi, mul2(aq2, mul2(ti[q], hi, z), z));
        }
      }
    }
    if (!*(volatile int*)&s.fail) store_rows<NG, IT, V4>(a, L->Q, s);
  }
  if (smooth) {
    const float beta = L->beta, ob = 1.f - beta;
    float* Qs = L->Qs;
#pragma unroll
    for (int q = 0; q < 4 * NG; ++q) {
      const int i = s.row0 + 4 * (warp + CW * (q >> 2)) + (q & 3);
      if (i >= M) continue;
      float* row = Qs + (size_t)i * M;
#pragma unroll
      for (int it = 0; it < IT; ++it) {
        const int c = 4 * (lane + 32 * it);
        if (c >= M) continue;
        float4 r;
        unpack2(a[q][it].lo, r.x, r.y);
        unpack2(a[q][it].hi, r.z, r.w);
        if (V4) {
          float4 o = *reinterpret_cast<float4*>(row + c);
          o.x = fmaf(beta, o.x, ob * r.x); o.y = fmaf(beta, o.y, ob * r.y);
          o.z = fmaf(beta, o.z, ob * r.z); o.w = fmaf(beta, o.w, ob * r.w);
          *reinterpret_cast<float4*>(row + c) = o;
        } else {
          row[c] = fmaf(beta, row[c], ob * r.x);
          if (c + 1 < M) row[c + 1] = fmaf(beta, row[c + 1], ob * r.y);
          if (c + 2 < M) row[c + 2] = fmaf(beta, row[c + 2], ob * r.z);
          if (c + 3 < M) row[c + 3] = fmaf(beta, row[c + 3], ob * r.w);
        }
      }
    }
  }
}

// All steps of a launch for a warp that owns NG groups of four rows of IT float4 columns per lane; from Phi_y in global
// memory and back.  tr: where the trace of the launch's first step goes, or null.
template <int NG, int IT>
__device__ __noinline__ void run_steps(Slab& s, const Link l, const LayerDev* L, float* tr, int K, int P, bool last) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int slot = s.row0 + 4 * warp;       // the warp's first group in a result vector
  const uint32_t tx = s.tx;
  Quad a[4 * NG][IT];
  if ((s.M & 3) == 0) load_rows<NG, IT, true>(a, L->Phiy, s);
  else load_rows<NG, IT, false>(a, L->Phiy, s);
  sm100::cluster_wait();                       // every CTA is ready to receive
  uint32_t e = 0;                              // exchanges so far
  for (int step = 0; step < K; ++step) {
    // S1: squared column norms (= row norms, Phi_y is exactly symmetric)             (Eq. 45)
    arm(l, e, tx);
    pass<PASS_SELF, NG, IT>(a, nullptr, 1.f, l, csm + s.xi2 + slot, e);
    wait_exchange(l, e, &s.fail); ++e;
    // S2: m' = argmax xi, x = row m' of Phi_y, c = Phi_y x                            (Eqs. 46-47)
    const int mp = argmax_xi(s);
    arm(l, e, tx);
    send_column<NG, IT>(a, mp, l, csm + s.wvec + slot, e);
    wait_exchange(l, e, &s.fail); ++e;
    arm(l, e, tx);
    pass<PASS_SCALE, NG, IT>(a, csm + s.wvec, 1.f, l, csm + s.cvec + slot, e);
    wait_exchange(l, e, &s.fail); ++e;
    // S3: coherent set and aligned average                                          (Eqs. 48-49)
    arm(l, e, tx);
    const int cnt = align_weights(s, l, mp);
    pass<PASS_SCALE, NG, IT>(a, csm + s.wvec, cnt > 0 ? 1.f / (float)cnt : 0.f, l, csm + s.buf0 + slot, e);
    wait_exchange(l, e, &s.fail); ++e;
    // S4: P power iterations u = Phi_y (prev / ||prev||); prev is sc times the vector at xo
    int xo = s.buf0, yo = xo + s.Mv;
    float sc = 1.f;
    for (int p = 0; p < P; ++p) {
      arm(l, e, tx);
      sc = inv_norm(pass<PASS_NORM, NG, IT>(a, csm + xo, sc, l, csm + yo + slot, e));
      wait_exchange(l, e, &s.fail); ++e;
      const int t = xo; xo = yo; yo = t;
    }
    // S5: v = prev/||prev|| (Eq. 50), u = Phi_y v, lambda_e = v.u (Eq. 36)
    const float* x = csm + xo;
    arm(l, e, tx);
    const float n2 = pass<PASS_UNIT, NG, IT>(a, x, sc, l, csm + s.uvec + slot, e);
    const float inv = inv_norm(n2);
    float* vh = csm + s.vh + step * s.Mv;
    wait_exchange(l, e, &s.fail); ++e;
    float l0 = 0.f, l1 = 0.f;
    const float4* x4 = reinterpret_cast<const float4*>(x);
    const float4* u4 = reinterpret_cast<const float4*>(csm + s.uvec);
#pragma unroll
    for (int k = 0; k < IT; ++k) {
      const float4 xv = x4[lane + 32 * k], uv = u4[lane + 32 * k];
      const float4 vv = make_float4(xv.x * sc * inv, xv.y * sc * inv, xv.z * sc * inv, xv.w * sc * inv);
      l0 = fmaf(vv.x, uv.x, l0); l1 = fmaf(vv.y, uv.y, l1);
      l0 = fmaf(vv.z, uv.z, l0); l1 = fmaf(vv.w, uv.w, l1);
      if (warp == 0) reinterpret_cast<float4*>(vh)[lane + 32 * k] = vv;      // every CTA keeps the whole vector for T
    }
    const float lam_e = warp_sum(l0 + l1);
    // S6: g_e, a_e (Eqs. 40-41), rank update of Phi_y.  All warps of all CTAs sum in the same order, so they hold the
    // same bits.
    const bool ok = cnt > 0 && n2 > 0.f && isfinite(n2) && isfinite(lam_e);
    float g_e = 1.f, aa = 0.f;
    if (ok) {
      g_e = s.delta * s.lam_bar / fmaxf(lam_e, s.eps);
      aa = sqrtf(g_e) - 1.f;
    }
    // Phi_y += a (v u^T + u v^T) + a^2 lambda_e v v^T, symmetric in (i, j)
    if (aa != 0.f) {
      const u64 z = pack2(s.negz, s.negz), a2 = pack2(aa, aa), l2 = pack2(aa * aa * lam_e, aa * aa * lam_e);
      u64 vi[4 * NG], ui[4 * NG];
#pragma unroll
      for (int q = 0; q < 4 * NG; ++q) {
        const int i = slot + 4 * CW * (q >> 2) + (q & 3);
        const float v = x[i] * sc * inv, u = csm[s.uvec + i];
        vi[q] = pack2(v, v); ui[q] = pack2(u, u);
      }
#pragma unroll
      for (int k = 0; k < IT; ++k) {
        const int c = lane + 32 * k;
        float4 vj = x4[c];
        const float4 uj = u4[c];
        vj.x = vj.x * sc * inv; vj.y = vj.y * sc * inv; vj.z = vj.z * sc * inv; vj.w = vj.w * sc * inv;
        const u64 va = pack2(vj.x, vj.y), vb = pack2(vj.z, vj.w), ua = pack2(uj.x, uj.y), ub = pack2(uj.z, uj.w);
#pragma unroll
        for (int q = 0; q < 4 * NG; ++q) {
          a[q][k].lo = rank2(a[q][k].lo, vi[q], ui[q], va, ua, a2, l2, z);
          a[q][k].hi = rank2(a[q][k].hi, vi[q], ui[q], vb, ub, a2, l2, z);
        }
      }
    }
    if (threadIdx.x == 0) s.ah[step] = aa;
    if (threadIdx.x == 0 && s.sub == 0) {
      if (!ok) L->iscal[IS_STATUS_NOSUB] = 1;
      if (!isfinite(n2) || !isfinite(lam_e)) L->iscal[IS_STATUS_NONFINITE] = 1;
      if (tr) {
        tr[4 * step] = lam_e; tr[4 * step + 1] = g_e; tr[4 * step + 2] = (float)cnt; tr[4 * step + 3] = (float)mp;
      }
      if (last && step + 1 == K) {
        L->scal[SC_LAMBDA_E] = lam_e; L->scal[SC_G_E] = g_e; L->scal[SC_A_E] = aa;
        L->iscal[IS_MPRIME] = mp; L->iscal[IS_SETSIZE] = cnt;
      }
    }
  }
  rows_sync(l);                                // v_e and a_e of the steps
  const bool smooth = last && L->Qs != L->Q;
  if ((s.M & 3) == 0) {
    if (!*(volatile int*)&s.fail) store_rows<NG, IT, true>(a, L->Phiy, s);
    apply_steps<NG, IT, true>(s, l, L, K, smooth);
  } else {
    if (!*(volatile int*)&s.fail) store_rows<NG, IT, false>(a, L->Phiy, s);
    apply_steps<NG, IT, false>(s, l, L, K, smooth);
  }
}

// ---- layers of at most 64 features: one CTA, a row on 8 lanes ----
// No exchange leaves the CTA, so a pass is its own latency: a row on 8 lanes takes three shuffle rounds instead of five,
// every lane has work, and one block barrier ends it (M = 64: 0.26 us a power iteration, 0.46 with four rows per warp;
// at 128 features, 4 lanes per row were no faster than that).
constexpr int LPR = 8;                           // lanes per row: 64 rows on 512 threads
__device__ __forceinline__ float row_sum(float x) {
#pragma unroll
  for (int o = LPR / 2; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  return x;
}
__device__ __noinline__ void run_solo(Slab& s, const LayerDev* L, float* tr, int K, int P, bool last) {
  constexpr int KM = 64 / (4 * LPR);             // float4 per lane
  const int tid = threadIdx.x, row = tid / LPR, sub = tid % LPR;
  const int M = s.M;
  auto load = [&](float4 (&r)[KM], const float* G) {
#pragma unroll
    for (int k = 0; k < KM; ++k) {
      const int c = 4 * (sub + LPR * k);
      float x[4] = {0.f, 0.f, 0.f, 0.f};
      if (row < M && c < M) {
        const float* p = G + (size_t)row * M + c;
        if ((M & 3) == 0) *reinterpret_cast<float4*>(x) = *reinterpret_cast<const float4*>(p);
        else
#pragma unroll
          for (int e = 0; e < 4; ++e) if (c + e < M) x[e] = p[e];
      }
      r[k] = make_float4(x[0], x[1], x[2], x[3]);
    }
  };
  auto save = [&](const float4 (&r)[KM], float* G) {
#pragma unroll
    for (int k = 0; k < KM; ++k) {
      const int c = 4 * (sub + LPR * k);
      if (row < M && c < M) {
        float* p = G + (size_t)row * M + c;
        if ((M & 3) == 0) *reinterpret_cast<float4*>(p) = r[k];
        else {
          p[0] = r[k].x;
          if (c + 1 < M) p[1] = r[k].y;
          if (c + 2 < M) p[2] = r[k].z;
          if (c + 3 < M) p[3] = r[k].w;
        }
      }
    }
  };
  float4 a[KM];
  load(a, L->Phiy);
  // Sums are formed as the warp of a larger layer forms them (a pair of sums per float4, then a tree over the float4s), so
  // that a layer's result does not depend on what else is in the launch.
  auto four = [](float4 x, float4 y) {
    return fmaf(x.z, y.z, __fmul_rn(x.x, y.x)) + fmaf(x.w, y.w, __fmul_rn(x.y, y.y));
  };
  // y = row . x into dst, as pass() does it: SCALE times scale; NORM: row . (scale x), returns ||scale x||^2 of the next scale;
  // UNIT: row . (scale x / ||scale x||)
  auto dot = [&](const float* x, float scale, int mode, float* dst) {
    const float4* x4 = reinterpret_cast<const float4*>(x);
    float d = 0.f, n2 = 0.f, inv = 1.f;
    float4 b[KM];
#pragma unroll
    for (int k = 0; k < KM; ++k) {
      b[k] = x4[sub + LPR * k];
      if (mode == PASS_SCALE) continue;
      b[k].x *= scale; b[k].y *= scale; b[k].z *= scale; b[k].w *= scale;
      n2 = k ? n2 + four(b[k], b[k]) : four(b[k], b[k]);
    }
    if (mode == PASS_UNIT) { n2 = row_sum(n2); inv = inv_norm(n2); }
#pragma unroll
    for (int k = 0; k < KM; ++k) {
      if (mode == PASS_UNIT) { b[k].x *= inv; b[k].y *= inv; b[k].z *= inv; b[k].w *= inv; }
      d = k ? d + four(a[k], b[k]) : four(a[k], b[k]);
    }
    d = row_sum(d);
    if (sub == 0) dst[row] = mode == PASS_SCALE ? d * scale : d;
    if (mode == PASS_NORM) n2 = row_sum(n2);
    return n2;
  };
  for (int step = 0; step < K; ++step) {
    // squared norms (Eq. 45), m' (Eq. 46): every warp finds it for itself
    float q0 = four(a[0], a[0]);
#pragma unroll
    for (int k = 1; k < KM; ++k) q0 += four(a[k], a[k]);
    q0 = row_sum(q0);
    if (sub == 0) csm[s.xi2 + row] = q0;
    __syncthreads();
    const int mp = argmax_xi(s);
    if (row == mp) {
#pragma unroll
      for (int k = 0; k < KM; ++k) reinterpret_cast<float4*>(csm + s.wvec)[sub + LPR * k] = a[k];
    }
    __syncthreads();
    dot(csm + s.wvec, 1.f, PASS_SCALE, csm + s.cvec);                       // Eq. 47
    __syncthreads();
    // coherent set, aligned average (Eqs. 48-49)
    int cnt = 1;
    {
      float wv = 0.f;
      bool in = false;
      if (s.maxcol) {
        wv = tid == mp ? 1.f : 0.f;
      } else if (tid < M) {
        const float c = csm[s.cvec + tid];
        const float thr = fmaxf(s.c_rel * sqrtf(csm[s.xi2 + mp]) * sqrtf(csm[s.xi2 + tid]), s.c_abs);
        in = fabsf(c) >= thr;       // false for NaN
        wv = in ? (1.f / c) : 0.f;
      }
      if (tid < 64) csm[s.wvec + tid] = wv;
      const int n = __syncthreads_count(in);
      if (!s.maxcol) cnt = n;
    }
    int xo = s.buf0, yo = xo + s.Mv;
    dot(csm + s.wvec, cnt > 0 ? 1.f / (float)cnt : 0.f, PASS_SCALE, csm + xo);
    __syncthreads();
    float sc = 1.f;                                                         // x is sc times the vector at xo
    for (int p = 0; p < P; ++p) {
      const float n2 = dot(csm + xo, sc, PASS_NORM, csm + yo);
      __syncthreads();
      sc = inv_norm(n2);
      const int t = xo; xo = yo; yo = t;
    }
    const float n2 = dot(csm + xo, sc, PASS_UNIT, csm + s.uvec);           // u = Phi_y v, v = x / ||x|| (Eq. 50)
    const float inv = inv_norm(n2);
    __syncthreads();
    const float4* x4 = reinterpret_cast<const float4*>(csm + xo);
    const float4* u4 = reinterpret_cast<const float4*>(csm + s.uvec);
    float l0 = 0.f;
#pragma unroll
    for (int k = 0; k < KM; ++k) {
      float4 x = x4[sub + LPR * k];
      x.x = x.x * sc * inv; x.y = x.y * sc * inv; x.z = x.z * sc * inv; x.w = x.w * sc * inv;
      l0 = k ? l0 + four(x, u4[sub + LPR * k]) : four(x, u4[sub + LPR * k]);
    }
    const float lam_e = row_sum(l0);                              // Eq. 36
    const bool ok = cnt > 0 && n2 > 0.f && isfinite(n2) && isfinite(lam_e);
    float g_e = 1.f, aa = 0.f;
    if (ok) {
      g_e = s.delta * s.lam_bar / fmaxf(lam_e, s.eps);                 // Eqs. 40-41
      aa = sqrtf(g_e) - 1.f;
    }
    // Phi_y += a (v u^T + u v^T) + a^2 lambda_e v v^T, as in run_steps
    if (aa != 0.f) {
      const float v = csm[xo + row] * sc * inv, u = csm[s.uvec + row], l = aa * aa * lam_e;
#pragma unroll
      for (int k = 0; k < KM; ++k) {
        float4 vj = x4[sub + LPR * k];
        const float4 uj = u4[sub + LPR * k];
        vj.x = vj.x * sc * inv; vj.y = vj.y * sc * inv; vj.z = vj.z * sc * inv; vj.w = vj.w * sc * inv;
        a[k] = rank2(a[k], pack2(v, v), pack2(u, u), pack2(vj.x, vj.y), pack2(vj.z, vj.w), pack2(uj.x, uj.y), pack2(uj.z, uj.w),
                     pack2(aa, aa), pack2(l, l), pack2(s.negz, s.negz));
      }
    }
    if (tid < 64) csm[s.vh + step * s.Mv + tid] = csm[xo + tid] * sc * inv;
    if (tid == 0) {
      s.ah[step] = aa;
      if (!ok) L->iscal[IS_STATUS_NOSUB] = 1;
      if (!isfinite(n2) || !isfinite(lam_e)) L->iscal[IS_STATUS_NONFINITE] = 1;
      if (tr) {
        tr[4 * step] = lam_e; tr[4 * step + 1] = g_e; tr[4 * step + 2] = (float)cnt; tr[4 * step + 3] = (float)mp;
      }
      if (last && step + 1 == K) {
        L->scal[SC_LAMBDA_E] = lam_e; L->scal[SC_G_E] = g_e; L->scal[SC_A_E] = aa;
        L->iscal[IS_MPRIME] = mp; L->iscal[IS_SETSIZE] = cnt;
      }
    }
    __syncthreads();
  }
  // ---- the recorded steps in T, then Q (Eqs. 42, 44), as in apply_steps ----
  float4 t[KM], o[KM];
  load(t, L->Tt);
#pragma unroll 1
  for (int j = 0; j < K; ++j) {
    const float ak = s.ah[j];
    if (ak == 0.f) continue;
    const float4* v4 = reinterpret_cast<const float4*>(csm + s.vh + j * s.Mv);
    float d = four(t[0], v4[sub]);
#pragma unroll
    for (int k = 1; k < KM; ++k) d += four(t[k], v4[sub + LPR * k]);
    d = row_sum(d);
    const float at = ak * d;
    if (sub == 0) csm[s.th + j * s.Mv + row] = d;
#pragma unroll
    for (int k = 0; k < KM; ++k) {
      const float4 b = v4[sub + LPR * k];
      t[k].x = fmaf(at, b.x, t[k].x); t[k].y = fmaf(at, b.y, t[k].y); t[k].z = fmaf(at, b.z, t[k].z); t[k].w = fmaf(at, b.w, t[k].w);
    }
  }
  save(t, L->Tt);
  if (L->round_t) {                    // rows of whole float4s
#pragma unroll
    for (int k = 0; k < KM; ++k)
      o[k] = make_float4(sm100::tf32_rna(t[k].x), sm100::tf32_rna(t[k].y), sm100::tf32_rna(t[k].z), sm100::tf32_rna(t[k].w));
    save(o, L->tmp);
  }
  load(t, L->Q);
  __syncthreads();
#pragma unroll 1
  for (int j = 0; j < K; ++j) {
    const float ak = s.ah[j];
    if (ak == 0.f) continue;
    const float aq = ak * (ak + 2.f), ti = csm[s.th + j * s.Mv + row];
    const float4* t4 = reinterpret_cast<const float4*>(csm + s.th + j * s.Mv);
#pragma unroll
    for (int k = 0; k < KM; ++k) {
      const float4 b = t4[sub + LPR * k];
      t[k].x = __fadd_rn(t[k].x, __fmul_rn(aq, __fmul_rn(ti, b.x))); t[k].y = __fadd_rn(t[k].y, __fmul_rn(aq, __fmul_rn(ti, b.y)));
      t[k].z = __fadd_rn(t[k].z, __fmul_rn(aq, __fmul_rn(ti, b.z))); t[k].w = __fadd_rn(t[k].w, __fmul_rn(aq, __fmul_rn(ti, b.w)));
    }
  }
  save(t, L->Q);
  if (last && L->Qs != L->Q) {            // Eq. 35
    const float beta = L->beta, ob = 1.f - beta;
    load(o, L->Qs);
#pragma unroll
    for (int k = 0; k < KM; ++k) {
      o[k].x = fmaf(beta, o[k].x, ob * t[k].x); o[k].y = fmaf(beta, o[k].y, ob * t[k].y);
      o[k].z = fmaf(beta, o[k].z, ob * t[k].z); o[k].w = fmaf(beta, o[k].w, ob * t[k].w);
    }
    save(o, L->Qs);
  }
  __syncthreads();
  save(a, L->Phiy);
}

// groups of four rows this warp owns in a slab of R rows
__device__ __forceinline__ int warp_groups(int R) {
  const int warp = threadIdx.x >> 5, ng = R >> 2;
  return ng > warp ? (ng - warp + CW - 1) / CW : 0;
}

__host__ __device__ inline int slab_rows(int M, int n) { return (((M + n - 1) / n) + 3) & ~3; }
__host__ __device__ inline int slab_trips(int M) { return (((M + 3) >> 2) + 31) / 32; }
__host__ __device__ inline int slab_vec(int M, int n) {
  const int a = n * slab_rows(M, n), b = 128 * slab_trips(M);
  return a > b ? a : b;
}
constexpr int kVecs = 6 + 2 * KH;

// SOLO: all layers take one CTA and eight lanes a row; any number of steps.  (A kernel of its own: the loop round run_solo costs
// run_steps registers where both are called, M = 576, K = 8, P = 16 160 -> 162 us.)
template <bool SOLO>
__global__ void __launch_bounds__(CT, 1) recursion_cluster_kernel(const __grid_constant__ ClusterArgs a) {
  dep_sync();
  cg::cluster_group cluster = cg::this_cluster();
  const int rank = (int)cluster.block_rank();
  const int lane = threadIdx.x & 31;
  // my layer: the one whose CTA range holds this CTA (none: a filler CTA of a cluster)
  int layer = -1;
#pragma unroll 1
  for (int l = 0; l < a.g.n; ++l)
    if ((int)blockIdx.x >= a.first_cta[l] && (int)blockIdx.x < a.first_cta[l] + a.ncta[l]) layer = l;
  if (layer < 0) {
    cluster.sync();     // the two cluster-wide meetings of the kernel
    cluster.sync();
    return;
  }
  const LayerDev* L = a.g.layer[layer];
  __shared__ __align__(8) uint64_t xbar[3];
  __shared__ Slab s;
  Link l;
  l.n = a.ncta[layer];
  l.active = 0;
  l.bar0 = smem_u32(&xbar[0]);                       // the three barriers are 8 bytes apart
  if (threadIdx.x == 0) {
    const int M = L->M, n = l.n;
    s.M = M; s.Mp = (M + 3) & ~3; s.R = slab_rows(M, n); s.n = n;
    s.Mv = slab_vec(M, n);
    s.sub = (int)blockIdx.x - a.first_cta[layer];
    s.row0 = s.sub * s.R;
    s.xi2 = 0;
    s.cvec = s.xi2 + s.Mv; s.wvec = s.cvec + s.Mv; s.buf0 = s.wvec + s.Mv; s.uvec = s.buf0 + 2 * s.Mv;
    s.vh = s.uvec + s.Mv; s.th = s.vh + KH * s.Mv;
    s.tx = (uint32_t)n * (uint32_t)s.R * 4u;
    s.maxcol = L->init == FW_INIT_MAXCOL;
    s.c_rel = L->c_rel; s.c_abs = L->c_abs; s.delta = L->delta; s.eps = L->eps;
    s.lam_bar = L->scal[SC_LAMBDA_BAR];
    s.fail = 0; s.negz = -0.f;
    sm100::mbar_init(l.bar0, 1);
    sm100::mbar_init(l.bar0 + 8, 1);
    sm100::mbar_init(l.bar0 + 16, 1);
    sm100::mbar_fence_init();
  }
  __syncthreads();
  const int M = s.M, R = s.R;
  l.active = 32 * min(CW, R >> 2);

  // what no exchange fills of the vectors stays zero (rows past the matrix are zero rows)
  const int filled = l.n * R, tail = s.Mv - filled;
  for (int i = threadIdx.x; i < kVecs * tail; i += CT) csm[s.xi2 + i / tail * s.Mv + filled + i % tail] = 0.f;
  // A CTA's window of the cluster address space is this CTA's window shifted by a constant; the stores rely on it,
  // so it is checked on two addresses far apart before anything is sent.
  const uint32_t peer_rank = (uint32_t)(rank - s.sub + min(lane, l.n - 1));
  l.rdelta = map_cluster(l.bar0, peer_rank) - l.bar0;
  const bool linear = (map_cluster(smem_u32(csm + s.th), peer_rank) - smem_u32(csm + s.th)) == l.rdelta;
  const bool usable = __syncthreads_or(!linear) == 0;
  sm100::cluster_arrive();   // every barrier is initialised before the first remote store can arrive: waited for in run_steps

  const int ng = M <= kSolo ? 0 : warp_groups(R), it = slab_trips(M);
  if (!usable || ng == 0 || a.K < 1) sm100::cluster_wait();
  if (usable && a.K > 0) {
    float* tr = const_cast<float*>(reinterpret_cast<const float*>(a.traces.p[layer]));
    if (tr) tr += 4 * a.k0;
    const bool last = a.last != 0;
    if (SOLO) {
      for (int k = 0; k < a.K; k += KH) run_solo(s, L, tr ? tr + 4 * k : nullptr, min(KH, a.K - k), a.P, last && k + KH >= a.K);
    } else if (M <= kSolo) {
      run_solo(s, L, tr, a.K, a.P, last);
    } else if (ng == 1) {
      switch (it) {
        case 1: run_steps<1, 1>(s, l, L, tr, a.K, a.P, last); break;
        case 2: run_steps<1, 2>(s, l, L, tr, a.K, a.P, last); break;
        case 3: run_steps<1, 3>(s, l, L, tr, a.K, a.P, last); break;
        case 4: run_steps<1, 4>(s, l, L, tr, a.K, a.P, last); break;
        default: run_steps<1, 5>(s, l, L, tr, a.K, a.P, last); break;
      }
    } else if (ng == 2) {
      switch (it) {
        case 1: run_steps<2, 1>(s, l, L, tr, a.K, a.P, last); break;
        default: run_steps<2, 2>(s, l, L, tr, a.K, a.P, last); break;
      }
    }
  }
  __syncthreads();
  if (s.fail || !usable) {
    // a wait gave up: the state of this layer is not to be trusted; report and leave in step with the peers
    if (threadIdx.x == 0) L->iscal[IS_STATUS_TIMEOUT] = 1;
  } else {
    if (s.sub == 0 && !s.maxcol)
      for (int m = threadIdx.x; m < M; m += CT) L->wvec[m] = csm[s.wvec + m];    // alignment weights of the last step
  }
  cluster.sync();   // no CTA leaves while a peer may still read or write its shared memory
}

size_t cluster_smem(int M, int n) {
  return (size_t)kVecs * slab_vec(M, n) * sizeof(float);
}

bool cluster_fits(int M, int n) {
  const int it = slab_trips(M);
  return M <= kMaxM && it <= kMaxIt && slab_rows(M, n) <= 4 * CW * max_groups(it) && cluster_smem(M, n) <= kSmemLimit;
}

// What a pass costs a layer on n CTAs, in units of the work of one group of four rows and one trip over the columns:
// the work of the busiest of the four SM partitions, and the fixed part of an exchange (less within one CTA).
int cluster_cost(int M, int n) {
  const int groups = slab_rows(M, n) / 4;
  if (M <= kSolo) return 4;         // one CTA, and no gain from more
  return ((groups + 3) / 4) * slab_trips(M) + (n > 1 ? 20 : 8);
}

// first-fit of the layers' CTA counts (largest first) into clusters of cl: the clusters needed; first[i] (optional)
// receives the first CTA of layer i.  A layer never straddles a cluster.
int cluster_pack(const int* cnt, int n, int cl, int32_t* first) {
  int order[FW_MAX_GROUP], used[FW_MAX_GROUP];
  for (int i = 0; i < n; ++i) { order[i] = i; used[i] = 0; }
  for (int i = 1; i < n; ++i)                       // insertion sort, stable
    for (int j = i; j > 0 && cnt[order[j]] > cnt[order[j - 1]]; --j) {
      const int t = order[j]; order[j] = order[j - 1]; order[j - 1] = t;
    }
  int bins = 0;
  for (int oi = 0; oi < n; ++oi) {
    const int i = order[oi];
    int b = 0;
    while (b < bins && used[b] + cnt[i] > cl) ++b;
    if (b == bins) ++bins;
    if (first) first[i] = b * cl + used[b];
    used[b] += cnt[i];
  }
  return bins;
}

// CTA counts of the layers in clusters of cl, of which `resident` run together.  Every layer starts on the fewest CTAs
// that hold it; then, while the clusters of one wave allow, the layer whose passes cost most is spread over more CTAs
// (the launch ends with its slowest layer).  Returns the cost of the launch: waves x slowest layer; 0: does not fit.
int cluster_plan(const int* layer_M, int n, int cl, int resident, int* cnt) {
  for (int i = 0; i < n; ++i) {
    cnt[i] = recursion_cluster_ctas(layer_M[i]);
    if (cnt[i] == 0 || cnt[i] > cl) return 0;
  }
  for (int round = 0; round < 16 * FW_MAX_GROUP; ++round) {
    int worst_cost = 0;
    for (int i = 0; i < n; ++i) worst_cost = std::max(worst_cost, cluster_cost(layer_M[i], cnt[i]));
    // all layers at the worst cost have to improve for the launch to gain: try them together
    int trial[FW_MAX_GROUP];
    bool improved = true;
    for (int i = 0; i < n && improved; ++i) {
      trial[i] = cnt[i];
      if (cluster_cost(layer_M[i], cnt[i]) != worst_cost) continue;
      int n2 = cnt[i] + 1;
      while (n2 <= cl && !(cluster_fits(layer_M[i], n2) && cluster_cost(layer_M[i], n2) < worst_cost)) ++n2;
      improved = n2 <= cl;                           // else this layer cannot get cheaper: the maximum stays
      trial[i] = n2;
    }
    if (!improved || cluster_pack(trial, n, cl, nullptr) > resident) break;
    for (int i = 0; i < n; ++i) cnt[i] = trial[i];
  }
  int worst = 0;
  for (int i = 0; i < n; ++i) worst = std::max(worst, cluster_cost(layer_M[i], cnt[i]));
  const int bins = cluster_pack(cnt, n, cl, nullptr);
  return worst * ((bins + resident - 1) / resident);
}

// The plan of the last set of layers a thread launched (a training loop repeats one set).
struct ClusterPlan {
  int dev = -1, n = 0, cl = 0, bins = 0;
  int dims[FW_MAX_GROUP], cnt[FW_MAX_GROUP];
  int32_t first[FW_MAX_GROUP];
};

}  // namespace

// CTAs a layer of size M needs at least: the smallest count whose slab of Phi_y fits a CTA; 0: not on chip
int recursion_cluster_ctas(int M) {
  for (int n = 1; n <= CLMAX; ++n)
    if (cluster_fits(M, n)) return n;
  return 0;
}

bool recursion_cluster_supported(int M) { return recursion_cluster_ctas(M) > 0; }

cudaError_t launch_recursion_cluster(const GroupDev& g, const PtrTable& traces, const int* layer_M, int K, int P,
                                     cudaStream_t s) {
  static SmemAttrCache attr, solo_attr;
  static std::mutex mu;
  static int resident[64][5];        // clusters of 1, 2, 4, 8, 16 CTAs that run together (16: 7 on a B200)
  thread_local ClusterPlan plan;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) { cudaGetLastError(); dev = 0; }
  auto config = [&](cudaLaunchConfig_t& cfg, cudaLaunchAttribute* at, int cl, int ctas, size_t smem) {
    memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3(ctas); cfg.blockDim = dim3(CT); cfg.dynamicSmemBytes = smem; cfg.stream = s;
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = cl; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;      // as launch_dep
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at; cfg.numAttrs = 2;
  };
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute at[2];
  {
    std::lock_guard<std::mutex> lock(mu);
    if (resident[dev][0] == 0) {
      // clusters of 16 CTAs are beyond the portable size of 8
      cudaError_t e = cudaFuncSetAttribute(recursion_cluster_kernel<false>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
      if (e == cudaSuccess) e = cudaFuncSetAttribute(recursion_cluster_kernel<true>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
      if (e == cudaSuccess) e = ensure_dyn_smem(recursion_cluster_kernel<false>, kSmemLimit, attr);
      if (e == cudaSuccess) e = ensure_dyn_smem(recursion_cluster_kernel<true>, kSmemLimit, solo_attr);
      if (e != cudaSuccess) return e;
      for (int b = 4; b >= 0; --b) {
        int nc = 0;
        config(cfg, at, 1 << b, CLMAX * 64, kSmemLimit);
        if (cudaOccupancyMaxActiveClusters(&nc, recursion_cluster_kernel<false>, &cfg) != cudaSuccess || nc < 1) {
          cudaGetLastError();
          nc = 1;
        }
        resident[dev][b] = nc;
      }
    }
  }
  if (plan.dev != dev || plan.n != g.n || memcmp(plan.dims, layer_M, g.n * sizeof(int)) != 0) {
    // the cluster size whose plan costs least; the larger one where two tie (layers can spread further)
    int best = 0;
    plan.dev = -1;
    for (int b = 4; b >= 0; --b) {
      int cnt[FW_MAX_GROUP];
      const int c = cluster_plan(layer_M, g.n, 1 << b, resident[dev][b], cnt);
      if (c == 0 || (best != 0 && c >= best)) continue;
      best = c;
      plan.cl = 1 << b;
      memcpy(plan.cnt, cnt, g.n * sizeof(int));
    }
    if (best == 0) return cudaErrorInvalidValue;
    plan.bins = cluster_pack(plan.cnt, g.n, plan.cl, plan.first);
    memcpy(plan.dims, layer_M, g.n * sizeof(int));
    plan.n = g.n; plan.dev = dev;
  }
  ClusterArgs a;
  memset(&a, 0, sizeof(a));
  a.g = g; a.traces = traces; a.P = P;
  size_t smem = 0;
  bool solo = true;
  for (int i = 0; i < g.n; ++i) {
    a.first_cta[i] = plan.first[i]; a.ncta[i] = plan.cnt[i];
    smem = std::max(smem, cluster_smem(layer_M[i], plan.cnt[i]));
    solo &= layer_M[i] <= kSolo;
  }
  config(cfg, at, plan.cl, plan.bins * plan.cl, smem);
  // A launch is KH steps.  Layers of one CTA each take all of the call's in one: a launch of theirs costs as much as two steps
  // without power iterations (M = 64, K = 32, P = 0: 93 us in four launches, 77 in one).  Where a cluster exchanges, the steps
  // are long and a loop round run_steps costs each of them more than it saves launches (M = 576, K = 8, P = 16: 160 us, with the
  // loop 172; K = 64, P = 4: 559 and 560).
  const int most = solo ? K : KH;
  for (int k0 = 0; k0 < K; k0 += most) {
    a.k0 = k0; a.K = std::min(most, K - k0); a.last = k0 + a.K == K;
    ProfScope ps(FW_PROF_RECUR_CHIP, s);
    const cudaError_t e = solo ? cudaLaunchKernelEx(&cfg, recursion_cluster_kernel<true>, a)
                               : cudaLaunchKernelEx(&cfg, recursion_cluster_kernel<false>, a);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace fw
