// Block sweeps: L L^T x = b with a batch of banded Cholesky factors (the
// local solves A_j^{-1} of the preconditioner, Section 3, and the eigensolver's
// K_j^{-1} block solves, Section 4.4), each matrix solved by a cluster of
// C = 1, 2, 4 or 8 thread blocks.
//
// A sweep is a chain: block k of B rows needs every earlier block.  What
// bounds it is the latency of one link (product with the newest block, the
// diagonal block, a block barrier or two), not bandwidth, until the links are
// few and cheap.  So the links are long (B = 64 rows where the staging fits,
// not 16), the diagonal blocks are inverted once after the factorisation, in
// place in the band (k_band_blkinv; no extra traffic, the strip under the
// diagonal of a block is not needed otherwise), and everything that does not
// depend on the newest block is kept off the chain.
//
// Row block k belongs to block k mod C of the cluster.
//  forward: the owner has summed L(k, j) y_j over all older j while the chain
//    ran elsewhere; when y_{k-1} arrives it adds that product, applies the
//    inverted diagonal block and stores y_k into the ring of solved rows of
//    every block of the cluster.  A value is its own flag: the receiver clears
//    the slot to a NaN pattern no computation gives and polls for anything else
//    (an mbarrier per message cost a link about 170 cycles more).
//  backward: the owner of k gathers the other blocks' partial sums
//    sum_r L(r, k)^T x_r from its mailbox, applies the transposed inverse,
//    then computes its contribution to block k - 1 first and sends it on;
//    contributions to older blocks accumulate in its own ring.
// Every block streams only its own rows (1/C of the factor), by bulk copies
// into a ring of row slots.  One right-hand side: one product per (row,
// column phase) thread; several, FP32 factors: m16n8k8 TF32 MMAs in one or
// three passes; several, FP64 factors: FP64 or double-single
// multiply-adds, a register tile of NC columns per thread.
//
// Measured against one thread block per matrix in 16-row steps of forward
// substitution: one column of 64 FP32 bands of order 5832, half width 340,
// 785 -> 267 us; a solve with the 8 bands of a 32^3 grid 24.4 -> 7.1 ms; an FP64
// apply at 64^3 2.9 -> 1.4 ms; the eigensolver's sweeps at 48^3 in FP64 (11
// columns, 27 bands) 653 -> 138 ms, where the FP64 pipe bounds them.  With more
// matrices than SMs HBM bounds the one-column sweep (512 bands of a 128^3 grid,
// 1.74 ms for 9.23 GB: 5.3 TB/s).
//
// All sums run in a fixed order.  Every wait is bounded; a wait that gives up
// records GENEO_ERR_TIMEOUT and the block goes on without waiting.  A slot's clears
// and fills are ordered by release and acquire fences (release_cluster).
#include <algorithm>
#include <atomic>
#include <type_traits>

#include "common.cuh"
#include "ds.cuh"
#include "ptx.cuh"
#include "sweep_index.h"

namespace geneo {
namespace {

constexpr int kThreads = 256;  // compute threads; one more warp copies the factor rows
constexpr int kMaxSlots = 8;   // row slots of the factor stream
constexpr int kMaxC = 8;

// ---------------------------------------------------------------------------
// Cluster helpers.
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t map_rank(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// Values pass between the blocks of a cluster as plain 4- or 8-byte stores into
// shared memory that holds kUnset until then: the value is its own flag, so a
// reader polls the word itself (one shared load) and neither side touches an
// mbarrier (about 170 cycles to test here, with every warp testing).  The
// pattern is a signalling NaN, which no arithmetic returns.  Other threads of the
// reader's block read the word after a block barrier.
constexpr uint32_t kUnset32 = 0x7fbadbadu;
constexpr uint64_t kUnset64 = 0x7ff4badbad7fbadbull;
__device__ __forceinline__ void st_cluster(uint32_t dst, float v) {
  asm volatile("st.relaxed.cluster.shared::cluster.b32 [%0], %1;" ::"r"(dst), "r"(__float_as_uint(v)) : "memory");
}
__device__ __forceinline__ void st_cluster(uint32_t dst, double v) {
  asm volatile("st.relaxed.cluster.shared::cluster.b64 [%0], %1;" ::"r"(dst), "l"(__double_as_longlong(v))
               : "memory");
}
__device__ __forceinline__ void st_cluster(uint32_t dst, dsv v) {
  const uint64_t b = ((uint64_t)__float_as_uint(v.l) << 32) | __float_as_uint(v.h);
  asm volatile("st.relaxed.cluster.shared::cluster.b64 [%0], %1;" ::"r"(dst), "l"(b) : "memory");
}
__device__ __forceinline__ void unset(float* p) { *reinterpret_cast<uint32_t*>(p) = kUnset32; }
__device__ __forceinline__ void unset(double* p) { *reinterpret_cast<uint64_t*>(p) = kUnset64; }
__device__ __forceinline__ void unset(dsv* p) { *reinterpret_cast<uint64_t*>(p) = kUnset64; }
// A slot is cleared by its owner and filled again by another block: what orders
// the two is a message from the owner (release, after a block barrier that follows
// the clears) that the other block has polled (acquire, after the polls and before
// the block barrier that precedes its stores).  Both fences cover shared memory
// only.  With and without them: eight columns, 64 bands of order 6859, half width
// 381, 491 and 486 us a sweep; 12 columns 574 and 560; one column, 64 bands of 5832,
// 340, 231 and 230.
__device__ __forceinline__ void release_cluster() {
  asm volatile("fence.release.sync_restrict::shared::cta.cluster;" ::: "memory");
}
__device__ __forceinline__ void acquire_cluster() {
  asm volatile("fence.acquire.sync_restrict::shared::cluster.cluster;" ::: "memory");
}
__device__ __forceinline__ float ld_cluster(const float* p) {
  uint32_t v;
  asm volatile("ld.relaxed.cluster.shared::cta.b32 %0, [%1];" : "=r"(v) : "r"(smem_u32(p)) : "memory");
  return __uint_as_float(v);
}
__device__ __forceinline__ uint64_t ld_cluster64(const void* p) {
  uint64_t v;
  asm volatile("ld.relaxed.cluster.shared::cta.b64 %0, [%1];" : "=l"(v) : "r"(smem_u32(p)) : "memory");
  return v;
}
__device__ __forceinline__ double ld_cluster(const double* p) {
  return __longlong_as_double((long long)ld_cluster64(p));
}
__device__ __forceinline__ dsv ld_cluster(const dsv* p) {
  const uint64_t v = ld_cluster64(p);
  return dsv(__uint_as_float((uint32_t)v), __uint_as_float((uint32_t)(v >> 32)));
}
__device__ __forceinline__ bool is_unset(float v) { return __float_as_uint(v) == kUnset32; }
__device__ __forceinline__ bool is_unset(double v) { return (uint64_t)__double_as_longlong(v) == kUnset64; }
__device__ __forceinline__ bool is_unset(dsv v) {
  return __float_as_uint(v.h) == (uint32_t)kUnset64 && __float_as_uint(v.l) == (uint32_t)(kUnset64 >> 32);
}
// bounded wait (a second or so) until the N values at(0 .. N - 1), those with
// in(i), are set; all of them are read at once
template <int N, typename A, typename At, typename In>
__device__ __forceinline__ bool wait_set(A* v, At at, In in, DevStatus* st, int id, int64_t where) {
  for (int it = 0; it < (1 << 24); ++it) {
    bool all = true;
#pragma unroll
    for (int i = 0; i < N; ++i) {
      if (in(i)) {
        v[i] = ld_cluster(at(i));
        all &= !is_unset(v[i]);
      }
    }
    if (all) return true;
  }
  record_error(st, GENEO_ERR_TIMEOUT, id, where);
  return false;
}

__device__ __forceinline__ void mma_tf32(float* c, const uint32_t* a, const uint32_t* b) {
  asm volatile(
      "mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}
__device__ __forceinline__ void split_tf32(float x, uint32_t& hi, uint32_t& lo) {
  float h, l;
  split_tf32_rn(x, h, l);
  hi = __float_as_uint(h);
  lo = __float_as_uint(l);
}

__device__ __forceinline__ float shfl_xor(float v, int o) { return __shfl_xor_sync(0xffffffffu, v, o); }
__device__ __forceinline__ double shfl_xor(double v, int o) { return __shfl_xor_sync(0xffffffffu, v, o); }
__device__ __forceinline__ dsv shfl_xor(dsv v, int o) {
  return dsv(__shfl_xor_sync(0xffffffffu, v.h, o), __shfl_xor_sync(0xffffffffu, v.l, o));
}

// The factor rows of the blocks rank, rank + C, ... in visiting order
// (ascending, then descending), streamed into a ring of slots of SR rows, HB
// slots per block, by a warp of their own: a slot is filled again as soon as
// the compute warps have released it.
template <typename T, int B>
struct RowStream {
  static constexpr int SR = B < 128 / (int)sizeof(T) ? B : 128 / (int)sizeof(T);
  static constexpr int HB = B / SR;   // slots per block
  uint64_t *full, *empty;
  T* slots;
  int ld, nslot;
  int cur = 0;                        // slot of the current block's first part
  uint32_t par = 0;                   // its phase
  __device__ __forceinline__ T* slot(int part) const {
    const int s = cur + part;
    return slots + (size_t)(s >= nslot ? s - nslot : s) * SR * ld;
  }
  __device__ __forceinline__ uint32_t slot_at(int part) const { return smem_u32(slot(part)); }
  __device__ __forceinline__ bool wait_part(int part, DevStatus* st, int id, int64_t where) const {
    const int s = cur + part;
    return mbar_wait_bounded(&full[s >= nslot ? s - nslot : s], s >= nslot ? par ^ 1 : par, st, id, where);
  }
  __device__ __forceinline__ bool wait(DevStatus* st, int id, int64_t where) const {
    bool ok = true;
#pragma unroll
    for (int h = 0; h < HB; ++h)
      if (ok) ok = wait_part(h, st, id, where);
    return ok;
  }
  // this warp has read the current block's rows for the last time
  __device__ __forceinline__ void release() {
    __syncwarp();
    if ((threadIdx.x & 31) == 0) {
#pragma unroll
      for (int h = 0; h < HB; ++h) {
        const int s = cur + h;
        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&empty[s >= nslot ? s - nslot : s]))
                     : "memory");
      }
    }
    cur += HB;
    if (cur >= nslot) {
      cur -= nslot;
      par ^= 1;
    }
  }
  // one lane of the copy warp
  __device__ __forceinline__ void produce(const T* L, int n, int rank, int C, int own, DevStatus* st, int id) {
    int s = 0, q = 0;
    uint32_t pe = 1;                  // phase parity of the slot's last release
    bool ok = true;
    for (int v = 0; v < 2 * own && ok; ++v) {
      const int kk = rank + C * (v < own ? v : 2 * own - 1 - v);
      for (int h = 0; h < HB; ++h, ++q) {
        if (q >= nslot) {
          ok = mbar_wait_bounded(&empty[s], pe, st, id, q);
          if (!ok) break;
        }
        const int r0 = kk * B + h * SR, rows = max(0, min(SR, n - r0));
        const uint32_t bytes = (uint32_t)((size_t)rows * ld * sizeof(T));
        fence_proxy_async();
        mbar_arrive_expect_tx(&full[s], bytes);
        if (bytes) bulk_load(slots + (size_t)s * SR * ld, L + (int64_t)r0 * ld, bytes, &full[s]);
        if (++s == nslot) {
          s = 0;
          pe ^= 1;
        }
      }
    }
    // every copy lands before the block ends (bounded): the last phase of
    // each slot used
    for (int i = 0; i < min(q, nslot); ++i) {
      const int uses = (q - i + nslot - 1) / nslot;
      mbar_wait_bounded(&full[i], (uint32_t)((uses - 1) & 1), st, id, -1);
    }
  }
};

// Shared memory ahead of the slots.
struct Bars {
  uint64_t full[kMaxSlots], empty[kMaxSlots];
  uint64_t pad[48];
};
static_assert(sizeof(Bars) == kSlotLead && kSlotLead % 128 == 0, "slot alignment");

// barrier of the compute warps
template <int N = kThreads>
__device__ __forceinline__ void csync() {
  asm volatile("bar.sync 1, %0;" ::"n"(N) : "memory");
}
// compute warps of the multiply-add sweep: four for small blocks (a row's sum
// over its lanes costs more than more warps gain; the lanes of a row must cover
// the NC columns), else eight
template <int NC, int B>
__host__ __device__ constexpr int sweep_warps() {
  return B <= 16 && NC <= 4 ? 4 : 8;
}

// N consecutive values from shared memory, by 16-byte loads where N fills them
// (p is then 16-byte aligned)
template <int N, typename A>
__device__ __forceinline__ void load_n(const A* p, A* o) {
  constexpr int V = 16 / sizeof(A);
  if constexpr (N % V == 0) {
#pragma unroll
    for (int i = 0; i < N / V; ++i) {
      const float4 q = reinterpret_cast<const float4*>(p)[i];
      if constexpr (std::is_same_v<A, float>) {
        o[4 * i] = q.x; o[4 * i + 1] = q.y; o[4 * i + 2] = q.z; o[4 * i + 3] = q.w;
      } else if constexpr (std::is_same_v<A, dsv>) {
        o[2 * i] = dsv(q.x, q.y);
        o[2 * i + 1] = dsv(q.z, q.w);
      } else {
        o[2 * i] = __hiloint2double(__float_as_int(q.y), __float_as_int(q.x));
        o[2 * i + 1] = __hiloint2double(__float_as_int(q.w), __float_as_int(q.z));
      }
    }
  } else {
#pragma unroll
    for (int i = 0; i < N; ++i) o[i] = p[i];
  }
}
// a factor value in arithmetic type A
template <typename A, typename T>
__device__ __forceinline__ A factor_value(T x) {
  if constexpr (std::is_same_v<A, dsv> && sizeof(T) == 4) return dsv(x, 0.f);
  else return to_arith<A>(x);
}
// acc[c] += sum L(e) X(e, c) over I entries of each of R groups of 32 (entry i
// of group q at index 32 q + i): L(e) = at(e), rows X(e, .) of NC values one
// after another at x, entries skipped where !in(e)
// (of the NC columns the first KC are formed)
template <int I, int R, int NC, int KC, typename T, typename A, typename At, typename In>
__device__ __forceinline__ void madd(A* acc, const A* x, At at, In in) {
  if constexpr (NC == 1) {
    constexpr int N = I * R, W = N >= 8 && sizeof(T) == 4 ? 4 : N >= 4 ? 2 : 1;   // chains
    A xv[N];
    T lv[N];
#pragma unroll
    for (int q = 0; q < R; ++q) load_n<I>(x + 32 * q, xv + I * q);
#pragma unroll
    for (int e = 0; e < N; ++e) {
      const bool p = in(32 * (e / I) + e % I);
      lv[e] = p ? at(32 * (e / I) + e % I) : T(0);
      xv[e] = p ? xv[e] : A();   // an entry outside may not have been set
    }
    A a[W];
    a[0] = acc[0];
#pragma unroll
    for (int u = 1; u < W; ++u) a[u] = A();
#pragma unroll
    for (int e = 0; e < N; ++e) a[e % W] += factor_value<A>(lv[e]) * xv[e];
    if constexpr (W == 4) acc[0] = (a[0] + a[1]) + (a[2] + a[3]);
    else if constexpr (W == 2) acc[0] = a[0] + a[1];
    else acc[0] = a[0];
  } else {
#pragma unroll
    for (int e = 0; e < I * R; ++e) {
      const int i = 32 * (e / I) + e % I;
      if (in(i)) {
        const A a = factor_value<A>(at(i));
        A xv[NC];
        load_n<NC>(x + i * NC, xv);
#pragma unroll
        for (int c = 0; c < KC; ++c) acc[c] += a * xv[c];
      }
    }
  }
}

// The one-column form on 32-bit shared addresses, every entry taken (the links
// of the chain are bound by instruction issue: 64-bit address arithmetic and
// predicates per entry doubled them): L(e) at address la(e), X at xa
__device__ __forceinline__ void lds(uint32_t a, float& v) {
  asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(a));
}
__device__ __forceinline__ void lds(uint32_t a, double& v) {
  asm volatile("ld.shared.f64 %0, [%1];" : "=d"(v) : "r"(a));
}
template <int N>
__device__ __forceinline__ void lds_n(uint32_t a, float* o) {
  if constexpr (N % 4 == 0) {
#pragma unroll
    for (int i = 0; i < N; i += 4)
      asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                   : "=f"(o[i]), "=f"(o[i + 1]), "=f"(o[i + 2]), "=f"(o[i + 3])
                   : "r"(a + 4 * i));
  } else {
#pragma unroll
    for (int i = 0; i < N; ++i) lds(a + 4 * i, o[i]);
  }
}
template <int N>
__device__ __forceinline__ void lds_n(uint32_t a, double* o) {
  if constexpr (N % 2 == 0) {
#pragma unroll
    for (int i = 0; i < N; i += 2)
      asm volatile("ld.shared.v2.f64 {%0, %1}, [%2];" : "=d"(o[i]), "=d"(o[i + 1]) : "r"(a + 8 * i));
  } else {
#pragma unroll
    for (int i = 0; i < N; ++i) lds(a + 8 * i, o[i]);
  }
}
template <int I, int R, int W, typename T, typename La, typename Op>
__device__ __forceinline__ void dot_lds(T (&a)[W], uint32_t xa, La la, Op op) {
  constexpr int N = I * R;
  T xv[N], lv[N];
#pragma unroll
  for (int e = 0; e < N; ++e) lds(la(e), lv[e]);
#pragma unroll
  for (int q = 0; q < R; ++q) lds_n<I>(xa + (uint32_t)(32 * sizeof(T)) * q, xv + I * q);
#pragma unroll
  for (int e = 0; e < N; ++e) a[e % W] += op(lv[e], e) * xv[e];
}
template <int W, typename T>
__device__ __forceinline__ T chains(const T (&a)[W]) {
  if constexpr (W == 4) return (a[0] + a[1]) + (a[2] + a[3]);
  else if constexpr (W == 2) return a[0] + a[1];
  else return a[0];
}

// ---------------------------------------------------------------------------
// Multiply-add sweep (T factor storage, A arithmetic, NC columns).  NW = four or
// eight warps of RPW = B / NW rows each (backward: columns); the PH = 32 / RPW lanes
// that share a row take RPW consecutive columns (rows) of every 32, so a
// warp's 32 band addresses fall in distinct banks (ld - 1 is odd), and the
// row's sum ends in two to five shuffles instead of a block barrier.
// ---------------------------------------------------------------------------
template <typename T, typename A, int NC, int B, int KC>
__global__ void __launch_bounds__(32 * sweep_warps<NC, B>() + 32, NC == 1 && sizeof(T) == 4 && B < 64 ? 2 : 1)
k_sweep(const T* __restrict__ base, const BandDesc* __restrict__ descs, double* __restrict__ xbase,
        const int64_t* __restrict__ xoff, int col0, int kcap, const int32_t* __restrict__ nrhs_dev,
        const int32_t* __restrict__ skip, int cpp, int C, int nslot, int rwb, DevStatus* st) {
  using RS = RowStream<T, B>;
  constexpr int SR = RS::SR, HB = RS::HB;
  constexpr int NW = sweep_warps<NC, B>(), kThreads = 32 * NW;
  constexpr int RPW = B / NW, PH = 32 / RPW;
  constexpr int R = B > 32 ? B / 32 : 1;        // groups of 32 per block
  // backward sums of a column: over the lanes that share it (one column, FP32:
  // shuffles are cheap), or by one thread per column (FP64 additions are not)
  constexpr bool kQuad = NC == 1 && sizeof(T) == 4;
  constexpr int W = RPW * R >= 8 ? 4 : RPW * R >= 4 ? 2 : 1;   // chains of a lane's sum (NC = 1)
  constexpr int ZB = B < 32 ? 32 : B;
  const int rank = C > 1 ? (int)cluster_rank() : 0;
  const int mat = (int)blockIdx.x / C;
  const BandDesc d = descs[mat];
  const int mi = d.id >= 0 ? d.id : mat;
  if (skip && skip[mi]) return;
  col0 += (int)blockIdx.y * cpp;       // cpp <= KC <= NC columns per block
  int k = min(kcap - (int)blockIdx.y * cpp, cpp);
  if (nrhs_dev) k = min(k, nrhs_dev[mi] - col0);
  if (k <= 0 || d.n <= 0) return;  // the same decision in every block of the cluster
  const int n = d.n, w = d.w, ld = d.ld;
  const T* Sg = sizeof(T) == 4 && d.scl >= 0 ? base + d.scl : nullptr;  // equilibrated band: solve with S A S
  double* X = xbase + xoff[mi] + (int64_t)col0 * n;
  const int nb = (n + B - 1) / B;
  const int RW = rwb * B;

  extern __shared__ __align__(128) unsigned char smem_raw[];
  Bars* bars = reinterpret_cast<Bars*>(smem_raw);
  T* slots = reinterpret_cast<T*>(smem_raw + sizeof(Bars));
  A* win = reinterpret_cast<A*>(slots + (size_t)nslot * SR * ld);   // RW * NC: solved rows, then partial sums
  A* zb = win + (size_t)RW * NC;                                // ZB * NC
  A* xb = zb + (size_t)ZB * NC;                                     // ZB * NC
  A* mail = xb + (size_t)ZB * NC;                                   // C * B * NC (C > 1)
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int ph = lane & (PH - 1), row = wid * RPW + lane / PH;      // this lane's row
  const int p0 = ph * RPW;                                          // first column (row) of 32 of this lane
  // the column whose sum this lane ends up with, and whether it is the one
  // lane of its row that stores it
  constexpr int LC = PH / NC;
  static_assert(LC >= 1, "a row's lanes must cover the columns");
  const int col = ph / LC;
  const bool mine = ph % LC == 0 && col < k;

  RS rs;
  rs.full = bars->full;
  rs.empty = bars->empty;
  rs.slots = slots;
  rs.ld = ld;
  rs.nslot = nslot;
  const int own = rank < nb ? (nb - rank + C - 1) / C : 0;  // row blocks of this thread block

  for (int i = tid; i < RW * NC; i += kThreads) {
    if (C > 1) unset(win + i);
    else win[i] = A();
  }
  if (C > 1)
    for (int i = tid; i < C * B * NC; i += kThreads) unset(mail + i);
  for (int i = tid; i < ZB * NC; i += kThreads) {
    zb[i] = A();
    xb[i] = A();
  }
  if (tid == 0) {
    for (int s = 0; s < nslot; ++s) {
      mbar_init(&bars->full[s], 1);
      mbar_init(&bars->empty[s], NW);
    }
    fence_barrier_init();
  }
  __syncthreads();
  if (C > 1) cluster_sync();
  if (wid == kThreads / 32) {
    if (lane == 0) rs.produce(base + d.off, n, rank, C, own, st, d.id);
    __syncwarp();
    if (C > 1) cluster_sync();
    return;
  }
  bool ok = true;

  // this lane's element of a block's vector, fetched one visit ahead and
  // converted when it is used (a conversion would wait for the load)
  double xnext = 0.0;
  T snext = T(1);
  auto fetch = [&](int kk) {
    const int r = kk * B + row;
    if (mine && r < n) {
      xnext = X[(int64_t)col * n + r];
      if (Sg) snext = Sg[r];
    }
  };
  auto fetched = [&](double x, T sc) -> A {
    if constexpr (sizeof(T) == 4) return to_arith<A>(cv<T>(x) * sc);
    else return to_arith<A>(x);
  };
  auto value = [](A y) -> double {
    if constexpr (std::is_same_v<A, float>) return f2d_bits(y);
    else return to_double(y);
  };
  // in the diagonal block, within the group of 32 that holds this lane's row:
  // bits of the entries in the lower triangle (forward: columns <= row;
  // backward: rows >= column); the other group of a 64-row block is full or empty
  constexpr bool kMask = NC == 1 && sizeof(T) == 4 && B >= 32;
  uint32_t mf[kMask ? RPW : 1], mb[kMask ? RPW : 1];
  if constexpr (kMask) {
#pragma unroll
    for (int e = 0; e < RPW; ++e) {
      mf[e] = p0 + e <= row % 32 ? 0xffffffffu : 0u;
      mb[e] = p0 + e >= row % 32 ? 0xffffffffu : 0u;
    }
  }
  const int rgrp = R > 1 ? wid * RPW / 32 : 0;   // this warp's group
  auto masked = [](float x, uint32_t m) { return __uint_as_float(__float_as_uint(x) & m); };
  uint32_t rstep[RPW];                 // bytes from this lane's first row to the others, down a column
#pragma unroll
  for (int i = 0; i < RPW; ++i) rstep[i] = (uint32_t)(i * (ld - 1) * (int)sizeof(T));
  // sums over the PH lanes of a row, of which this lane returns column `col`:
  // halving exchanges while a lane still holds several columns
  auto reduce = [&](A* acc) -> A {
    int m = NC;
#pragma unroll
    for (int o = PH / 2; o > 0; o >>= 1) {
      if (m > 1) {
        m >>= 1;
        const bool up = (ph & o) != 0;
#pragma unroll
        for (int c = 0; c < NC / 2; ++c)
          if (c < m) {
            const A give = up ? acc[c] : acc[c + m], keep = up ? acc[c + m] : acc[c];
            acc[c] = keep + shfl_xor(give, o);
          }
      } else {
        acc[0] += shfl_xor(acc[0], o);
      }
    }
    return acc[0];
  };
  // the columns below `seen` that this lane multiplies by (NC > 1: all of them)
  // have arrived
  int seen = 0;
  auto see = [&](const A* yw, int c0, int kb) {   // the group(s) of 32 columns at c0
    if constexpr (NC == 1) {
      if (ok && c0 + 32 * R > seen) {
        A v[RPW * R];
        ok = wait_set<RPW * R>(v, [&](int e) { return yw + 32 * (e / RPW) + e % RPW; },
                               [&](int e) { return B >= 32 || c0 + p0 + e < kb; }, st, d.id, c0);
      }
    }
  };
  auto see_block = [&](int j, int slot) {         // NC > 1: block j, in ring block `slot`
    if ((j & (C - 1)) != rank) {
      A v[1];
      if (mine && ok)
        ok = wait_set<1>(v, [&](int) { return win + (size_t)(slot * B + row) * NC + col; }, [](int) { return true; },
                         st, d.id, j);
      csync<kThreads>();
    }
  };
  const uint32_t win_at = smem_u32(win);

  // ------------------------------------------------------------- forward
  if (own > 0) fetch(rank);
  int rb = rank;                       // ring block of kk (rwb >= C)
  for (int v = 0; v < own; ++v) {
    const int kk = rank + C * v, kb = kk * B;
    const int b = min(B, n - kb);
    const A rhs = fetched(xnext, snext);
    if (v + 1 < own) fetch(kk + C);
    const int part = row / SR;
    if (ok) ok = rs.wait_part(part, st, d.id, v);   // this warp's rows
    // Lr[c] = L(kb + row, c)
    const T* Lr = rs.slot(part) + (ptrdiff_t)(row - part * SR) * ld + (w - kb - row) + p0;
    const uint32_t la = smem_u32(Lr);
    const int cmin = kb + row - w - p0, cmax = kb - p0;   // columns in band, as seen by Lr
    const bool in = row < b;
    if (C > 1) {  // the slots of the blocks that arrive before this one reads on
      for (int i = tid; i < (C - 1) * B * NC; i += kThreads) {
        const int q = rb + 1 + i / (B * NC);
        unset(win + (size_t)(q >= rwb ? q - rwb : q) * B * NC + i % (B * NC));
      }
    }
    A acc[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) acc[c] = A();
    A aw[W];
#pragma unroll
    for (int u = 0; u < W; ++u) aw[u] = A();
    // 32 R columns at a time, aligned; the first ones may lie before the band,
    // the last (B < 32) reach beyond kb
    int c0 = max(0, min(kb - w, (kk - C + 1) * B)) / (32 * R) * (32 * R);
    int pos = rb - (kk - c0 / B);
    pos = (pos < 0 ? pos + rwb : pos) * B + c0 % B;
    const int cfull = kb + B - 1 - w;     // from here every row of the block is in band
    for (; c0 < kb; c0 += 32 * R) {
      const A* yw = win + (size_t)(pos + p0) * NC;
      const T* Lc = Lr + c0;
      if (C > 1) {
        if constexpr (NC == 1) {
          see(yw, c0, kb);
        } else {
          for (; seen < min(c0 + 32 * R, kb); seen += B) {
            const int j = seen / B, q = rb - (kk - j);
            if (j >= c0 / B) see_block(j, q < 0 ? q + rwb : q);
          }
        }
      }
      if (in) {
        if (c0 >= cfull && (B >= 32 || c0 + 32 <= kb)) {
          if constexpr (NC == 1)
            dot_lds<RPW, R>(aw, win_at + (uint32_t)((pos + p0) * sizeof(A)),
                            [&](int e) { return la + (uint32_t)((c0 + 32 * (e / RPW) + e % RPW) * (int)sizeof(T)); },
                            [](T l, int) { return l; });
          else
            madd<RPW, R, NC, KC, T>(acc, yw, [&](int i) { return Lc[i]; }, [](int) { return true; });
        } else
        {
          madd<RPW, R, NC, KC, T>(acc, yw, [&](int i) { return Lc[i]; },
                              [&](int i) { return c0 + i >= cmin && c0 + i < cmax; });
        }
      }
      pos = pos + 32 * R == RW ? 0 : pos + 32 * R;
    }
    if constexpr (NC == 1) {
      seen = kb;
      acc[0] += chains(aw);
    }
    {
      const A t = reduce(acc);
      if (mine) zb[row * NC + col] = in ? rhs - t : A();
    }
    if (C > 1) acquire_cluster();
    csync<kThreads>();
    if (C > 1) release_cluster();
    // y = M z, M the inverted diagonal block (its lower triangle)
#pragma unroll
    for (int c = 0; c < NC; ++c) acc[c] = A();
    if constexpr (kMask) {
      const uint32_t ld0 = la + (uint32_t)(kb * (int)sizeof(T)), z0 = smem_u32(zb + p0), g0 = 32u * sizeof(T) * rgrp;
      A a2[W];
#pragma unroll
      for (int u = 0; u < W; ++u) a2[u] = A();
      if (rgrp > 0)
        dot_lds<RPW, 1>(a2, z0, [&](int e) { return ld0 + (uint32_t)(e * (int)sizeof(T)); },
                        [](T l, int) { return l; });
      dot_lds<RPW, 1>(a2, z0 + g0, [&](int e) { return ld0 + g0 + (uint32_t)(e * (int)sizeof(T)); },
                      [&](T l, int e) { return masked(l, mf[e]); });
      acc[0] = chains(a2);
    } else if (in) {
      madd<RPW, R, NC, KC, T>(acc, zb + (size_t)p0 * NC, [&](int i) { return Lr[kb + i]; },
                          [&](int i) { return p0 + i <= row; });
    }
    {
      const A t = reduce(acc);
      const A y = in ? t : A();
      A* dst = win + (size_t)(rb * B + row) * NC + col;
      const uint32_t off = (uint32_t)((rb * B + row) * NC + col) * (uint32_t)sizeof(A);
      if constexpr (NC == 1) {  // every lane of the row has y
        for (int q = 1 + ph; q < C; q += PH) st_cluster(map_rank(win_at, (uint32_t)((rank + q) & (C - 1))) + off, y);
      } else if (mine) {
        for (int q = 1; q < C; ++q) st_cluster(map_rank(win_at, (uint32_t)((rank + q) & (C - 1))) + off, y);
      }
      if (mine) *dst = y;
      rs.release();
      rb += C;
      if (rb >= rwb) rb -= rwb;
      csync<kThreads>();
      if (mine && in) X[(int64_t)col * n + kb + row] = value(y);
    }
  }
  if (C > 1) {  // every solved block has arrived before the ring changes its use
    const int last = own > 0 ? rank + C * (own - 1) : -1;   // this block's last one
    for (int j = max(last + 1, 0); j < nb; ++j)
    {
      A v[1];
      if (mine && ok)
        ok = wait_set<1>(v, [&](int) { return win + (size_t)((j % rwb) * B + row) * NC + col; },
                         [](int) { return true; }, st, d.id, j);
    }
  }
  csync<kThreads>();

  // ------------------------------------------------------------ backward
  // win now holds one partial sum per row
  for (int i = tid; i < RW * NC; i += kThreads) win[i] = A();
  // mailboxes: mail[q] takes the sums that rank q sends, this block's next row
  // block; a value is unset again by the thread that reads it, before the chain
  // can reach a block whose sum would follow it
  const uint32_t mail_at = smem_u32(mail) + (uint32_t)(rank * B * NC * sizeof(A));
  if (own > 0) fetch(rank + C * (own - 1));
  csync<kThreads>();
  for (int v = own; v < 2 * own; ++v) {
    const int kk = rank + C * (2 * own - 1 - v), kb = kk * B;
    const int b = min(B, n - kb);
    const int nsrc = C > 1 ? min(C - 1, nb - 1 - kk) : 0;
    rb -= C;                                       // ring block of kk
    if (rb < 0) rb += rwb;
    const A yk = fetched(xnext, T(1));
    const T sc = snext;
    if (kk - C >= 0) fetch(kk - C);
    auto ring = [&](int back) -> A* {              // row 0 of block kk - back
      const int q = rb - back;
      return win + (size_t)((q < 0 ? q + rwb : q) * B) * NC;
    };
    // send the sum of (block kk - back, row r, column c) to its owner
    auto send = [&](int back, int r, int c, A s) {
      st_cluster(map_rank(mail_at, (uint32_t)((rank - back) & (C - 1))) + (uint32_t)((r * NC + c) * sizeof(A)), s);
    };
    if (ok) ok = rs.wait(st, d.id, v);
    // rows of the block this lane sums over: 32 q + p0 + i, in slot part of q
    auto rows_of = [&](int q) -> const T* {
      const int t0 = 32 * q + p0, part = t0 / SR;
      return rs.slot(part < HB ? part : 0) - (ptrdiff_t)part * SR * ld + (ptrdiff_t)t0 * (ld - 1) + (row + w);
    };
    const T* S0 = rows_of(0);
    const T* S1 = R > 1 ? rows_of(1) - (ptrdiff_t)32 * (ld - 1) : S0;
    // z = y - the partial sums of this block
    if (mine) {
      A* a = ring(0) + row * NC + col;
      A z = yk - *a;
      *a = A();
      if (nsrc > 0) {
        A v[kMaxC - 1];
        auto at = [&](int q) { return mail + ((size_t)((rank + 1 + q) & (C - 1)) * B + row) * NC + col; };
        if (ok) ok = wait_set<kMaxC - 1>(v, at, [&](int q) { return q < nsrc; }, st, d.id, -1 - kk);
#pragma unroll
        for (int q = kMaxC - 2; q >= 0; --q)
          if (q < nsrc) {
            z -= v[q];
            unset(at(q));
          }
      }
      zb[row * NC + col] = row < b ? z : A();
    }
    if (C > 1) acquire_cluster();
    csync<kThreads>();
    if (C > 1) release_cluster();
    const uint32_t sa0 = smem_u32(S0), sa1 = smem_u32(S1) + (uint32_t)(32 * (ld - 1) * (int)sizeof(T));
    // shared address of entry e of this lane's column, `shift` columns on
    auto row_at = [&](int e, int shift) -> uint32_t {
      return (e < RPW ? sa0 : sa1) + rstep[e % RPW] + (uint32_t)(shift * (int)sizeof(T));
    };
    // sum over the block's rows t = first..last of L(kb + t, kb + row + shift)
    // X(t, .); full: every lane sums over all B rows
    auto column_sum = [&](A* acc, const A* x, int shift, int first, int last, bool full) {
#pragma unroll
      for (int c = 0; c < NC; ++c) acc[c] = A();
      const T *Sa = S0 + shift, *Sb = S1 + shift;
      auto at = [&](int i) { return (i < 32 ? Sa : Sb)[(ptrdiff_t)i * (ld - 1)]; };
      if (full) {
        if constexpr (NC == 1) {
          A a2[W];
#pragma unroll
          for (int u = 0; u < W; ++u) a2[u] = A();
          dot_lds<RPW, R>(a2, smem_u32(x + p0), [&](int e) { return row_at(e, shift); }, [](T l, int) { return l; });
          acc[0] = chains(a2);
        } else
          madd<RPW, R, NC, KC, T>(acc, x + (size_t)p0 * NC, at, [](int) { return true; });
      } else
        madd<RPW, R, NC, KC, T>(acc, x + (size_t)p0 * NC, at,
                            [&](int i) { return p0 + i >= first && p0 + i <= last; });
    };
    // x = M^T z: column `row` of the inverted block
    A acc[NC];
    if constexpr (kMask) {
      if (b == B) {
        const uint32_t z0 = smem_u32(zb + p0);
        A a2[W];
#pragma unroll
        for (int u = 0; u < W; ++u) a2[u] = A();
        dot_lds<RPW, 1>(a2, z0 + 32u * sizeof(T) * rgrp, [&](int e) { return (rgrp > 0 ? sa1 : sa0) + rstep[e]; },
                        [&](T l, int e) { return masked(l, mb[e]); });
        if (R > 1 && rgrp == 0)
          dot_lds<RPW, 1>(a2, z0 + 32u * sizeof(T), [&](int e) { return sa1 + rstep[e]; }, [](T l, int) { return l; });
        acc[0] = chains(a2);
      } else {
        column_sum(acc, zb, 0, row, b - 1, false);
      }
    } else {
      column_sum(acc, zb, 0, row, b - 1, false);
    }
    const A x = reduce(acc);
    if (mine) xb[row * NC + col] = row < b ? x : A();
    csync<kThreads>();
    if (kk > 0) {
      // the link of the chain: contribution to block kk - 1
      {
        A* a = ring(1) + row * NC + col;
        const A old = mine ? *a : A();
        column_sum(acc, xb, -B, 0, min(b - 1, row - B + w), B >= 32 && b == B && w >= 2 * B - 1);
        const A s = reduce(acc) + old;
        if (mine) {
          if (C > 1) send(1, row, col, s);
          *a = C > 1 ? A() : s;
        }
      }
      const int back1 = min(kk, (w + B - 1) / B);   // the band reaches block kk - back1
      if constexpr (kQuad) {
        for (int back = 2; back <= max(back1, min(C - 1, kk)); ++back) {
          A* a = ring(back) + row;
          const A old = mine ? *a : A();
          column_sum(acc, xb, -back * B, 0, min(b - 1, row - back * B + w),
                     B >= 32 && b == B && w >= (back + 1) * B - 1);
          const A s = reduce(acc) + old;
          if (mine) {
            if (back < C) send(back, row, 0, s);
            *a = back < C ? A() : s;
          }
        }
      } else {
        // older blocks: one thread per column, tasks of 32 columns
        const int clo = max(0, kb - w), chi = kb - B;
        if (chi > clo) {
          constexpr int TU = SR < 16 ? SR : 16;
          const int ncg = (chi - clo + 31) >> 5;
          for (int task = wid; task < ncg; task += kThreads / 32) {
            const int cc = chi - 1 - task * 32 - lane;
            if (cc >= clo) {
              const int tmx = min(b - 1, cc - kb + w);
              A a2[NC];
#pragma unroll
              for (int c = 0; c < NC; ++c) a2[c] = A();
#pragma unroll
              for (int t0 = 0; t0 < B; t0 += TU) {
                const int part = t0 / SR;
                const T* S = rs.slot(part) - (ptrdiff_t)part * SR * ld + (cc - kb + w) + (ptrdiff_t)t0 * (ld - 1);
                if (tmx >= t0 + TU - 1)
                  madd<TU, 1, NC, KC, T>(a2, xb + (size_t)t0 * NC, [&](int i) { return S[(ptrdiff_t)i * (ld - 1)]; },
                                     [](int) { return true; });
                else
                  madd<TU, 1, NC, KC, T>(a2, xb + (size_t)t0 * NC, [&](int i) { return S[(ptrdiff_t)i * (ld - 1)]; },
                                     [&](int i) { return t0 + i <= tmx; });
              }
              const int jb = cc / B;
              A* a = ring(kk - jb) + (size_t)(cc - jb * B) * NC;
#pragma unroll
              for (int c = 0; c < KC; ++c) a[c] += a2[c];
            }
          }
        }
        if (C > 2) {
          csync<kThreads>();
          // this block's last word on the blocks kk - 2 .. kk - C + 1
          for (int i = tid; i < (C - 2) * B * k; i += kThreads) {
            const int r = i % B, c = (i / B) % k, back = 2 + i / (B * k);
            if (kk - back < 0) continue;
            A* a = ring(back) + r * NC + c;
            send(back, r, c, *a);
            *a = A();
          }
        }
      }
      rs.release();
    }
    csync<kThreads>();
    if (mine && row < b) {
      if constexpr (std::is_same_v<A, float>) X[(int64_t)col * n + kb + row] = f2d_bits(x * sc);
      else X[(int64_t)col * n + kb + row] = value(x);
    }
  }
  if (C > 1) cluster_sync();  // no block leaves while another may still store into it
}

// ---------------------------------------------------------------------------
// Tensor-core sweep for several right-hand sides (FP32 factors): the same
// chain with every product an m16n8k8 TF32 MMA (three passes: hi*hi + hi*lo +
// lo*hi; PASSES = 1: one pass off the diagonal blocks).  B / 16 row
// tiles x KP k-parts of warps.  The k index of an MMA is permuted so that a
// quad's four lanes read columns (backward: rows) CGS apart: with the band's
// odd address stride ld - 1 that makes the 32 fragment addresses distinct
// banks, and odd column strides of win and zb do the same for B.
// ---------------------------------------------------------------------------
// Sixteen warps: a link is a chain of short steps (shared loads, splits, a few
// MMAs, a barrier), and twice the warps halve each warp's share of all but the
// barrier (elasticity 38x31x24, half width about 500, 24 columns: the 56 sweeps of
// the eigensolver 81 ms with eight warps, 54 ms with sixteen).
constexpr int kMmaWarps = 16;
template <int B, int NT, int PASSES>
__global__ void __launch_bounds__(32 * kMmaWarps + 32, 1)
k_sweep_mma(const float* __restrict__ base, const BandDesc* __restrict__ descs, double* __restrict__ xbase,
            const int64_t* __restrict__ xoff, int col0, int kcap, const int32_t* __restrict__ nrhs_dev,
            const int32_t* __restrict__ skip, int C, int nslot, int rwb, DevStatus* st) {
  using RS = RowStream<float, B>;
  constexpr int SR = RS::SR;
  constexpr int NC = 8 * NT;
  constexpr int NW = kMmaWarps, kThreads = 32 * NW;
  constexpr int MT = B / 16, KP = NW / MT;      // row tiles, k-parts
  constexpr int ST = B / 8;                     // k-steps per block
  constexpr int SPW = ST / KP > 0 ? ST / KP : 1;  // k-steps per warp and block
  constexpr int KPB = ST / SPW;                 // k-parts that share a block
  constexpr int G = KP / KPB;                   // blocks handled side by side
  constexpr int P = kThreads / B;
  constexpr int E = (B * NC + kThreads - 1) / kThreads;
  constexpr int RB = B + 4;                     // column stride of the partial tiles
  constexpr int ZS = B + 1;                     // column stride of zb
  const int rank = C > 1 ? (int)cluster_rank() : 0;
  const int mat = (int)blockIdx.x / C;
  const BandDesc d = descs[mat];
  const int mi = d.id >= 0 ? d.id : mat;
  if (skip && skip[mi]) return;
  col0 += (int)blockIdx.y * NC;
  int k = min(kcap - (int)blockIdx.y * NC, NC);
  if (nrhs_dev) k = min(k, nrhs_dev[mi] - col0);
  if (k <= 0 || d.n <= 0) return;
  const int n = d.n, w = d.w, ld = d.ld;
  const float* Sg = d.scl >= 0 ? base + d.scl : nullptr;
  double* X = xbase + xoff[mi] + (int64_t)col0 * n;
  const int nb = (n + B - 1) / B;
  const int RW = rwb * B, YS = RW + 1;

  extern __shared__ __align__(128) unsigned char smem_raw[];
  Bars* bars = reinterpret_cast<Bars*>(smem_raw);
  float* slots = reinterpret_cast<float*>(smem_raw + slot_lead(C));
  float* win = slots + (size_t)nslot * SR * ld;        // NC columns of YS: solved rows, then partial sums
  float* red = win + (size_t)NC * YS;                  // KP x NC x RB
  float* zb = red + (size_t)KP * NC * RB;              // NC x ZS
  float* mail = zb + (size_t)NC * ZS;                  // C x NC x B (C > 1)
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int g = lane >> 2, tg = lane & 3;
  const int row = tid % B, ph = tid / B;
  const int mt = wid % MT, kp = wid / MT;

  RS rs;
  rs.full = bars->full;
  rs.empty = bars->empty;
  rs.slots = slots;
  rs.ld = ld;
  rs.nslot = nslot;
  const int own = rank < nb ? (nb - rank + C - 1) / C : 0;  // row blocks of this thread block

  for (int i = tid; i < NC * YS; i += kThreads) {
    if (C > 1) unset(win + i);
    else win[i] = 0.f;
  }
  if (C > 1)
    for (int i = tid; i < C * NC * B; i += kThreads) unset(mail + i);
  for (int i = tid; i < NC * ZS; i += kThreads) zb[i] = 0.f;
  if (tid == 0) {
    for (int s = 0; s < nslot; ++s) {
      mbar_init(&bars->full[s], 1);
      mbar_init(&bars->empty[s], NW);
    }
    fence_barrier_init();
  }
  __syncthreads();
  if (C > 1) cluster_sync();
  if (wid == kThreads / 32) {
    if (lane == 0) rs.produce(base + d.off, n, rank, C, own, st, d.id);
    __syncwarp();
    if (C > 1) cluster_sync();
    return;
  }
  bool ok = true;

  // this thread's elements of a block's vectors, fetched one visit ahead and
  // converted when they are used (a conversion would wait for the load)
  double xn[E], xc[E];
  float sn = 1.f, sc = 1.f;
  auto fetch = [&](int kk) {
    const int r = kk * B + row;
    if (Sg && r < n) sn = Sg[r];
#pragma unroll
    for (int e = 0; e < E; ++e) {
      const int c = ph + e * P;
      xn[e] = (c < k && r < n) ? X[(int64_t)c * n + r] : 0.0;
    }
  };
  auto take = [&]() {
    sc = sn;
#pragma unroll
    for (int e = 0; e < E; ++e) xc[e] = xn[e];
  };
  // accumulators: lo * hi, hi * lo, hi * hi (independent chains)
  float acc[NT][3][4];
  auto clear = [&]() {
#pragma unroll
    for (int nt = 0; nt < NT; ++nt)
#pragma unroll
      for (int p = 0; p < 3; ++p)
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[nt][p][q] = 0.f;
  };
  // one k-step: A values x (rows g, g + 8 at the first k; then at the second),
  // B values at shared address b and 4 bytes on, column tiles `bs` bytes apart
  auto step = [&](const float* x, uint32_t b, uint32_t bs, bool three) {
    uint32_t ah[4], al[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      if (PASSES == 3 || three) split_tf32(x[q], ah[q], al[q]);
      else ah[q] = __float_as_uint(tf32_rn(x[q]));
    }
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) {
      float y[2];
      lds(b + bs * nt, y[0]);
      lds(b + bs * nt + 4, y[1]);
      uint32_t bh[2], bl[2];
      if (PASSES == 3 || three) {
        split_tf32(y[0], bh[0], bl[0]);
        split_tf32(y[1], bh[1], bl[1]);
        mma_tf32(acc[nt][0], al, bh);
        mma_tf32(acc[nt][1], ah, bl);
      } else {
        bh[0] = __float_as_uint(tf32_rn(y[0]));
        bh[1] = __float_as_uint(tf32_rn(y[1]));
      }
      mma_tf32(acc[nt][2], ah, bh);
    }
  };
  auto put_red = [&]() {
#pragma unroll
    for (int nt = 0; nt < NT; ++nt)
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int r = 16 * mt + g + ((q & 2) ? 8 : 0), c = 8 * nt + 2 * tg + (q & 1);
        red[((size_t)kp * NC + c) * RB + r] = (acc[nt][0][q] + acc[nt][1][q]) + acc[nt][2][q];
      }
  };
  auto red_sum = [&](int c) {
    float s = red[(size_t)c * RB + row];
#pragma unroll
    for (int p = 1; p < KP; ++p) s += red[((size_t)p * NC + c) * RB + row];
    return s;
  };
  // k positions of an MMA: a quad's lanes are 8 apart (4 in 16-row blocks), the
  // two halves of k next to each other: position kl + 2 i + half of k-step i
  const int gkp = kp / KPB;
  const int s0 = (kp % KPB) * SPW;               // this warp's first k-step in a block
  const int kq = B < 32 ? 0 : s0 >> 2, km = 2 * (B < 32 ? s0 : s0 & 3);   // its 32-row group and place there
  const int kl = 32 * kq + (B < 32 ? 4 : 8) * tg + km;
  const uint32_t win_at = smem_u32(win), zb_at = smem_u32(zb) + (uint32_t)((g * ZS + kl) * 4);
  const uint32_t ys8 = (uint32_t)(8 * YS * 4), zs8 = (uint32_t)(8 * ZS * 4);
  const uint32_t row8 = (uint32_t)(8 * (ld - 1) * 4);
  uint32_t rstep[8];                   // bytes to the following rows of a column
#pragma unroll
  for (int i = 0; i < 8; ++i) rstep[i] = (uint32_t)(i * (ld - 1) * 4);

  // ------------------------------------------------------------- forward
  if (own > 0) fetch(rank);
  int ready = 0, rbk = rank;           // blocks seen; ring block of kk (rwb >= C)
  for (int v = 0; v < own; ++v) {
    const int kk = rank + C * v, kb = kk * B;
    const int b = min(B, n - kb);
    take();
    if (v + 1 < own) fetch(kk + C);
    if (ok) ok = rs.wait(st, d.id, v);
    const int ra = 16 * mt + g, rb8 = ra + 8;     // this lane's rows of the block
    const int half = 16 * mt / SR;
    // shared address of L(kb + ra, kl) in the band (row ra + 8: row8 on)
    const uint32_t la = rs.slot_at(half) + (uint32_t)(slot_offset(kk, ra, kl, w, ld, B, SR) * 4);
    const bool va = ra < b, vb = rb8 < b;
    if (C > 1)  // the slots of the blocks that arrive before this one reads on
      for (int i = tid; i < (C - 1) * B * NC; i += kThreads) {
        const int q = rbk + 1 + (i % ((C - 1) * B)) / B;
        unset(win + (size_t)(i / ((C - 1) * B)) * YS + (q >= rwb ? q - rwb : q) * B + i % B);
      }
    clear();
    const int jlo = forward_first(kk, w, B, C);
    int rb = rbk - (kk - jlo);
    if (rb < 0) rb += rwb;
    for (int j = jlo; j < kk; ++j) {
      if (C > 1 && j >= ready) {
        if ((j & (C - 1)) != rank) {
          float v[E];
          if (ok)
            ok = wait_set<E>(v, [&](int e) { return win + (size_t)(ph + e * P) * YS + rb * B + row; },
                             [&](int e) { return ph + e * P < k; }, st, d.id, j);
          acquire_cluster();
          csync<kThreads>();
        }
        ready = j + 1;
      }
      if (G == 1 || (j - jlo) % G == gkp) {
        const bool fullb = b == B && j * B >= kb + B - 1 - w;
        const uint32_t lj = la + (uint32_t)(j * B * 4), wj = win_at + (uint32_t)((g * YS + rb * B + kl) * 4);
        const int ca = kb + ra - w - j * B - kl, cb = ca + 8;   // first columns in band, from kl
#pragma unroll
        for (int i = 0; i < SPW; ++i) {
          float x[4];
          lds(lj + 8 * i, x[0]);
          lds(lj + row8 + 8 * i, x[1]);
          lds(lj + 8 * i + 4, x[2]);
          lds(lj + row8 + 8 * i + 4, x[3]);
          if (!fullb) {
            x[0] = va && 2 * i >= ca ? x[0] : 0.f;
            x[1] = vb && 2 * i >= cb ? x[1] : 0.f;
            x[2] = va && 2 * i + 1 >= ca ? x[2] : 0.f;
            x[3] = vb && 2 * i + 1 >= cb ? x[3] : 0.f;
          }
          step(x, wj + 8 * i, ys8, false);
        }
      }
      rb = rb + 1 == rwb ? 0 : rb + 1;
    }
    put_red();
    csync<kThreads>();
#pragma unroll
    for (int e = 0; e < E; ++e) {
      const int c = ph + e * P;
      if (c < k) zb[c * ZS + row] = row < b ? d2f_bits(xc[e]) * sc - red_sum(c) : 0.f;
    }
    csync<kThreads>();
    if (C > 1) release_cluster();
    // y = M z
    clear();
    if (gkp == 0) {
      const uint32_t lj = la + (uint32_t)(kb * 4);
#pragma unroll
      for (int i = 0; i < SPW; ++i) {
        float x[4];
        lds(lj + 8 * i, x[0]);
        lds(lj + row8 + 8 * i, x[1]);
        lds(lj + 8 * i + 4, x[2]);
        lds(lj + row8 + 8 * i + 4, x[3]);
        x[0] = va && kl + 2 * i <= ra ? x[0] : 0.f;
        x[1] = vb && kl + 2 * i <= rb8 ? x[1] : 0.f;
        x[2] = va && kl + 2 * i + 1 <= ra ? x[2] : 0.f;
        x[3] = vb && kl + 2 * i + 1 <= rb8 ? x[3] : 0.f;
        step(x, zb_at + 8 * i, zs8, true);
      }
    }
    put_red();
    csync<kThreads>();
    {
#pragma unroll
      for (int e = 0; e < E; ++e) {
        const int c = ph + e * P;
        if (c < k) {
          const float y = row < b ? red_sum(c) : 0.f;
          float* dst = win + (size_t)c * YS + rbk * B + row;
          for (int q = 1; q < C; ++q)
            st_cluster(map_rank(win_at, (uint32_t)((rank + q) & (C - 1))) + (uint32_t)(c * YS + rbk * B + row) * 4u, y);
          *dst = y;
          if (row < b) X[(int64_t)c * n + kb + row] = f2d_bits(y);
        }
      }
    }
    rs.release();
    rbk += C;
    if (rbk >= rwb) rbk -= rwb;
    csync<kThreads>();
  }
  if (C > 1) {
    const int last = own > 0 ? rank + C * (own - 1) : -1;
    for (int j = max(last + 1, 0); j < nb; ++j)
    {
      float v[E];
      if (ok)
        ok = wait_set<E>(v, [&](int e) { return win + (size_t)(ph + e * P) * YS + (j % rwb) * B + row; },
                         [&](int e) { return ph + e * P < k; }, st, d.id, j);
    }
  }
  csync<kThreads>();

  // ------------------------------------------------------------ backward
  for (int i = tid; i < NC * YS; i += kThreads) win[i] = 0.f;
  const uint32_t mail_at = smem_u32(mail) + (uint32_t)(rank * NC * B) * 4u;
  if (own > 0) fetch(rank + C * (own - 1));
  csync<kThreads>();
  for (int v = own; v < 2 * own; ++v) {
    const int kk = rank + C * (2 * own - 1 - v), kb = kk * B;
    const int b = min(B, n - kb);
    const int nsrc = C > 1 ? min(C - 1, nb - 1 - kk) : 0;
    rbk -= C;
    if (rbk < 0) rbk += rwb;
    auto rpos = [&](int back) {  // ring position of block kk - back
      const int q = rbk - back;
      return (q < 0 ? q + rwb : q) * B;
    };
    take();
    if (kk - C >= 0) fetch(kk - C);
    if (ok) ok = rs.wait(st, d.id, v);
#pragma unroll
    for (int e = 0; e < E; ++e) {
      const int c = ph + e * P;
      if (c < k) {
        float* a = win + (size_t)c * YS + rbk * B + row;
        float s = *a;
        *a = 0.f;
        if (nsrc > 0) {
          float v[kMaxC - 1];
          auto at = [&](int q) { return mail + ((size_t)((rank + 1 + q) & (C - 1)) * NC + c) * B + row; };
          if (ok) ok = wait_set<kMaxC - 1>(v, at, [&](int q) { return q < nsrc; }, st, d.id, -1 - kk);
#pragma unroll
          for (int q = kMaxC - 2; q >= 0; --q)
            if (q < nsrc) {
              s += v[q];
              unset(at(q));
            }
        }
        zb[c * ZS + row] = row < b ? d2f_bits(xc[e]) - s : 0.f;
      }
    }
    if (C > 1) acquire_cluster();
    csync<kThreads>();
    if (C > 1) release_cluster();
    // x = M^T z: A(m = column, k = row t) = M(t, m)
    clear();
    const int ca = 16 * mt + g, cb = ca + 8;
    // shared address of (row 32 q + CL tg of the block, column kb), q = the
    // 32-row group; CL the distance of a quad's lanes
    constexpr int CL = B < 32 ? 4 : 8;
    uint32_t sq[B > 32 ? 2 : 1];
#pragma unroll
    for (int q = 0; q < (B > 32 ? 2 : 1); ++q)
      sq[q] = rs.slot_at(q) + (uint32_t)((CL * tg * ld - 32 * q - CL * tg + w) * 4);
    // this warp's k-steps: rows kl + 2 i + half
    const uint32_t sk = sq[B > 32 ? kq : 0] + (uint32_t)(km * (ld - 1) * 4);
    if (gkp == 0) {
#pragma unroll
      for (int i = 0; i < SPW; ++i) {
        const uint32_t s1 = sk + rstep[2 * i] + (uint32_t)(ca * 4), s2 = sk + rstep[2 * i + 1] + (uint32_t)(ca * 4);
        const int t1 = kl + 2 * i, t2 = t1 + 1;
        float x[4];
        lds(s1, x[0]);
        lds(s1 + 32, x[1]);
        lds(s2, x[2]);
        lds(s2 + 32, x[3]);
        x[0] = t1 < b && t1 >= ca ? x[0] : 0.f;
        x[1] = t1 < b && t1 >= cb ? x[1] : 0.f;
        x[2] = t2 < b && t2 >= ca ? x[2] : 0.f;
        x[3] = t2 < b && t2 >= cb ? x[3] : 0.f;
        step(x, zb_at + 8 * i, zs8, true);
      }
    }
    put_red();
    csync<kThreads>();
#pragma unroll
    for (int e = 0; e < E; ++e) {
      const int c = ph + e * P;
      if (c < k) {
        const float xx = row < b ? red_sum(c) : 0.f;
        zb[c * ZS + row] = xx;
        if (row < b) X[(int64_t)c * n + kb + row] = f2d_bits(xx * sc);
      }
    }
    csync<kThreads>();
    if (kk > 0) {
      // the link of the chain: contribution to block kk - 1
      clear();
      if (gkp == 0) {
        const int o0 = ca - B + w - kl;      // band offset of (first row, column a)
        const bool fullb = b == B && w >= 2 * B - 1;
#pragma unroll
        for (int i = 0; i < SPW; ++i) {
          const uint32_t s1 = sk + rstep[2 * i] + (uint32_t)((ca - B) * 4);
          const uint32_t s2 = sk + rstep[2 * i + 1] + (uint32_t)((ca - B) * 4);
          float x[4];
          lds(s1, x[0]);
          lds(s1 + 32, x[1]);
          lds(s2, x[2]);
          lds(s2 + 32, x[3]);
          if (!fullb) {
            const bool v1 = kl + 2 * i < b, v2 = kl + 2 * i + 1 < b;
            x[0] = v1 && o0 - 2 * i >= 0 ? x[0] : 0.f;
            x[1] = v1 && o0 + 8 - 2 * i >= 0 ? x[1] : 0.f;
            x[2] = v2 && o0 - 2 * i - 1 >= 0 ? x[2] : 0.f;
            x[3] = v2 && o0 + 7 - 2 * i >= 0 ? x[3] : 0.f;
          }
          step(x, zb_at + 8 * i, zs8, false);
        }
      }
      put_red();
      csync<kThreads>();
      {
        const uint32_t to = (uint32_t)((kk - 1) & (C - 1));
#pragma unroll
        for (int e = 0; e < E; ++e) {
          const int c = ph + e * P;
          if (c < k) {
            float* a = win + (size_t)c * YS + rpos(1) + row;
            const float s = *a + red_sum(c);
            if (C > 1) {
              *a = 0.f;
              st_cluster(map_rank(mail_at, to) + (uint32_t)(c * B + row) * 4u, s);
            } else {
              *a = s;
            }
          }
        }
      }
      // older blocks: tiles of 16 columns, one warp each, all rows
      const int jlo = max(0, (kb - w + B) / B - 1);
      const int ntile = (kk - 1 - jlo) * MT;
      for (int tile = wid; tile < ntile; tile += kThreads / 32) {
        const int j = jlo + tile / MT;
        const int cg = 16 * (tile % MT) + g;
        const uint32_t wp = win_at + (uint32_t)((2 * tg * YS + rpos(kk - j) + cg) * 4);
        const int c0 = (j - kk) * B + cg;     // column a relative to kb
        const bool fullb = b == B && j * B >= kb + B - 1 - w;
#pragma unroll
        for (int nt = 0; nt < NT; ++nt)
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            acc[nt][0][q] = acc[nt][1][q] = 0.f;
            lds(wp + ys8 * nt + ((q & 1) ? (uint32_t)(YS * 4) : 0u) + ((q & 2) ? 32u : 0u), acc[nt][2][q]);
          }
        const uint32_t zt = smem_u32(zb) + (uint32_t)((g * ZS + CL * tg) * 4);
#pragma unroll
        for (int q = 0; q < (B > 32 ? 2 : 1); ++q) {
          const uint32_t st0 = sq[q] + (uint32_t)(c0 * 4);
          const int o0 = c0 + w - 32 * q - CL * tg, tb = b - 32 * q - CL * tg;
#pragma unroll
          for (int i = 0; i < (B < 32 ? 2 : 4); ++i) {
            const uint32_t s1 = st0 + rstep[2 * i], s2 = st0 + rstep[2 * i + 1];
            float x[4];
            lds(s1, x[0]);
            lds(s1 + 32, x[1]);
            lds(s2, x[2]);
            lds(s2 + 32, x[3]);
            if (!fullb) {
              const bool v1 = 2 * i < tb, v2 = 2 * i + 1 < tb;
              x[0] = v1 && o0 - 2 * i >= 0 ? x[0] : 0.f;
              x[1] = v1 && o0 + 8 - 2 * i >= 0 ? x[1] : 0.f;
              x[2] = v2 && o0 - 2 * i - 1 >= 0 ? x[2] : 0.f;
              x[3] = v2 && o0 + 7 - 2 * i >= 0 ? x[3] : 0.f;
            }
            step(x, zt + (uint32_t)(32 * q * 4) + 8 * i, zs8, false);
          }
        }
#pragma unroll
        for (int nt = 0; nt < NT; ++nt)
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const uint32_t p = wp + ys8 * nt + ((q & 1) ? (uint32_t)(YS * 4) : 0u) + ((q & 2) ? 32u : 0u);
            asm volatile("st.shared.f32 [%0], %1;" ::"r"(p),
                         "f"((acc[nt][0][q] + acc[nt][1][q]) + acc[nt][2][q])
                         : "memory");
          }
      }
      rs.release();
      csync<kThreads>();
      if (C > 2) {
        for (int i = tid; i < (C - 2) * B * k; i += kThreads) {
          const int r = i % B, c = (i / B) % k, jb = kk - 2 - i / (B * k);
          if (jb < 0) continue;
          float* a = win + (size_t)c * YS + rpos(kk - jb) + r;
          const float s = *a;
          *a = 0.f;
          const uint32_t to = (uint32_t)(jb & (C - 1));
          st_cluster(map_rank(mail_at, to) + (uint32_t)(c * B + r) * 4u, s);
        }
        csync<kThreads>();
      }
    }
  }
  if (C > 1) cluster_sync();
}

// ---------------------------------------------------------------------------
// The inverses M of the blk x blk diagonal blocks of L, written over the
// blocks' lower triangles (w >= blk - 1, so the triangle lies in the band).
// One thread block per diagonal block; thread c forms column c by forward
// substitution in arithmetic A (double-single for FP32 bands: FP64 runs at
// 1/64 of the FP32 rate here) and rounds it to T.  Four rows at a time: four
// independent sums hide the latency of a double-single sum that one or two
// rows left bare, and share each loaded value of X.
// ---------------------------------------------------------------------------
template <typename A, typename T>
__device__ __forceinline__ void blkinv_fma(A& s, T l, const A& x) {
  if constexpr (std::is_same_v<A, dsv> && std::is_same_v<T, float>) {
    DS v{s.h, s.l};
    ds_fma1(v, l, x.h, x.l);
    s = dsv(v.h, v.l);
  } else {
    s += factor_value<A>(l) * x;
  }
}
template <typename T, typename A, int B>
constexpr size_t blkinv_smem() {
  return sizeof(A) * (B * B + B) + sizeof(T) * B * (B + 4);
}
template <typename T, typename A, int B>
__global__ void __launch_bounds__(B < 32 ? 32 : B)
k_band_blkinv(T* __restrict__ base, const BandDesc* __restrict__ descs) {
  constexpr int LT = B + 4;
  const BandDesc d = descs[blockIdx.y];
  const int kb = (int)blockIdx.x * B;
  if (kb >= d.n || d.blk != B) return;
  const int b = min(B, d.n - kb), w = d.w, ld = d.ld;
  T* L = base + d.off + (int64_t)kb * ld + w;   // L(kb + r, kb + c) at r * ld + c - r
  extern __shared__ __align__(128) unsigned char smem_raw[];
  A* Xs = reinterpret_cast<A*>(smem_raw);   // B x B
  A* Rs = Xs + B * B;                       // reciprocal pivots
  T* Lt = reinterpret_cast<T*>(Rs + B);     // L(r, t) at t * LT + r
  const int nt = blockDim.x, c = threadIdx.x;
#pragma unroll 8
  for (int i = c; i < B * B; i += nt) {
    const int r = i / B, cc = i % B;
    Lt[cc * LT + r] = (r < b && cc <= r) ? L[(int64_t)r * ld + cc - r] : T(0);
  }
  if (c < B) Rs[c] = c < b ? recip_arith<A>(L[(int64_t)c * ld]) : A();
  __syncthreads();
  if (c < B) {
    const int w0 = c & ~31;   // this warp's columns are zero above row w0
    for (int r0 = w0; r0 < b; r0 += 4) {
      A s[4] = {};
#pragma unroll 2
      for (int t = w0; t < r0; ++t) {
        T l[4];
        load_n<4>(Lt + t * LT + r0, l);
        const A x = Xs[t * B + c];
#pragma unroll
        for (int i = 0; i < 4; ++i) blkinv_fma<A>(s[i], l[i], x);
      }
      A x[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
#pragma unroll
        for (int q = 0; q < i; ++q) blkinv_fma<A>(s[i], Lt[(r0 + q) * LT + r0 + i], x[q]);
        const A one = r0 + i == c ? to_arith<A>(1.0) : A();
        x[i] = (one - s[i]) * Rs[r0 + i];
        Xs[(r0 + i) * B + c] = x[i];
      }
    }
    for (int r = c; r < b; ++r) L[(int64_t)r * ld + c - r] = (T)to_double(Xs[r * B + c]);
  }
}

// ---------------------------------------------------------------------------
// Launches.
// ---------------------------------------------------------------------------
constexpr size_t kSmemMax = 227 * 1024;

template <typename T, typename A, int NC, int B>
size_t sweep_smem(int w, int C, int nslot) {
  constexpr size_t SR = RowStream<T, B>::SR, ZB = B < 32 ? 32 : B;
  return sizeof(Bars) + sizeof(T) * nslot * SR * band_ld(w) +
         sizeof(A) * NC * ((size_t)ring_blocks(w, B, C) * B + 2 * ZB + (C > 1 ? (size_t)C * B : 0));
}
template <int B, int NT>
size_t mma_smem(int w, int C, int nslot) {
  const size_t SR = B < 32 ? B : 32, NC = 8 * NT, KP = kMmaWarps / (B / 16);
  return slot_lead(C) + sizeof(float) * (nslot * SR * band_ld(w) + NC * ((size_t)ring_blocks(w, B, C) * B + 1) +
                                         KP * NC * (B + 4) + NC * (B + 1) + (C > 1 ? (size_t)C * NC * B : 0));
}

template <typename K, typename... Args>
geneo_status_t launch_cluster(K kern, int threads, dim3 grid, int C, size_t smem, cudaStream_t s, Args... args) {
  GENEO_CUDA(allow_smem(kern));
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)C;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = C > 1 ? 1 : 0;
  GENEO_CUDA(cudaLaunchKernelEx(&cfg, kern, args...));
  note_launch();
  return GENEO_OK;
}

struct SweepArgs {
  const BandDesc* d;
  double* x;
  const int64_t* xoff;
  int count, w, c0, kc;
  const int32_t *nrhs_dev, *skip;
  DevStatus* st;
  cudaStream_t s;
  int live;    // matrices of the whole solve set
  int slots;   // wanted row slots (2-4), 0 = as many as fit
};

// Clusters of C = 1 << i thread blocks, one block per SM, that the current device
// runs at the same time (any thread), looked up once per device.  A cluster lies in
// one GPC: of 152 SMs, 76 clusters of 2, 36 of 4 and 15 of 8.
inline int cluster_count(int i) {
  static std::atomic<int> fit[64][4];
  const int C = 1 << i;
  int dev = 0, n = 0;
  if (C == 1 || cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return std::max(sm_count() / C, 1);
  if ((n = fit[dev][i].load(std::memory_order_relaxed)) > 0) return n;
  const auto kern = k_sweep<float, float, 1, 64, 1>;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(C);
  cfg.blockDim = dim3(32 * sweep_warps<1, 64>() + 32);
  cfg.dynamicSmemBytes = 114 * 1024;   // more than half of an SM's
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)C;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  if (allow_smem(kern) != cudaSuccess || cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess || n <= 0) {
    cudaGetLastError();
    return std::max(sm_count() / C, 1);
  }
  fit[dev][i].store(n, std::memory_order_relaxed);
  return n;
}

// slots that fit beside the rest, capped at `want` (0 = kMaxSlots); 0 = none
template <typename F>
int fit_slots(F bytes, int need, int want) {
  for (int s = std::min(want > 0 ? want : kMaxSlots, kMaxSlots); s >= need; --s)
    if (bytes(s) <= kSmemMax) return s;
  return 0;
}

template <typename T, typename A, int NC, int B, int KC = NC>
geneo_status_t run_sweep(const T* base, const SweepArgs& a, int C, int parts, int cpp = KC) {
  constexpr int HB = RowStream<T, B>::HB;
  const int want = a.slots;
  int nslot = 0;
  for (;; C >>= 1) {
    nslot = fit_slots([&](int s) { return sweep_smem<T, A, NC, B>(a.w, C, s); }, HB, std::max(want, HB));
    if (nslot == 0 || want == 0)
      nslot = fit_slots([&](int s) { return sweep_smem<T, A, NC, B>(a.w, C, s); }, HB, 0);
    if (nslot > 0 || C == 1) break;
  }
  if (nslot == 0) return GENEO_ERR_ARG;
  return launch_cluster(k_sweep<T, A, NC, B, KC>, 32 * sweep_warps<NC, B>() + 32, dim3(a.count * C, parts), C,
                        sweep_smem<T, A, NC, B>(a.w, C, nslot), a.s, base, a.d, a.x, a.xoff, a.c0, a.kc, a.nrhs_dev,
                        a.skip, cpp, C, nslot, ring_blocks(a.w, B, C), a.st);
}

template <int B, int NT>
geneo_status_t run_mma(const float* base, const SweepArgs& a, int C, int parts, int passes) {
  constexpr int HB = RowStream<float, B>::HB;
  int nslot = 0;
  for (;; C >>= 1) {
    nslot = fit_slots([&](int s) { return mma_smem<B, NT>(a.w, C, s); }, HB, 0);
    if (nslot > 0 || C == 1) break;
  }
  if (nslot == 0) return GENEO_ERR_ARG;
  return launch_cluster(passes == 1 ? k_sweep_mma<B, NT, 1> : k_sweep_mma<B, NT, 3>, 32 * kMmaWarps + 32,
                        dim3(a.count * C, parts), C, mma_smem<B, NT>(a.w, C, nslot), a.s, base, a.d, a.x, a.xoff, a.c0,
                        a.kc, a.nrhs_dev, a.skip, C, nslot, ring_blocks(a.w, B, C), a.st);
}

}  // namespace

// Rows per block of the sweeps for a band of half width w (w >= 15): the most
// whose rows fit in shared memory at once beside the windows.  Room to stream
// ahead counts for less than longer links (half width 660, 27 matrices, C = 4:
// 466 us with 32 rows and a second block streaming in, 283 us with 64 and none;
// the other blocks of the cluster work while the rows arrive).  0: too wide,
// the factor stays as it is for the streamed kernels of band.cu.
int sweep_block(int w, bool f64) {
  if (f64) {
    if (w >= 31 && sweep_smem<double, double, 4, 32>(w, 1, 2) <= kSmemMax) return 32;
    if (sweep_smem<double, double, 4, 16>(w, 1, 1) <= kSmemMax) return 16;
    if (sweep_smem<double, double, 4, 8>(w, 1, 1) <= kSmemMax) return 8;
    return 0;
  }
  if (w >= 63 && mma_smem<64, 1>(w, 1, 2) <= kSmemMax) return 64;
  if (w >= 31 && mma_smem<32, 1>(w, 1, 1) <= kSmemMax) return 32;
  if (mma_smem<16, 1>(w, 1, 1) <= kSmemMax) return 16;
  if (sweep_smem<float, float, 4, 8>(w, 1, 1) <= kSmemMax) return 8;
  return 0;
}

void sweep_prepare() {
  for (int i = 1; i < 4; ++i) cluster_count(i);
}

template <typename T>
geneo_status_t band_blkinv(T* base, const BandDesc* d_desc, int count, int max_n, int blk_mask, cudaStream_t s) {
  using A = std::conditional_t<sizeof(T) == 4, dsv, double>;
#define GENEO_INV(B)                                                                                       \
  if (blk_mask & B) {                                                                                      \
    GENEO_CUDA(allow_smem(k_band_blkinv<T, A, B>));                                                        \
    k_band_blkinv<T, A, B><<<dim3((max_n + B - 1) / B, count), B < 32 ? 32 : B, blkinv_smem<T, A, B>(), s>>>( \
        base, d_desc);                                                                                     \
    note_launch();                                                                                         \
  }
  if constexpr (sizeof(T) == 4) { GENEO_INV(64) }
  GENEO_INV(32) GENEO_INV(16) GENEO_INV(8)
#undef GENEO_INV
  GENEO_CUDA(cudaGetLastError());
  return GENEO_OK;
}

// The batch is cut so that its blocks fill the GPU: first by the cluster size
// C (each doubling halves what every block streams and multiplies), then by
// columns.
template <typename T, bool DS>
geneo_status_t sweep_solve(const T* base, const BandDesc* d_desc, int count, int blk, int max_w, int max_n,
                           double* xbase, const int64_t* xoff, int nrhs, const int32_t* nrhs_dev,
                           const int32_t* skip_dev, DevStatus* st, cudaStream_t s, int tc_passes, int slots,
                           int live) {
  SweepArgs a{d_desc, xbase, xoff, count, max_w, 0, nrhs, nrhs_dev, skip_dev, st, s, live, slots};
  // C thread blocks per matrix: the waves of blocks times the length of one
  // matrix's sweep, relative to C = 1 (rel: between what the kernels measured at
  // half widths 307-463: FP32 one column 1, 0.57, 0.35, 0.36; MMA 1, 0.54, 0.44;
  // FP64 1, 0.54, 0.45); a
  // block is solved from the ceil(w / blk) before it, which bounds what C can
  // share, and each thread block has at least two.  (Waves of SMs / C clusters sent
  // 16 to 19 matrices to C = 8 in what are two waves: one column of 18 FP32 bands of
  // order 9000, half width 672, 402 us, and 312 on C = 4; FP64, 6859 and 381, 2245
  // and 1119.)
  auto clusters = [&](int units, double* len = nullptr) {
    const double rel[4] = {1.0, 0.56, 0.40, 0.38};
    int best = 1;
    double least = 1e300;
    for (int i = 0, C = 1; C <= kMaxC; ++i, C *= 2) {
      if (C > 1 && (C * blk > max_w + blk - 1 || (max_n > 0 && max_n < 2 * C * blk))) break;
      const int64_t per_wave = cluster_count(i), waves = ((int64_t)live * units + per_wave - 1) / per_wave;
      if (waves * rel[i] < least - 1e-9) {
        least = waves * rel[i];
        best = C;
      }
    }
    if (len) *len = least;
    return best;
  };
  if (nrhs == 1) {
    const int C = clusters(1);
    a.kc = 1;
    if constexpr (sizeof(T) == 4) {
      if (blk == 64) return run_sweep<T, T, 1, 64>(base, a, C, 1);
    }
    if (blk == 32) return run_sweep<T, T, 1, 32>(base, a, C, 1);
    if (blk == 16) return run_sweep<T, T, 1, 16>(base, a, C, 1);
    return run_sweep<T, T, 1, 8>(base, a, C, 1);
  }
  if constexpr (sizeof(T) == 4) {
    if (blk >= 16) {
      for (int c0 = 0; c0 < nrhs; c0 += 32) {
        a.c0 = c0;
        a.kc = std::min(32, nrhs - c0);
        // one or two column tiles of 8 per block: two take 1.5 times as long per
        // block and need half as many (64 bands of order 6859, half width 381,
        // 12 columns: 662 us in two parts of one tile on single blocks, 562 us in
        // one part of two on clusters of 2; 27 of order 9261, half width 463:
        // 593 and 645 us)
        int parts = (a.kc + 7) / 8;
        double len1;
        int C = clusters(parts, &len1);
        bool two = parts > 1 && (blk == 64   ? mma_smem<64, 2>(max_w, 1, 2)
                                 : blk == 32 ? mma_smem<32, 2>(max_w, 1, 2)
                                             : mma_smem<16, 2>(max_w, 1, 2)) <= kSmemMax;
        if (two) {
          double len2;
          const int C2 = clusters((parts + 1) / 2, &len2);
          two = 1.5 * len2 < len1;
          if (two) {
            C = C2;
            parts = (parts + 1) / 2;
          }
        }
        geneo_status_t rc;
        if (two)
          rc = blk == 64 ? run_mma<64, 2>(base, a, C, parts, tc_passes)
             : blk == 32 ? run_mma<32, 2>(base, a, C, parts, tc_passes) : run_mma<16, 2>(base, a, C, parts, tc_passes);
        else
          rc = blk == 64 ? run_mma<64, 1>(base, a, C, parts, tc_passes)
             : blk == 32 ? run_mma<32, 1>(base, a, C, parts, tc_passes) : run_mma<16, 1>(base, a, C, parts, tc_passes);
        GENEO_TRY(rc);
      }
      return GENEO_OK;
    }
    const int parts = (nrhs + 3) / 4;
    return run_sweep<T, T, 4, 8>(base, a, clusters(parts), parts);
  } else {
    using A = std::conditional_t<DS, dsv, double>;
    // the columns cut into parts of cpp per block (kernels for 3, 4 and 8); the
    // FP64 and double-single pipes are full with one block per SM, so the time
    // is the waves times the columns formed times the sweep's relative length
    // (27 FP64 bands of order 9261, half width 463, single blocks: 8.9 ms for 3
    // columns, 11.4 for 4, 21.9 for 8, and 0.52 and 0.40 of that on clusters of 2 and
    // 4; so 11 columns take 8.9 ms in four parts of 3, 11.4 in three of 4 or in two
    // of 6 on clusters of 2)
    const bool fit8 = (blk == 32   ? sweep_smem<double, A, 8, 32>(max_w, 1, 2)
                       : blk == 16 ? sweep_smem<double, A, 8, 16>(max_w, 1, 1)
                                   : sweep_smem<double, A, 8, 8>(max_w, 1, 1)) <= kSmemMax;
    const int most = fit8 ? 8 : 4;
    int parts = (nrhs + most - 1) / most, C = 1;
    double least = 1e300;
    for (int p = parts; p <= nrhs; ++p) {
      const int cpp = (nrhs + p - 1) / p;
      if (p > parts && cpp == (nrhs + p - 2) / (p - 1)) continue;   // no narrower than with one part less
      double len;
      const int c = clusters(p, &len);
      len *= cpp <= 3 ? 3.7 : cpp <= 4 ? 4.7 : 8.7;   // and the latency of a link
      if (len < least - 1e-9) {
        least = len;
        parts = p;
        C = c;
      }
      if (cpp <= 3) break;
    }
    const int cpp = (nrhs + parts - 1) / parts;
    if (cpp <= 3) {
      if (blk == 32) return run_sweep<T, A, 4, 32, 3>(base, a, C, parts, cpp);
      if (blk == 16) return run_sweep<T, A, 4, 16, 3>(base, a, C, parts, cpp);
    }
    if (cpp <= 4) {
      if (blk == 32) return run_sweep<T, A, 4, 32>(base, a, C, parts, cpp);
      if (blk == 16) return run_sweep<T, A, 4, 16>(base, a, C, parts, cpp);
      return run_sweep<T, A, 4, 8>(base, a, C, parts, cpp);
    }
    if (blk == 32) return run_sweep<T, A, 8, 32>(base, a, C, parts, cpp);
    if (blk == 16) return run_sweep<T, A, 8, 16>(base, a, C, parts, cpp);
    return run_sweep<T, A, 8, 8>(base, a, C, parts, cpp);
  }
}

template geneo_status_t band_blkinv<float>(float*, const BandDesc*, int, int, int, cudaStream_t);
template geneo_status_t band_blkinv<double>(double*, const BandDesc*, int, int, int, cudaStream_t);
template geneo_status_t sweep_solve<float, false>(const float*, const BandDesc*, int, int, int, int, double*,
                                                  const int64_t*, int, const int32_t*, const int32_t*, DevStatus*,
                                                  cudaStream_t, int, int, int);
template geneo_status_t sweep_solve<double, false>(const double*, const BandDesc*, int, int, int, int, double*,
                                                   const int64_t*, int, const int32_t*, const int32_t*, DevStatus*,
                                                   cudaStream_t, int, int, int);
template geneo_status_t sweep_solve<double, true>(const double*, const BandDesc*, int, int, int, int, double*,
                                                  const int64_t*, int, const int32_t*, const int32_t*, DevStatus*,
                                                  cudaStream_t, int, int, int);

}  // namespace geneo
