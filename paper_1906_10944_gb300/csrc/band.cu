// Batched banded Cholesky factorisation and triangular solves.
//
// The local Dirichlet matrices A_j = R_j A R_j^T (Section 3), the shifted
// Neumann matrices K_j = Atilde_j - sigma B_j of the spectral transformation
// (Section 4.4) and the coarse matrix A_H (Section 4.5) are all banded in the
// natural (lexicographic) dof order of a box subdomain, so one banded kernel
// family serves all three.  One thread block owns one matrix; the batch is
// the grid (FP64 batches smaller than the GPU: every panel over all SMs, below).
// Storage: lower band by rows (BandDesc in common.cuh).
//
// Factorisation (right-looking, block width NB): per step the NB x NB
// diagonal block is factored by one warp, the panel rows below are solved
// against it (one thread per row, registers), and the trailing w x w
// triangle receives the rank-NB update in 4x4 register tiles.  Pivots that
// are not positive are reported (GENEO_ERR_NOT_SPD) and replaced by 1 so the
// kernel always finishes.
//
// The solves run in sweep.cu; what follows is the kernel for bands too wide for
// its row blocks.  L L^T x = b, in place: the factor is streamed block row by block
// row (SNB rows, one contiguous chunk) into shared memory by bulk copies on
// an mbarrier pipeline.  The forward sweep is left-looking (each new row is
// a dot product with the last w solved rows, kept in a shared ring), the
// backward sweep right-looking (the rows above the current block are
// updated in the shared ring); diagonal blocks are solved by warp shuffles.
// The factor is read once per sweep; b and x once each.
#include "common.cuh"
#include "ds.cuh"
#include "pivot.h"
#include "ptx.cuh"

namespace geneo {

namespace {

constexpr int kThreads = 256;

template <typename T>
__device__ __forceinline__ bool finite_pos(T v) { return v > T(0) && isfinite(v); }

// four consecutive values from 16-byte aligned shared memory
__device__ __forceinline__ void load4(const float* p, float* o) {
  const float4 v = *reinterpret_cast<const float4*>(p);
  o[0] = v.x; o[1] = v.y; o[2] = v.z; o[3] = v.w;
}
__device__ __forceinline__ void load4(const double* p, double* o) {
  const double2 a = *reinterpret_cast<const double2*>(p);
  const double2 c = *reinterpret_cast<const double2*>(p + 2);
  o[0] = a.x; o[1] = a.y; o[2] = c.x; o[3] = c.y;
}

__device__ __forceinline__ void store4(float* p, const float* o) {
  *reinterpret_cast<float4*>(p) = make_float4(o[0], o[1], o[2], o[3]);
}
__device__ __forceinline__ void store4(double* p, const double* o) {
  *reinterpret_cast<double2*>(p) = make_double2(o[0], o[1]);
  *reinterpret_cast<double2*>(p + 2) = make_double2(o[2], o[3]);
}

__device__ __forceinline__ void load4(const dsv* p, dsv* o) {
  const float4 a = *reinterpret_cast<const float4*>(p);
  const float4 c = *reinterpret_cast<const float4*>(p + 2);
  o[0] = dsv(a.x, a.y); o[1] = dsv(a.z, a.w); o[2] = dsv(c.x, c.y); o[3] = dsv(c.z, c.w);
}
__device__ __forceinline__ void store4(dsv* p, const dsv* o) {
  *reinterpret_cast<float4*>(p) = make_float4(o[0].h, o[0].l, o[1].h, o[1].l);
  *reinterpret_cast<float4*>(p + 2) = make_float4(o[2].h, o[2].l, o[3].h, o[3].l);
}

__device__ __forceinline__ int64_t bidx(int r, int c, int w, int64_t ld) {
  return (int64_t)r * ld + (c - r + w);
}

template <typename T, int NB, bool SMEMP>
__global__ void __launch_bounds__(kThreads, sizeof(T) == 4 ? 2 : 1)
k_band_potrf(T* __restrict__ base, const BandDesc* __restrict__ descs, int phmax,
             DevStatus* st, int32_t* __restrict__ weak, float weak_tol) {
  const BandDesc d = descs[blockIdx.x];
  const int n = d.n, w = d.w;
  const int64_t ld = d.ld;
  T* L = base + d.off;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* Dk = reinterpret_cast<T*>(smem_raw);   // [NB][NB+1]
  T* Ps = Dk + NB * (NB + 1);               // [NB][phmax] (SMEMP only)
  const int tid = threadIdx.x, nt = blockDim.x;
  constexpr int DS = NB + 1;

  for (int kb = 0; kb < n; kb += NB) {
    const int b = min(NB, n - kb);
    const int h = min(w, n - kb - b);
    // 1. diagonal block
    for (int idx = tid; idx < NB * NB; idx += nt) {
      const int r = idx / NB, c = idx % NB;
      T v = T(0);
      if (r < b && c < b && r >= c && r - c <= w) v = L[bidx(kb + r, kb + c, w, ld)];
      Dk[r * DS + c] = v;
    }
    __syncthreads();
    // 2. unblocked Cholesky of the diagonal block by warp 0
    if (tid < 32) {
      const int lane = tid;
      for (int t = 0; t < b; ++t) {
        if (lane == t) {
          T dv = Dk[t * DS + t];
          if (weak) {
            if (!(dv > T(weak_tol))) weak[d.id] = 1;
            if (!finite_pos(dv)) dv = T(1);
          } else if (!finite_pos(dv)) {
            record_error(st, isfinite(dv) ? GENEO_ERR_NOT_SPD : GENEO_ERR_NONFINITE, d.id, (int64_t)kb + t);
            dv = T(1);
          }
          Dk[t * DS + t] = sqrt(dv);
        }
        __syncwarp();
        const T piv = Dk[t * DS + t];
        if (lane > t && lane < b) Dk[lane * DS + t] /= piv;
        __syncwarp();
        if (lane > t && lane < b) {
          const T lrt = Dk[lane * DS + t];
          for (int u = t + 1; u <= lane; ++u) Dk[lane * DS + u] -= lrt * Dk[u * DS + t];
        }
        __syncwarp();
      }
    }
    __syncthreads();
    // 3. store the factored diagonal block
    for (int idx = tid; idx < NB * NB; idx += nt) {
      const int r = idx / NB, c = idx % NB;
      if (r < b && c < b && r >= c && r - c <= w) L[bidx(kb + r, kb + c, w, ld)] = Dk[r * DS + c];
    }
    // 4. panel: rows kb+b+i solve x L_kk^T = a
    for (int i = tid; i < h; i += nt) {
      const int rr = kb + b + i;
      T x[NB];
#pragma unroll
      for (int t = 0; t < NB; ++t) {
        T v = T(0);
        if (t < b && rr - (kb + t) <= w) v = L[bidx(rr, kb + t, w, ld)];
        x[t] = v;
      }
#pragma unroll
      for (int t = 0; t < NB; ++t) {
        if (t < b) {
          T v = x[t];
#pragma unroll
          for (int u = 0; u < t; ++u) v -= x[u] * Dk[t * DS + u];
          x[t] = v / Dk[t * DS + t];
        }
      }
#pragma unroll
      for (int t = 0; t < NB; ++t) {
        if (t < b) {
          const bool inb = rr - (kb + t) <= w;
          if (inb) L[bidx(rr, kb + t, w, ld)] = x[t];
          if (SMEMP) Ps[t * phmax + i] = inb ? x[t] : T(0);
        }
      }
    }
    if (SMEMP) {
      const int h4 = (h + 3) & ~3;
      for (int idx = tid; idx < b * (h4 - h); idx += nt) {
        const int t = idx / (h4 - h), i = h + idx % (h4 - h);
        Ps[t * phmax + i] = T(0);
      }
    }
    __syncthreads();
    // 5. trailing update of the h x h window, 4x4 register tiles
    //    (consecutive threads take consecutive column tiles of one row tile)
    const int T4 = (h + 3) >> 2;
    for (int idx = tid; idx < T4 * T4; idx += nt) {
      const int ti = idx / T4, tj = idx % T4;
      if (tj > ti) continue;
      T acc[4][4];
#pragma unroll
      for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int p = 0; p < 4; ++p) acc[q][p] = T(0);
      for (int t = 0; t < b; ++t) {
        T pr[4], pc[4];
        if (SMEMP) {
          // the panel rows beyond h are zero in shared memory (phmax >= h
          // rounded up to 4), so whole 4-vectors can be read: pr is the same
          // address for the warp (broadcast), pc one 16-byte vector per thread
          const T* prow = Ps + (size_t)t * phmax;
#pragma unroll
          for (int q = 0; q < 4; ++q) pr[q] = prow[4 * ti + q];
          load4(prow + 4 * tj, pc);
        } else {
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const int i = 4 * ti + q, j = 4 * tj + q;
            pr[q] = (i < h && b + i - t <= w) ? L[bidx(kb + b + i, kb + t, w, ld)] : T(0);
            pc[q] = (j < h && b + j - t <= w) ? L[bidx(kb + b + j, kb + t, w, ld)] : T(0);
          }
        }
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
          for (int p = 0; p < 4; ++p) acc[q][p] += pr[q] * pc[p];
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int i = 4 * ti + q;
        if (i >= h) continue;
#pragma unroll
        for (int p = 0; p < 4; ++p) {
          const int j = 4 * tj + p;
          if (j < h && i >= j) L[bidx(kb + b + i, kb + b + j, w, ld)] -= acc[q][p];
        }
      }
    }
    __syncthreads();
  }
}

// Right-looking factorisation of FP64 bands over many SMs: the coarse matrix
// A_H, and batches of fewer subdomain bands than the GPU has SMs.  GB300 issues
// FP64 at 2 fused multiply-adds per clock per SM, so one thread block per
// matrix (k_band_potrf) leaves a batch of 27 bands of order 9261 and half width
// 463 to 27 SMs: 202 ms, against 33 ms of FP64 work for all 152.  Per panel of
// 32 columns, every matrix at once (grid y): the diagonal block
// (k_band_panel_diag), the panel rows below it, one row per thread
// (k_band_panel_rows), and the rank-32 update of the trailing window in 32 x 32
// tiles (k_band_trail).  Three launches per panel; the stream orders them.
constexpr int kPN = 32;   // panel width

// Four warps, lane r holds row r of the columns c with c % 4 = warp: the warp of
// column t takes pivot and column, the block passes the column on through
// shared memory, and every warp updates its own columns.  The four warps run on
// the SM's four FP64 units.
template <typename T>
__global__ void __launch_bounds__(128)
k_band_panel_diag(T* __restrict__ base, const BandDesc* __restrict__ descs, int kb, DevStatus* st) {
  const BandDesc d = descs[blockIdx.x];
  const int n = d.n, w = d.w;
  if (kb >= n) return;
  const int64_t ld = d.ld;
  T* L = base + d.off;
  __shared__ T col[2][kPN];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int b = min(kPN, n - kb);
  T a[kPN / 4];
#pragma unroll
  for (int i = 0; i < kPN / 4; ++i) {
    const int c = 4 * i + wid;
    a[i] = (lane < b && c <= lane && lane - c <= w) ? L[bidx(kb + lane, kb + c, w, ld)] : T(0);
  }
#pragma unroll
  for (int t = 0; t < kPN; ++t) {
    if (t < b) {   // the same for the whole block
      if (wid == (t & 3)) {
        T p = __shfl_sync(0xffffffffu, a[t >> 2], t);
        if (!finite_pos(p)) {
          if (lane == 0)
            record_error(st, isfinite(p) ? GENEO_ERR_NOT_SPD : GENEO_ERR_NONFINITE, d.id, (int64_t)kb + t);
          p = T(1);
        }
        // one reciprocal square root instead of a square root and a division:
        // both are long dependent chains on the FP64 pipe (66 -> 41 us
        // a panel of 27 bands of half width 463, 46 -> 20 us of narrower ones)
        const T r = rsqrt(p), d = pivot_root(p, r);
        a[t >> 2] = lane == t ? d : lane > t ? pivot_quotient(a[t >> 2], d, r) : T(0);
        col[t & 1][lane] = a[t >> 2];
      }
      __syncthreads();
      const T lrt = col[t & 1][lane];
#pragma unroll
      for (int i = 0; i < kPN / 4; ++i) {
        const int c = 4 * i + wid;
        if (4 * i + 3 > t && c > t && lane >= c) a[i] -= lrt * col[t & 1][c];
      }
    }
  }
#pragma unroll
  for (int i = 0; i < kPN / 4; ++i) {
    const int c = 4 * i + wid;
    if (lane < b && c <= lane && lane - c <= w) L[bidx(kb + lane, kb + c, w, ld)] = a[i];
  }
}

// Rows kb + b + 32 blockIdx.x + lane of the panel of matrix blockIdx.y:
// x L_kk^T = a (the diagonal block already factored), multiplying by the
// pivots' reciprocals.
template <typename T>
__global__ void __launch_bounds__(32)
k_band_panel_rows(T* __restrict__ base, const BandDesc* __restrict__ descs, int kb) {
  const BandDesc d = descs[blockIdx.y];
  const int n = d.n, w = d.w;
  const int b = min(kPN, n - kb);
  const int h = min(w, n - kb - b);
  if (kb >= n || 32 * (int)blockIdx.x >= h) return;
  const int64_t ld = d.ld;
  T* L = base + d.off;
  __shared__ T Dk[kPN * (kPN + 1)];
  __shared__ T rp[kPN];
  constexpr int DS = kPN + 1;
  const int lane = threadIdx.x;
  for (int idx = lane; idx < kPN * kPN; idx += 32) {
    const int r = idx / kPN, c = idx % kPN;
    Dk[r * DS + c] = (r < b && c < b && r >= c && r - c <= w) ? L[bidx(kb + r, kb + c, w, ld)] : T(0);
  }
  __syncwarp();
  rp[lane] = lane < b ? T(1) / Dk[lane * DS + lane] : T(0);
  __syncwarp();
  const int i = 32 * blockIdx.x + lane;
  if (i >= h) return;
  const int rr = kb + b + i;
  T x[kPN];
#pragma unroll
  for (int t = 0; t < kPN; ++t) x[t] = (t < b && rr - (kb + t) <= w) ? L[bidx(rr, kb + t, w, ld)] : T(0);
#pragma unroll
  for (int t = 0; t < kPN; ++t) {
    if (t < b) {
      T v = x[t];
#pragma unroll
      for (int u = 0; u < t; ++u) v -= x[u] * Dk[t * DS + u];
      x[t] = v * rp[t];
    }
  }
#pragma unroll
  for (int t = 0; t < kPN; ++t)
    if (t < b && rr - (kb + t) <= w) L[bidx(rr, kb + t, w, ld)] = x[t];
}

// Trailing update of panel kb of matrix blockIdx.y: C(i, i') -= sum_t P(i, t)
// P(i', t) over the h x h window below the panel, tile (ti, tj) of 32 x 32
// (ti >= tj), one 4 x 4 register tile per thread, panel rows staged in shared
// memory.  Tiles of 32 rather than 64 keep the share of the work outside the
// window's lower triangle small (14 % at h = 463, not 37 %) and give a batch
// enough blocks to even out.
constexpr int kTT = 32;
template <typename T>
__global__ void __launch_bounds__(64)
k_band_trail(T* __restrict__ base, const BandDesc* __restrict__ descs, int kb) {
  const BandDesc d = descs[blockIdx.y];
  const int n = d.n, w = d.w;
  const int b = min(kPN, n - kb);
  const int h = min(w, n - kb - b);
  // block index -> (ti, tj) in the lower triangle, row-major
  const int t = blockIdx.x;
  int ti = (int)((sqrtf(8.f * t + 1.f) - 1.f) * 0.5f);
  while ((ti + 1) * (ti + 2) / 2 <= t) ++ti;
  while (ti * (ti + 1) / 2 > t) --ti;
  const int tj = t - ti * (ti + 1) / 2;
  const int i0 = kTT * ti, j0 = kTT * tj;
  if (kb >= n || i0 >= h) return;
  const int64_t ld = d.ld;
  T* L = base + d.off;
  // row-major in t: a thread's four rows (columns) are one 32-byte read
  __shared__ __align__(16) T Pi[kPN][kTT + 2], Pj[kPN][kTT + 2];
  for (int idx = threadIdx.x; idx < kPN * kTT; idx += 64) {
    const int tt = idx % kPN, r = idx / kPN;   // consecutive threads along a band row
    const int ii = i0 + r, jj = j0 + r;
    Pi[tt][r] = (tt < b && ii < h && b + ii - tt <= w) ? L[bidx(kb + b + ii, kb + tt, w, ld)] : T(0);
    Pj[tt][r] = (tt < b && jj < h && b + jj - tt <= w) ? L[bidx(kb + b + jj, kb + tt, w, ld)] : T(0);
  }
  __syncthreads();
  const int tr = threadIdx.x >> 3, tc = threadIdx.x & 7;
  if (ti == tj && 4 * tc > 4 * tr + 3) return;   // above the diagonal
  T acc[4][4];
#pragma unroll
  for (int q = 0; q < 4; ++q)
#pragma unroll
    for (int p = 0; p < 4; ++p) acc[q][p] = T(0);
#pragma unroll 4
  for (int tt = 0; tt < kPN; ++tt) {
    T pr[4], pc[4];
    load4(&Pi[tt][4 * tr], pr);
    load4(&Pj[tt][4 * tc], pc);
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
      for (int p = 0; p < 4; ++p) acc[q][p] += pr[q] * pc[p];
  }
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int i = i0 + 4 * tr + q;
    if (i >= h) continue;
#pragma unroll
    for (int p = 0; p < 4; ++p) {
      const int c = j0 + 4 * tc + p;
      if (c < h && i >= c) L[bidx(kb + b + i, kb + b + c, w, ld)] -= acc[q][p];
    }
  }
}

// Equilibration of a band before its FP32 factorisation: s_r = a_rr^{-1/2}
// (1 where a_rr is not positive: the factorisation reports it), then every
// entry a_rc *= s_r s_c, so the factor is that of S A S (unit diagonal) and
// A^{-1} = S (S A S)^{-1} S.  Grid: (row blocks, matrices).
template <typename T>
__global__ void k_band_equil_s(T* __restrict__ base, const BandDesc* __restrict__ descs) {
  const BandDesc d = descs[blockIdx.y];
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (d.scl < 0 || r >= d.n) return;
  const T a = base[d.off + (int64_t)r * d.ld + d.w];
  base[d.scl + r] = a > T(0) ? T(1) / sqrt(a) : T(1);
}

template <typename T>
__global__ void __launch_bounds__(256)
k_band_equil_a(T* __restrict__ base, const BandDesc* __restrict__ descs) {
  const BandDesc d = descs[blockIdx.y];
  if (d.scl < 0) return;
  const T* S = base + d.scl;
  for (int i = 0; i < 16; ++i) {
    const int r = blockIdx.x * 16 + i;
    if (r >= d.n) return;
    const T sr = S[r];
    T* row = base + d.off + (int64_t)r * d.ld;
    for (int off = max(0, d.w - r) + (int)threadIdx.x; off <= d.w; off += blockDim.x)
      row[off] *= sr * S[r - d.w + off];
  }
}

// x = s o x on columns [0, k) of the solve vectors (before and after the
// solves that do not apply the scaling themselves)
template <typename T>
__global__ void k_band_scale_x(const T* __restrict__ base, const BandDesc* __restrict__ descs,
                               double* __restrict__ xbase, const int64_t* __restrict__ xoff, int col0,
                               int kcap, const int32_t* __restrict__ nrhs_dev, const int32_t* __restrict__ skip) {
  const BandDesc d = descs[blockIdx.y];
  // vectors, counts and skip flags are indexed by the subdomain id (a
  // batch may hold a subset of the subdomains)
  const int mi = d.id >= 0 ? d.id : (int)blockIdx.y;
  if (skip && skip[mi]) return;
  if (d.scl < 0) return;
  int k = kcap;
  if (nrhs_dev) k = min(k, nrhs_dev[mi] - col0);
  const T* S = base + d.scl;
  double* X = xbase + xoff[mi] + (int64_t)col0 * d.n;
  for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < (int64_t)k * d.n;
       idx += (int64_t)gridDim.x * blockDim.x)
    X[idx] *= (double)S[idx % d.n];
}

// ---------------------------------------------------------------------------
// Left-looking FP32 band Cholesky on the tensor cores.
//
// Panel j (columns j .. j+b-1, b <= 32) of the rows r in [j, j + R),
// R = min(n, j + b + w) - j, is first brought up to date with all finished
// columns k in [j - w, j):
//   U(r, c) = A(r, c) - sum_k L(r, k) L(c, k),
// an (R x w) x (w x 32) product whose operands are whole band rows: the
// panel's own rows (staged once per panel) and the rows r (streamed in
// chunks of 16 by bulk copies, two buffers).  For each chunk's 16 x 32 tile
// every warp takes an eighth of the k range and accumulates it with m16n8k8
// TF32 MMAs in three passes (hi*hi + hi*lo + lo*hi with x = hi + lo, both
// TF32, split_tf32_rn), which keeps close to FP32 accuracy; the eight partial tiles go
// to one of two shared buffers and are summed in a fixed order while the next
// chunk multiplies (one block barrier per chunk).  Then the 32 x 32 diagonal
// block is factored by one warp in registers and the rows below by
// substitution, one row per thread.  Only the panel columns are written; the
// trailing window is never rewritten.
// ---------------------------------------------------------------------------
// x = hi + lo, both TF32 (split_tf32_rn), as the MMA's operand bits
__device__ __forceinline__ void split_tf32(float x, uint32_t& hi, uint32_t& lo) {
  float h, l;
  split_tf32_rn(x, h, l);
  hi = __float_as_uint(h);
  lo = __float_as_uint(l);
}
__device__ __forceinline__ void mma_tf32(float* c, const uint32_t* a, const uint32_t* b) {
  asm volatile(
      "mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

constexpr int kPB = 32;   // panel width of the tensor-core factorisation
constexpr int kMC = 16;   // rows per streamed chunk (one 16-row MMA tile)
constexpr int kUS = kPB + 1;  // row stride of the panel block in shared memory

// Shared memory of the tensor-core factorisation for half-bandwidth w.
inline size_t potrf_tc_smem(int w) {
  const size_t ld = (size_t)band_ld(w);
  return 128 + sizeof(float) * ((kPB + 2 * kMC) * ld + (size_t)(w + kPB) * kUS + kPB + 2 * 8 * 16 * 32);
}

__global__ void __launch_bounds__(kThreads, 1)
k_band_potrf_tc(float* __restrict__ base, const BandDesc* __restrict__ descs, DevStatus* st,
                int32_t* __restrict__ weak, float weak_tol) {
  const BandDesc d = descs[blockIdx.x];
  const int n = d.n, w = d.w;
  const int ld = d.ld;
  float* L = base + d.off;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem_raw);                  // 0: panel rows, 1-2: chunks
  float* Cs = reinterpret_cast<float*>(smem_raw + 128);                    // kPB x ld
  float* Rs = Cs + (size_t)kPB * ld;                                       // 2 x kMC x ld
  float* Us = Rs + (size_t)2 * kMC * ld;                                   // (w + kPB) x kUS panel block
  float* Dinv = Us + (size_t)(w + kPB) * kUS;                              // kPB reciprocal pivots
  float* Red = Dinv + kPB;                                                 // 2 x 8 warps x 16 x 32 partials
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int g = lane >> 2, tg = lane & 3;
  if (tid == 0) {
    for (int i = 0; i < 3; ++i) mbar_init(&bars[i], 1);
    fence_barrier_init();
  }
  __syncthreads();
  uint32_t ph[3] = {0, 0, 0};      // next phase to wait for, per barrier
  int issued[3] = {0, 0, 0};       // thread 0: copies issued per barrier
  bool ok = true;                  // warp 0's view (thread 0 issues the copies)
  auto load_rows = [&](int bar, float* dst, int r0, int rows) {
    const uint32_t bytes = (uint32_t)((size_t)rows * ld * sizeof(float));
    mbar_arrive_expect_tx(&bars[bar], bytes);
    bulk_load(dst, L + (int64_t)r0 * ld, bytes, &bars[bar]);
    ++issued[bar];
  };
  // warp 0 waits; the block is released by the barrier that follows
  auto wait_bar = [&](int bar, int64_t where) {
    if (wid == 0 && ok) {
      ok = mbar_wait_bounded(&bars[bar], ph[bar] & 1, st, d.id, where);
    }
    ++ph[bar];
    __syncthreads();
  };

  for (int j = 0; j < n; j += kPB) {
    const int b = min(kPB, n - j);
    const int R = min(n, j + b + w) - j;
    const int kbeg = max(0, j - w);
    const int nch = (R + kMC - 1) / kMC;
    // the previous panel's columns were written by ordinary stores: order
    // them before the bulk copies that read them
    if (tid == 0 && ok) {
      fence_proxy_async_global();
      fence_proxy_async();
      load_rows(0, Cs, j, b);
      load_rows(1, Rs, j, min(kMC, R));
    }
    wait_bar(0, j);
    // One block barrier per chunk: the partial tiles of chunk ch go to
    // Red[ch & 1] and are summed in the next iteration (or after the loop),
    // with the A values each thread needs captured in registers before the
    // chunk's rows are overwritten; the next chunk's copy is issued after the
    // barrier, when no warp still reads the buffer it refills.
    const int nt2 = wid & 3, qh = wid >> 2;   // this thread's two reduce outputs
    float pa[2] = {0.f, 0.f};                 // A values of the pending chunk
    int prow = -1;                            // first row of the pending chunk (-1: none)
    auto reduce_pending = [&]() {
      if (prow < 0) return;
      const float* Rp = Red + (size_t)(((prow - j) / kMC) & 1) * (8 * 16 * 32);
#pragma unroll
      for (int h2 = 0; h2 < 2; ++h2) {
        const int q = 2 * qh + h2;
        float sum = 0.f;
#pragma unroll
        for (int kk = 0; kk < 8; ++kk) sum += Rp[((size_t)kk * 16 + nt2 * 4 + q) * 32 + lane];
        const int r = prow + g + ((q & 2) ? 8 : 0);  // c0,c1: row g; c2,c3: row g+8
        const int cl = 8 * nt2 + 2 * tg + (q & 1), c = j + cl;
        if (r < j + R) {
          float u = 0.f;
          if (cl < b && c <= r && r - c <= w) u = pa[h2] - sum;
          Us[(size_t)(r - j) * kUS + cl] = u;
        }
      }
    };
    for (int ch = 0; ch < nch; ++ch) {
      const int buf = ch & 1;
      const int r0 = j + ch * kMC;
      wait_bar(1 + buf, (int64_t)j * 1024 + ch);
      if (tid == 0 && ok && ch + 1 < nch)
        load_rows(1 + (buf ^ 1), Rs + (size_t)(buf ^ 1) * kMC * ld, r0 + kMC, min(kMC, R - (ch + 1) * kMC));
      const float* Rb = Rs + (size_t)buf * kMC * ld;
      // warp kq: rows r0 .. r0 + 15, all 32 panel columns, over the kq-th
      // eighth of the k-steps of the tile's range
      const int kq = wid;
      const int ra = r0 + g, rb = r0 + g + 8;
      const bool va = ra < j + R, vb = rb < j + R;
      // element offsets of L(r, 0) in the staged rows (may be negative; an
      // index is formed only for k in the row's band)
      const int ia = g * ld + (w - ra);
      const int ib = (g + 8) * ld + (w - rb);
      const int klo = max(kbeg, r0 - w);          // no row of the tile reaches below klo
      const int kst = kbeg + ((klo - kbeg) & ~7);
      const int nsteps = (j - kst + 7) >> 3;
      const int s0 = kst + 8 * ((nsteps * kq) >> 3), s1 = kst + 8 * ((nsteps * (kq + 1)) >> 3);
      // every row and column is in band from kfull on
      const int kfull = max(r0 + 15, j + b - 1) - w;
      float acc[4][3][4];
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 3; ++v)
#pragma unroll
          for (int q = 0; q < 4; ++q) acc[u][v][q] = 0.f;
      for (int k0 = s0; k0 < s1; k0 += 8) {
        const bool masked = k0 < kfull || k0 + 8 > j;
        const int k1 = k0 + tg, k2 = k0 + tg + 4;
        float x[4];
        if (!masked) {
          x[0] = va ? Rb[ia + k1] : 0.f;
          x[1] = vb ? Rb[ib + k1] : 0.f;
          x[2] = va ? Rb[ia + k2] : 0.f;
          x[3] = vb ? Rb[ib + k2] : 0.f;
        } else {
          x[0] = (va && k1 < j && k1 >= ra - w && k1 >= 0) ? Rb[ia + k1] : 0.f;
          x[1] = (vb && k1 < j && k1 >= rb - w && k1 >= 0) ? Rb[ib + k1] : 0.f;
          x[2] = (va && k2 < j && k2 >= ra - w && k2 >= 0) ? Rb[ia + k2] : 0.f;
          x[3] = (vb && k2 < j && k2 >= rb - w && k2 >= 0) ? Rb[ib + k2] : 0.f;
        }
        uint32_t ah[4], al[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) split_tf32(x[q], ah[q], al[q]);
#pragma unroll
        for (int nt = 0; nt < 4; ++nt) {
          const int cn = 8 * nt + g, cc = j + cn;
          const int ic = cn * ld + (w - cc);
          float y0, y1;
          if (!masked) {
            y0 = cn < b ? Cs[ic + k1] : 0.f;
            y1 = cn < b ? Cs[ic + k2] : 0.f;
          } else {
            y0 = (cn < b && k1 < j && k1 >= cc - w && k1 >= 0) ? Cs[ic + k1] : 0.f;
            y1 = (cn < b && k2 < j && k2 >= cc - w && k2 >= 0) ? Cs[ic + k2] : 0.f;
          }
          uint32_t bh[2], bl[2];
          split_tf32(y0, bh[0], bl[0]);
          split_tf32(y1, bh[1], bl[1]);
          mma_tf32(acc[nt][0], al, bh);
          mma_tf32(acc[nt][1], ah, bl);
          mma_tf32(acc[nt][2], ah, bh);
        }
      }
      // partial sums of this eighth (small terms first), lane-contiguous
      float* Rw = Red + (size_t)buf * (8 * 16 * 32);
#pragma unroll
      for (int nt = 0; nt < 4; ++nt)
#pragma unroll
        for (int q = 0; q < 4; ++q)
          Rw[((size_t)kq * 16 + nt * 4 + q) * 32 + lane] = (acc[nt][0][q] + acc[nt][1][q]) + acc[nt][2][q];
      // warp w: n-tile w & 3, outputs q of half w >> 2; U = A - sum into the
      // panel block (zero outside the lower band), for the previous chunk
      reduce_pending();
      // capture this chunk's A values for its reduction in the next iteration
#pragma unroll
      for (int h2 = 0; h2 < 2; ++h2) {
        const int q = 2 * qh + h2;
        const int r = r0 + g + ((q & 2) ? 8 : 0);
        const int cl = 8 * nt2 + 2 * tg + (q & 1), c = j + cl;
        pa[h2] = (r < j + R && cl < b && c <= r && r - c <= w) ? Rb[(size_t)(r - r0) * ld + (c - r + w)] : 0.f;
      }
      prow = r0;
    }
    __syncthreads();
    reduce_pending();
    __syncthreads();
    // ---- factor the panel's diagonal block in warp 0: lane r holds row r in
    // registers; step t takes pivot t from lane t (a pivot that is not
    // positive is reported and replaced by 1), scales column t and updates
    // the trailing part with shuffled column-t values (no block barriers).
    if (wid == 0) {
      float a[kPB];
#pragma unroll
      for (int u = 0; u < kPB; ++u) a[u] = (lane < b && u <= lane) ? Us[lane * kUS + u] : 0.f;
#pragma unroll
      for (int t = 0; t < kPB; ++t) {
        if (t < b) {  // uniform over the warp
          float p = __shfl_sync(0xffffffffu, a[t], t);
          if (weak) {
            if (lane == 0 && !(p > weak_tol)) weak[d.id] = 1;
            if (!finite_pos(p)) p = 1.f;
          } else if (!finite_pos(p)) {
            if (lane == 0) record_error(st, isfinite(p) ? GENEO_ERR_NOT_SPD : GENEO_ERR_NONFINITE, d.id, (int64_t)j + t);
            p = 1.f;
          }
          const float inv = rsqrtf(p);
          if (lane == t) {
            a[t] = p * inv;  // sqrt(pivot)
            Dinv[t] = inv;
          } else if (lane > t) {
            a[t] *= inv;
          }
#pragma unroll
          for (int u = t + 1; u < kPB; ++u) {
            const float lut = __shfl_sync(0xffffffffu, a[t], u);
            if (lane >= u) a[u] -= a[t] * lut;
          }
        }
      }
      if (lane < b) {
#pragma unroll
        for (int u = 0; u < kPB; ++u)
          if (u <= lane) Us[lane * kUS + u] = a[u];
      } else {
        Dinv[lane] = 0.f;
      }
    }
    __syncthreads();
    // rows below: x L_jj^T = u, one row per thread (stride kUS: no bank conflicts)
    for (int i = b + tid; i < R; i += kThreads) {
      float* ur = Us + (size_t)i * kUS;
      float x[kPB];
#pragma unroll
      for (int t = 0; t < kPB; ++t) x[t] = ur[t];
#pragma unroll
      for (int t = 0; t < kPB; ++t) {
        if (t < b) {
          float v = x[t];
#pragma unroll
          for (int u = 0; u < t; ++u) v -= x[u] * Us[t * kUS + u];
          x[t] = v * Dinv[t];
        }
      }
#pragma unroll
      for (int t = 0; t < kPB; ++t) ur[t] = x[t];
    }
    __syncthreads();
    // the panel's columns back to the band, one warp per row (coalesced)
    for (int i = wid; i < R; i += kThreads / 32) {
      const int r = j + i, c = j + lane;
      if (lane < b && c <= r && r - c <= w) L[(int64_t)r * ld + (c - r + w)] = Us[(size_t)i * kUS + lane];
    }
    __syncthreads();
  }
  // after a timed-out wait, let the copies still in flight land (bounded)
  if (tid == 0 && !ok)
    for (int bar = 0; bar < 3; ++bar)
      for (uint32_t p = ph[bar]; p < (uint32_t)issued[bar]; ++p)
        mbar_wait_bounded(&bars[bar], p & 1, st, d.id, -1);
}

// rows per streamed block: 16, or 4 for bands too wide for 16-row stages
// pipeline depth of the multi-right-hand-side solve: two stages leave room
// for the right-hand-side ring and two blocks per SM
template <typename T> struct Stages { static constexpr int v = 2; };

// Block v of the visit order 0..nb-1 (forward), nb-1..0 (backward).
__device__ __forceinline__ int visit_block(int v, int nb) { return v < nb ? v : 2 * nb - 1 - v; }

template <typename T, typename A, int kSNB, int kMaxRhsPerWarp, int kStages>
__global__ void __launch_bounds__(kThreads, kMaxRhsPerWarp == 1 ? (sizeof(T) == 4 ? 4 : 2) : 2)
k_band_solve(const T* __restrict__ base, const BandDesc* __restrict__ descs,
             double* __restrict__ xbase, const int64_t* __restrict__ xoff, int col0, int kcap,
             const int32_t* __restrict__ nrhs_dev, const int32_t* __restrict__ skip, int ring,
             DevStatus* st) {
  const BandDesc d = descs[blockIdx.x];
  // vectors, counts and skip flags are indexed by the subdomain id (a
  // batch may hold a subset of the subdomains)
  const int mi = d.id >= 0 ? d.id : (int)blockIdx.x;
  if (skip && skip[mi]) return;
  // column split: block y of gridDim.y takes its share of the kcap columns
  {
    const int cpp = (kcap + (int)gridDim.y - 1) / (int)gridDim.y;
    col0 += (int)blockIdx.y * cpp;
    kcap = min(cpp, kcap - (int)blockIdx.y * cpp);
  }
  int k = kcap;
  if (nrhs_dev) k = min(k, nrhs_dev[mi] - col0);
  if (k <= 0) return;
  const int n = d.n, w = d.w;
  if (n <= 0) return;
  const int ld = d.ld;
  const T* L = base + d.off;
  double* X = xbase + xoff[mi] + (int64_t)col0 * n;
  const int rmask = ring - 1;  // ring is a power of two >= w + 2 SNB

  extern __shared__ __align__(128) unsigned char smem_raw[];
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem_raw);                      // kStages
  T* stage = reinterpret_cast<T*>(smem_raw + 128);                             // kStages * SNB * ld
  A* win = reinterpret_cast<A*>(stage + (size_t)kStages * kSNB * ld);         // k columns of ring rows
  A* blk = win + (size_t)ring * k;                                             // SNB * k
  A* red = blk + (size_t)kSNB * k;                                             // 4 * kThreads
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, nw = kThreads >> 5;
  const int nb = (n + kSNB - 1) / kSNB;
  const int nvis = 2 * nb;

  for (int idx = tid; idx < ring * k; idx += kThreads) win[idx] = A();
  if (tid == 0) {
    for (int s = 0; s < kStages; ++s) mbar_init(&bars[s], 1);
    fence_barrier_init();
  }
  __syncthreads();
  auto issue = [&](int v) {
    const int kb = visit_block(v, nb) * kSNB;
    const int b = min(kSNB, n - kb);
    const int s = v % kStages;
    const uint32_t bytes = (uint32_t)((size_t)b * ld * sizeof(T));
    fence_proxy_async();
    mbar_arrive_expect_tx(&bars[s], bytes);
    bulk_load(stage + (size_t)s * kSNB * ld, L + (int64_t)kb * ld, bytes, &bars[s]);
  };
  int issued = 0;  // copies issued by thread 0
  if (tid == 0)
    for (; issued < min(kStages - 1, nvis); ++issued) issue(issued);
  bool ok = true;
  int waited = 0;  // stages this thread has waited for
  int lo = n;  // lowest row held in the ring during the backward sweep

  for (int v = 0; v < nvis; ++v) {
    const int s = v % kStages;
    const uint32_t parity = (uint32_t)((v / kStages) & 1);
    if (tid == 0 && ok && issued < nvis) issue(issued++);
    const int kb = visit_block(v, nb) * kSNB;
    const int b = min(kSNB, n - kb);
    if (v < nb) {
      // ---------------- forward, rows kb..kb+b-1 (left-looking)
      // right-hand sides of this block, fetched before the wait (lane i of
      // the warp owning right-hand side c holds b[kb + i][c])
      A xb[kMaxRhsPerWarp];
#pragma unroll
      for (int u = 0; u < kMaxRhsPerWarp; ++u) {
        const int c = wid + u * nw;
        xb[u] = (c < k && lane < b) ? to_arith<A>(X[(int64_t)c * n + kb + lane]) : A();
      }
      if (ok) {
        ok = mbar_wait_bounded(&bars[s], parity, st, d.id, v);
        waited += ok ? 1 : 0;
      }
      const T* S = stage + (size_t)s * kSNB * ld;
      // dot products with the solved rows [kb + i - w, kb) held in the ring:
      // a (b x w) x (w x k) product; a thread owns one row and CT right-hand
      // sides over one segment of the band, partials summed by the warp that
      // owns the right-hand side
      const int ct = k == 1 ? 1 : 4;
      const int ntc = (k + ct - 1) / ct;
      const int ntiles = b * ntc;
      const int nseg = max(1, min(32, kThreads / ntiles));
      for (int task = tid; task < ntiles * nseg; task += kThreads) {
        const int tile = task % ntiles, seg = task / ntiles;
        const int i = tile % b, c0 = (tile / b) * ct;
        const int r = kb + i;
        const int olo = max(0, w - r), ohi = w - i;  // columns r - w + oo in [0, kb)
        const int len = max(0, ohi - olo);
        const int s0 = olo + (int)((int64_t)len * seg / nseg);
        const int s1 = olo + (int)((int64_t)len * (seg + 1) / nseg);
        const T* srow = S + (size_t)i * ld;
        A a0 = A(), a1 = A(), a2 = A(), a3 = A();
        if (ct == 1) {
          const A* wc = win + (size_t)c0 * ring;
          int oo = s0;
          for (; oo + 1 < s1; oo += 2) {
            a0 += to_arith<A>(srow[oo]) * wc[(r - w + oo) & rmask];
            a1 += to_arith<A>(srow[oo + 1]) * wc[(r - w + oo + 1) & rmask];
          }
          if (oo < s1) a0 += to_arith<A>(srow[oo]) * wc[(r - w + oo) & rmask];
          a0 += a1;
          a1 = A();
        } else {
          const A* w0 = win + (size_t)c0 * ring;
          const bool h1 = c0 + 1 < k, h2 = c0 + 2 < k, h3 = c0 + 3 < k;
          const A* w1 = h1 ? w0 + ring : w0;
          const A* w2 = h2 ? w0 + 2 * ring : w0;
          const A* w3 = h3 ? w0 + 3 * ring : w0;
          for (int oo = s0; oo < s1; ++oo) {
            const A sv = to_arith<A>(srow[oo]);
            const int q = (r - w + oo) & rmask;
            a0 += sv * w0[q];
            a1 += sv * w1[q];
            a2 += sv * w2[q];
            a3 += sv * w3[q];
          }
        }
        A* rd = red + (size_t)(seg * ntiles + tile) * 4;
        rd[0] = a0;
        rd[1] = a1;
        rd[2] = a2;
        rd[3] = a3;
      }
      __syncthreads();
      // diagonal block by the warp owning each right-hand side: row of L and
      // the reciprocal pivot in registers, substitution by shuffles
      A lrow[kSNB];
#pragma unroll
      for (int t = 0; t < kSNB; ++t)
        lrow[t] = (lane < b && t < lane && lane - t <= w) ? to_arith<A>(S[lane * ld + (w - lane + t)]) : A();
      const A dinv = lane < b ? recip_arith<A>(S[lane * ld + w]) : A();
#pragma unroll
      for (int u = 0; u < kMaxRhsPerWarp; ++u) {
        const int c = wid + u * nw;
        if (c >= k) break;
        A y = A();
        if (lane < b) {
          const int tile = lane + (c / ct) * b, q = c % ct;
          A acc = A();
          for (int seg = 0; seg < nseg; ++seg) acc += red[(size_t)(seg * ntiles + tile) * 4 + q];
          y = xb[u] - acc;
        }
#pragma unroll
        for (int t = 0; t < kSNB; ++t) {
          if (t < b) {
            if (lane == t) y *= dinv;
            const A yt = shfl(y, t);
            if (lane > t) y -= lrow[t] * yt;
          }
        }
        if (lane < b) {
          win[(size_t)c * ring + ((kb + lane) & rmask)] = y;
          X[(int64_t)c * n + kb + lane] = to_double(y);
        }
      }
      if (v == nb - 1) lo = max(0, kb - w);  // the ring holds rows [lo, n) for the backward sweep
    } else {
      // ---------------- backward, block kb (right-looking on L^T)
      if (ok) {
        ok = mbar_wait_bounded(&bars[s], parity, st, d.id, v);
        waited += ok ? 1 : 0;
      }
      const T* S = stage + (size_t)s * kSNB * ld;
      A lcol[kSNB];
#pragma unroll
      for (int t = 0; t < kSNB; ++t)
        lcol[t] = (t < b && lane < t && t - lane <= w) ? to_arith<A>(S[t * ld + (w - t + lane)]) : A();
      const A dinv = lane < b ? recip_arith<A>(S[lane * ld + w]) : A();
      for (int c = wid; c < k; c += nw) {
        A y = lane < b ? win[(size_t)c * ring + ((kb + lane) & rmask)] : A();
#pragma unroll
        for (int t = kSNB - 1; t >= 0; --t) {
          if (t < b) {
            if (lane == t) y *= dinv;
            const A xt = shfl(y, t);
            if (lane < t) y -= lcol[t] * xt;
          }
        }
        if (lane < b) {
          blk[lane * k + c] = y;
          X[(int64_t)c * n + kb + lane] = to_double(y);
        }
      }
      __syncthreads();
      // rows [lo, kb) of the ring: y -= sum_t L(kb + t, row) x_t; at the same
      // time the rows the next block adds to the ring come from X (forward
      // results, not yet finalised by this sweep)
      const int cnt = kb - lo;
      const int ncg = (k + 3) / 4;
      for (int idx = tid; idx < cnt * ncg; idx += kThreads) {
        const int rr = lo + idx % cnt, c0 = (idx / cnt) * 4;
        A a0 = A(), a1 = A(), a2 = A(), a3 = A();
        const int tmax = min(b - 1, rr - kb + w);
        for (int t = 0; t <= tmax; ++t) {
          const A sv = to_arith<A>(S[t * ld + (rr - kb - t + w)]);
          const A* bt = blk + t * k + c0;
          a0 += sv * bt[0];
          if (c0 + 1 < k) a1 += sv * bt[1];
          if (c0 + 2 < k) a2 += sv * bt[2];
          if (c0 + 3 < k) a3 += sv * bt[3];
        }
        const int q = rr & rmask;
        win[(size_t)c0 * ring + q] -= a0;
        if (c0 + 1 < k) win[(size_t)(c0 + 1) * ring + q] -= a1;
        if (c0 + 2 < k) win[(size_t)(c0 + 2) * ring + q] -= a2;
        if (c0 + 3 < k) win[(size_t)(c0 + 3) * ring + q] -= a3;
      }
      if (kb > 0) {
        const int nlo = max(0, kb - kSNB - w);
        const int ncnt = lo - nlo;
        for (int idx = tid; idx < ncnt * k; idx += kThreads) {
          const int rr = nlo + idx % ncnt, c = idx / ncnt;
          win[(size_t)c * ring + (rr & rmask)] = to_arith<A>(X[(int64_t)c * n + rr]);
        }
        lo = nlo;
      }
    }
    __syncthreads();
  }
  // after a timed-out wait, let the copies still in flight land (bounded)
  if (tid == 0 && !ok)
    for (int v = waited; v < issued; ++v)
      mbar_wait_bounded(&bars[v % kStages], (uint32_t)((v / kStages) & 1), st, d.id, v);
}

constexpr int kNB = 32;
constexpr size_t kSmemCap = 200 * 1024;

inline int next_pow2(int v) {
  int p = 1;
  while (p < v) p <<= 1;
  return p;
}

}  // namespace

template <typename T>
geneo_status_t band_potrf(T* base, const BandDesc* d_desc, int count, int max_w, int max_n, int blk_mask,
                          DevStatus* st, cudaStream_t s, bool equil, int32_t* weak, float weak_tol,
                          const Tc5Plan* tc5) {
  if (count <= 0) return GENEO_OK;
  // FP32: fifth-generation tensor cores (tcgen05, TMA) when the batch fits;
  // the packing into the tiled band applies the equilibration
  if constexpr (sizeof(T) == 4) {
    if (tc5 && tc5->ok) {
      if (equil && max_n > 0) {
        k_band_equil_s<T><<<dim3((max_n + 255) / 256, count), 256, 0, s>>>(base, d_desc); note_launch();
        GENEO_CUDA(cudaGetLastError());
      }
      GENEO_TRY(tc5_factor(*tc5, base, d_desc, st, s, weak, weak_tol * kTf32PivotScale));
      return band_blkinv(base, d_desc, count, max_n, blk_mask, s);
    }
  }
  if (equil && max_n > 0) {
    k_band_equil_s<T><<<dim3((max_n + 255) / 256, count), 256, 0, s>>>(base, d_desc); note_launch();
    k_band_equil_a<T><<<dim3((max_n + 15) / 16, count), 256, 0, s>>>(base, d_desc); note_launch();
    GENEO_CUDA(cudaGetLastError());
  }
  // FP32: left-looking tensor-core kernel when a panel's rows and two chunk
  // buffers fit in shared memory
  if constexpr (sizeof(T) == 4) {
    const size_t tc_smem = potrf_tc_smem(max_w);
    if (tc_smem <= 227 * 1024) {
      GENEO_CUDA(allow_smem(k_band_potrf_tc));
      k_band_potrf_tc<<<count, kThreads, tc_smem, s>>>(base, d_desc, st, weak, weak_tol * kTf32PivotScale);
      note_launch();
      GENEO_CUDA(cudaGetLastError());
      return band_blkinv(base, d_desc, count, max_n, blk_mask, s);
    }
  }
  // FP64 bands too few for one SM each: every panel's work spread over the GPU.
  // Both sides in SM clocks per panel, of 2 multiply-adds: one block per matrix runs
  // the widest alone on its SM; spread, a panel's three launches cost about 75 us
  // (150e3 clocks at 2.0 GHz; measured: 20 to 41 + 24 to 28, and the gaps) whatever
  // the batch
  if constexpr (sizeof(T) == 8) {
    if (!weak && max_n > 256 && max_w >= 96) {
      const double panel = 0.5 * (double)max_w * max_w * kPN;          // multiply-adds of one panel's update
      const double alone = panel / 2.0 * ceil_div(count, sm_count());  // clocks, 2 per clock and SM
      const double spread = 1.2 * panel * count / (2.0 * sm_count()) + 150e3;
      if (spread < alone) {
        for (int kb = 0; kb < max_n; kb += kPN) {
          k_band_panel_diag<T><<<count, 128, 0, s>>>(base, d_desc, kb, st); note_launch();
          const int h = std::min(max_w, max_n - kb - std::min(kPN, max_n - kb));
          if (h > 0) {
            const int nt = (h + kTT - 1) / kTT;
            k_band_panel_rows<T><<<dim3((h + 31) / 32, count), 32, 0, s>>>(base, d_desc, kb); note_launch();
            k_band_trail<T><<<dim3(nt * (nt + 1) / 2, count), 64, 0, s>>>(base, d_desc, kb); note_launch();
          }
        }
        GENEO_CUDA(cudaGetLastError());
        return band_blkinv(base, d_desc, count, max_n, blk_mask, s);
      }
    }
  }
  // the panel starts at a 16-byte boundary (diag block: 32 x 33 values) and
  // its row stride phmax is a multiple of 4
  const size_t diag = (size_t)kNB * (kNB + 1) * sizeof(T);
  const int phmax = (max_w + 3) & ~3;
  const size_t panel = (size_t)phmax * kNB * sizeof(T);
  if (diag + panel <= kSmemCap) {
    auto kern = k_band_potrf<T, kNB, true>;
    GENEO_CUDA(allow_smem(kern));
    kern<<<count, kThreads, diag + panel, s>>>(base, d_desc, phmax, st, weak, weak_tol); note_launch();
  } else {
    auto kern = k_band_potrf<T, kNB, false>;
    kern<<<count, kThreads, diag, s>>>(base, d_desc, 0, st, weak, weak_tol); note_launch();
  }
  GENEO_CUDA(cudaGetLastError());
  return band_blkinv(base, d_desc, count, max_n, blk_mask, s);
}

// Shared memory of one solve launch with k right-hand sides.
template <typename T>
size_t solve_smem(int max_w, int k, int ring, int snb, int stages) {
  const int ld = band_ld(max_w);
  return 128 + sizeof(T) * ((size_t)stages * snb * ld + (size_t)ring * k + (size_t)snb * k + 4 * kThreads);
}

// Column split of a multi-right-hand-side launch: when a batch holds at most
// half as many matrices as the GPU has SMs, each matrix's columns are cut
// into parts (grid y) that run on otherwise idle SMs, each part a shorter
// dependent sweep with less work per step; at most `units` parts and no more
// blocks than SMs.
inline int split_parts(int count, int units) {
  const int sms = sm_count();
  if (count <= 0 || 2 * count > sms || units <= 1) return 1;
  return std::max(1, std::min(units, sms / count));
}

// Solves with the kernels that do not apply a band's row scaling (the
// caller scales the vectors around them).
template <typename T, typename A = T>
geneo_status_t band_solve_plain(const T* base, const BandDesc* d_desc, int count, int max_w,
                                double* xbase, const int64_t* xoff, int nrhs, const int32_t* nrhs_dev,
                                const int32_t* skip_dev, DevStatus* st, cudaStream_t s, int live = 0) {
  if (live <= 0) live = count;
  if (nrhs == 1) {
    int snb = 16;
    if (solve_smem<T>(max_w, 1, next_pow2(max_w + 32), 16, 2) > kSmemCap) snb = 4;
    const int ring = next_pow2(max_w + 2 * snb);
    const size_t smem = solve_smem<T>(max_w, 1, ring, snb, 2);
    if (smem > 227 * 1024) return GENEO_ERR_ARG;
    auto kern = snb == 16 ? k_band_solve<T, A, 16, 1, 2> : k_band_solve<T, A, 4, 1, 2>;
    GENEO_CUDA(allow_smem(kern));
    kern<<<count, kThreads, smem, s>>>(base, d_desc, xbase, xoff, 0, 1, nrhs_dev, skip_dev, ring, st); note_launch();
    GENEO_CUDA(cudaGetLastError());
    return GENEO_OK;
  }
  constexpr int stg = Stages<T>::v;
  int snb = 16;
  if (solve_smem<T>(max_w, 1, next_pow2(max_w + 32), 16, stg) > kSmemCap) snb = 4;
  const int ring = next_pow2(max_w + 2 * snb);
  // right-hand sides per launch: as many as fit in shared memory, at most 64
  // (8 warps x 8 register slots; the forward partial-sum buffer holds
  // 4 * kThreads values for b * ceil(k / 4) <= kThreads tiles)
  int kmax = std::min(nrhs, 64);
  while (kmax > 1 && solve_smem<T>(max_w, kmax, ring, snb, stg) > kSmemCap) kmax = (kmax + 1) / 2;
  const size_t smem = solve_smem<T>(max_w, kmax, ring, snb, stg);
  if (smem > 227 * 1024) return GENEO_ERR_ARG;  // band too wide for the streamed solve
  auto kern = snb == 16 ? k_band_solve<T, A, 16, 8, stg> : k_band_solve<T, A, 4, 8, stg>;
  GENEO_CUDA(allow_smem(kern));
  for (int c0 = 0; c0 < nrhs; c0 += kmax) {
    const int kc = std::min(kmax, nrhs - c0);
    const int nsplit = split_parts(live, (kc + 3) / 4);  // parts of at least 4 columns
    kern<<<dim3(count, nsplit), kThreads, smem, s>>>(base, d_desc, xbase, xoff, c0, kc, nrhs_dev, skip_dev, ring,
                                                     st);
    note_launch();
    GENEO_CUDA(cudaGetLastError());
  }
  return GENEO_OK;
}

template <typename T, bool DS>
geneo_status_t band_solve_impl(const T* base, const BandDesc* d_desc, int count, int blk, int max_w,
                               double* xbase, const int64_t* xoff, int nrhs, const int32_t* nrhs_dev,
                               const int32_t* skip_dev, DevStatus* st, cudaStream_t s, int max_n, int tc_passes,
                               int slots, int active) {
  if (count <= 0 || nrhs <= 0) return GENEO_OK;
  // matrices to solve side by side (this batch's, or those of all classes)
  const int live = active > 0 ? active : count;
  if (blk > 0)
    return sweep_solve<T, DS>(base, d_desc, count, blk, max_w, max_n, xbase, xoff, nrhs, nrhs_dev, skip_dev, st, s,
                              tc_passes, slots, live);
  // bands too wide for the sweeps: the streamed kernel on the factor itself,
  // the vectors scaled around the solve where the bands are equilibrated
  // (FP32 factors); double-single covers several right-hand sides
  if constexpr (sizeof(T) == 4) {
    const int gx = std::max(1, std::min(64, (max_n > 0 ? max_n : 4096) * nrhs / 256));
    k_band_scale_x<T><<<dim3(gx, count), 256, 0, s>>>(base, d_desc, xbase, xoff, 0, nrhs, nrhs_dev, skip_dev);
    note_launch();
    GENEO_TRY(band_solve_plain<T>(base, d_desc, count, max_w, xbase, xoff, nrhs, nrhs_dev, skip_dev, st, s, live));
    k_band_scale_x<T><<<dim3(gx, count), 256, 0, s>>>(base, d_desc, xbase, xoff, 0, nrhs, nrhs_dev, skip_dev);
    note_launch();
    GENEO_CUDA(cudaGetLastError());
    return GENEO_OK;
  } else if (DS && nrhs > 1) {
    return band_solve_plain<T, dsv>(base, d_desc, count, max_w, xbase, xoff, nrhs, nrhs_dev, skip_dev, st, s, live);
  } else {
    return band_solve_plain<T>(base, d_desc, count, max_w, xbase, xoff, nrhs, nrhs_dev, skip_dev, st, s, live);
  }
}

template <typename T>
geneo_status_t band_solve(const T* base, const BandDesc* d_desc, int count, int blk, int max_w,
                          double* xbase, const int64_t* xoff, int nrhs, const int32_t* nrhs_dev,
                          const int32_t* skip_dev, DevStatus* st, cudaStream_t s, int max_n, int tc_passes,
                          int slots, int active) {
  return band_solve_impl<T, false>(base, d_desc, count, blk, max_w, xbase, xoff, nrhs, nrhs_dev, skip_dev, st, s,
                                   max_n, tc_passes, slots, active);
}

geneo_status_t band_solve_ds(const double* base, const BandDesc* d_desc, int count, int blk, int max_w,
                             double* xbase, const int64_t* xoff, int nrhs, const int32_t* nrhs_dev,
                             const int32_t* skip_dev, DevStatus* st, cudaStream_t s, int max_n, int active) {
  return band_solve_impl<double, true>(base, d_desc, count, blk, max_w, xbase, xoff, nrhs, nrhs_dev, skip_dev, st,
                                       s, max_n, 3, 0, active);
}

template geneo_status_t band_potrf<double>(double*, const BandDesc*, int, int, int, int, DevStatus*,
                                           cudaStream_t, bool, int32_t*, float, const Tc5Plan*);
template geneo_status_t band_potrf<float>(float*, const BandDesc*, int, int, int, int, DevStatus*,
                                          cudaStream_t, bool, int32_t*, float, const Tc5Plan*);
template geneo_status_t band_solve<double>(const double*, const BandDesc*, int, int, int, double*,
                                           const int64_t*, int, const int32_t*, const int32_t*,
                                           DevStatus*, cudaStream_t, int, int, int, int);
template geneo_status_t band_solve<float>(const float*, const BandDesc*, int, int, int, double*,
                                          const int64_t*, int, const int32_t*, const int32_t*,
                                          DevStatus*, cudaStream_t, int, int, int, int);

}  // namespace geneo
