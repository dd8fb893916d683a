// Batched block inversion g = M^-1 of the sweeps of Eq. (1): Gauss-Jordan elimination with
// partial pivoting (largest |m|^2, lowest row on ties; magnitudes to FP64 accuracy, as FP32 pairs
// for FP32 storage) and the pivot reciprocal in the storage precision (the FP32 form is refined
// by Newton-Schulz steps afterwards).
//
// Small n: one CTA per matrix, the whole matrix in shared memory.
// Larger n: blocked Gauss-Jordan.  A panel of nb columns is eliminated, and the remaining columns get
// the rank-nb update  A[:, rest] += Panel * A[pivot rows, rest]  (pivot rows zeroed first).  FP64 form:
// the panel is eliminated in shared memory, the same kernel moves the exchanged rows of the whole
// matrix, and the update is a batched product in place.  FP32 form: the panel is eliminated in registers
// and no row is moved; the update reads the matrix through the panel's exchanges and writes it to a
// second buffer.  The column permutation that the pivoting leaves is undone at the end.
#include <algorithm>
#include <atomic>
#include <type_traits>
#include <utility>

#include "common.cuh"
#include "profile.cuh"
#include "tc_slice.cuh"

namespace negf {

namespace {

constexpr int kThreads = 256;
constexpr size_t kSmemBudget = 180 * 1024;

// Pivot magnitude |a|^2 = hi + lo.  FP64 storage: hi = |a|^2 in FP64, lo = 0.  FP32 storage: the
// exact squares as FP32 pairs (product and its fmaf residual) and the exact sum of the leading
// parts (TwoSum), so hi + lo carries about 48 bits: an FP64-class pivot decision without the
// FP64 pipe.  Intrinsics keep the compiler from fusing the steps.  (The entries of the blocks
// inverted here lie between about 1e-19 and 1e19 in magnitude, where no square over- or
// underflows in FP32.)
template <typename R>
struct Mag {
  R hi, lo;
};
template <typename R>
__device__ __forceinline__ Mag<R> mag2(cx<R> a) {
  if constexpr (sizeof(R) == 8) {
    const double v = a.re * a.re + a.im * a.im;
    // NaN, of either sign, gets a value that loses to every other one
    const bool nan = (unsigned long long)__double_as_longlong(v) > 0x7ff0000000000000ull;
    return Mag<R>{nan ? -0.5 : v, 0.0};
  } else {
    const float p = __fmul_rn(a.re, a.re), q = __fmul_rn(a.im, a.im);
    const float ep = fmaf(a.re, a.re, -p), eq = fmaf(a.im, a.im, -q);
    const float s = __fadd_rn(p, q);
    const float bq = __fsub_rn(s, p);
    const float t = __fadd_rn(__fsub_rn(p, __fsub_rn(s, bq)), __fsub_rn(q, bq));
    return Mag<R>{s, __fadd_rn(t, __fadd_rn(ep, eq))};
  }
}
// a (row ia) is a better pivot than b (row ib): larger magnitude, lower row on ties.  The sign of
// (a.hi - b.hi) + (a.lo - b.lo) is that of the exact difference except within FP64-level ties.
template <typename R>
__device__ __forceinline__ bool better(Mag<R> a, int ia, Mag<R> b, int ib) {
  if constexpr (sizeof(R) == 8) {
    // lo = 0; magnitudes order like their bit patterns (the start value -1 below all of them, the
    // -0.5 for NaN below that), and integer comparisons leave the scarce FP64 pipe alone
    const long long x = __double_as_longlong(a.hi), y = __double_as_longlong(b.hi);
    return x > y || (x == y && ia < ib);
  } else {
    const R d = (a.hi - b.hi) + (a.lo - b.lo);
    return d > R(0) || (d == R(0) && ia < ib);
  }
}

// 1 / a, flagging an exactly zero pivot (replaced by a tiny number so the sweep goes on).  FP64
// for FP64 storage; for FP32, a is first scaled by the power of two 2^-e that brings its larger
// component into [0.5, 1), so |a'|^2 lies in [0.25, 2) and 1/a = conj(a') 2^-e / |a'|^2 loses
// nothing to overflow or underflow.
template <typename R>
__device__ __forceinline__ cx<R> pivot_recip(cx<R> a, int32_t* st) {
  if (a.re == R(0) && a.im == R(0)) {
    if (st) atomicOr(st, NEGF_PT_SINGULAR);
    a.re = sizeof(R) == 8 ? R(1e-300) : R(1e-30);
  }
  if constexpr (sizeof(R) == 8) {
    return crecip(a);
  } else {
    int e;
    frexpf(fmaxf(fabsf(a.re), fabsf(a.im)), &e);
    const float ar = ldexpf(a.re, -e), ai = ldexpf(a.im, -e);
    const float inv = ldexpf(1.0f / __fmaf_rn(ar, ar, __fmul_rn(ai, ai)), -e);
    return mkc<float>(ar * inv, -ai * inv);
  }
}

// Per-CTA scratch of one Gauss-Jordan column step.
template <typename R>
struct GjScratch {
  Mag<R> sv[32];
  int si[32];
  cx<R> d;
};

// One Gauss-Jordan step on column jj of the shared-memory array P (rows x w, row stride w):
// pivot search over rows [j, rows) (largest |m|^2, lowest row on ties), swap of rows j and the
// pivot row, pivot reciprocal (pivot_recip), and elimination of column jj from all
// other rows.  f[rows] and prow[w] are shared scratch.  Three block barriers per column:
//   (1) after the per-warp argmax, (2) after the swap / column copy / reciprocal, (3) after the
//   update.  Every thread combines the per-warp winners itself, and the elimination scales the
//   pivot row on the fly from an unscaled copy, so no further barrier is needed.
// Returns the pivot row.
template <typename R>
__device__ int gj_column(cx<R>* P, int rows, int w, int j, int jj, cx<R>* f, cx<R>* prow,
                         GjScratch<R>& sc, int32_t* st) {
  const int tid = threadIdx.x, bd = blockDim.x, lane = tid & 31, wid = tid >> 5;
  Mag<R> best{R(-1), R(0)};
  int bi = rows;
  for (int r = j + tid; r < rows; r += bd) {
    const Mag<R> v = mag2(P[(long long)r * w + jj]);
    if (better(v, r, best, bi)) {
      best = v;
      bi = r;
    }
  }
  for (int off = 16; off > 0; off >>= 1) {
    const Mag<R> ov{__shfl_down_sync(0xffffffffu, best.hi, off),
                    __shfl_down_sync(0xffffffffu, best.lo, off)};
    const int oi = __shfl_down_sync(0xffffffffu, bi, off);
    if (better(ov, oi, best, bi)) {
      best = ov;
      bi = oi;
    }
  }
  if (lane == 0) {
    sc.sv[wid] = best;
    sc.si[wid] = bi;
  }
  __syncthreads();  // (1)
  Mag<R> b = sc.sv[0];
  int pi = sc.si[0];
  const int nw = bd >> 5;
  for (int k = 1; k < nw; ++k)
    if (better(sc.sv[k], sc.si[k], b, pi)) {
      b = sc.sv[k];
      pi = sc.si[k];
    }
  const int pr = (pi >= rows) ? j : pi;
  // swap rows j <-> pr, keep the unscaled pivot row, copy column jj (as it is after the swap)
  for (int c = tid; c < w; c += bd) {
    const cx<R> a = P[(long long)j * w + c], v = P[(long long)pr * w + c];
    P[(long long)j * w + c] = v;
    P[(long long)pr * w + c] = a;
    prow[c] = v;
    if (c == jj) {
      f[j] = v;
      f[pr] = a;
      sc.d = pivot_recip(v, st);
    }
  }
  for (int r = tid; r < rows; r += bd)
    if (r != j && r != pr) f[r] = P[(long long)r * w + jj];
  __syncthreads();  // (2)
  const cx<R> d = sc.d;
  if (w <= bd) {
    // Thread (r0, c) updates rows r0, r0 + rstep, ...  of column c, four rows per batch with the
    // loads ahead of the stores (P and f are disjoint).  The pivot column (c == jj) starts from 0
    // so that it becomes -f[r] d; row j is computed like the others and then overwritten with the
    // scaled pivot row by the thread that owns it.
    const int c = tid % w;
    const int r0 = tid / w, rstep = bd / w;
    if (r0 < rstep) {
      const bool pcol = (c == jj);
      const cx<R> pj = pcol ? d : prow[c] * d;
      const cx<R> zero = mkc<R>(R(0), R(0));
      int r = r0;
      for (; r + 3 * rstep < rows; r += 4 * rstep) {
        cx<R> v[4], fr[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          v[u] = P[(long long)(r + u * rstep) * w + c];
          fr[u] = f[r + u * rstep];
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          cx<R> x = pcol ? zero : v[u];
          x.re = x.re - (fr[u].re * pj.re - fr[u].im * pj.im);
          x.im = x.im - (fr[u].re * pj.im + fr[u].im * pj.re);
          P[(long long)(r + u * rstep) * w + c] = x;
        }
      }
      for (; r < rows; r += rstep) {
        const cx<R> fr = f[r];
        cx<R> x = pcol ? zero : P[(long long)r * w + c];
        x.re = x.re - (fr.re * pj.re - fr.im * pj.im);
        x.im = x.im - (fr.re * pj.im + fr.im * pj.re);
        P[(long long)r * w + c] = x;
      }
      if (j % rstep == r0) P[(long long)j * w + c] = pj;
    }
  } else {
    for (int r = 0; r < rows; ++r) {
      const cx<R> fr = f[r];
      for (int c = tid; c < w; c += bd) {
        const cx<R> pj = (c == jj) ? d : prow[c] * d;
        cx<R>* e = P + (long long)r * w + c;
        if (r == j) {
          *e = pj;
        } else if (c == jj) {
          *e = mkc<R>(R(0), R(0)) - fr * d;
        } else {
          cx<R> v = *e;
          v.re = v.re - (fr.re * pj.re - fr.im * pj.im);
          v.im = v.im - (fr.re * pj.im + fr.im * pj.re);
          *e = v;
        }
      }
    }
  }
  __syncthreads();  // (3)
  return pr;
}

template <typename R>
__global__ void __launch_bounds__(kThreads) k_gj_small(int n, BM<R> Mm, BM<R> X, int32_t* status,
                                                       const int32_t* active) {
  const int p = blockIdx.x;
  if (active && !active[p]) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cx<R>* A = reinterpret_cast<cx<R>*>(smem_raw);
  cx<R>* f = A + (size_t)n * n;
  cx<R>* prow = f + n;
  int* perm = reinterpret_cast<int*>(prow + n);
  int* src = perm + n;
  __shared__ GjScratch<R> sc;
  int32_t* st = status ? status + p : nullptr;
  const cx<R>* m = bat(Mm, p);
  for (int r = 0; r < n; ++r)
    for (int c = threadIdx.x; c < n; c += blockDim.x) A[r * n + c] = m[(long long)r * Mm.ld + c];
  __syncthreads();
  for (int j = 0; j < n; ++j) {
    const int pr = gj_column(A, n, n, j, j, f, prow, sc, st);
    if (threadIdx.x == 0) perm[j] = pr;
  }
  if (threadIdx.x == 0) {
    for (int c = 0; c < n; ++c) src[c] = c;
    for (int j = n - 1; j >= 0; --j) {
      int t = src[j];
      src[j] = src[perm[j]];
      src[perm[j]] = t;
    }
  }
  __syncthreads();
  cx<R>* x = bat(X, p);
  for (int r = 0; r < n; ++r)
    for (int c = threadIdx.x; c < n; c += blockDim.x)
      x[(long long)r * X.ld + c] = A[r * n + src[c]];
}

// The multiply-adds of a step are written out, each rounding in its place, so that the result does
// not depend on how the compiler contracts them.  `other` takes the imaginary part's products in
// the other order: the elimination has always done so in the rows that its unrolling by four left
// over, and the results stay the same bit for bit.
__device__ __forceinline__ float fma_rn(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double fma_rn(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float sub_rn(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ double sub_rn(double a, double b) { return __dsub_rn(a, b); }
template <typename R>
__device__ __forceinline__ cx<R> cmul(cx<R> a, cx<R> b) {
  return mkc<R>(fma_rn(a.re, b.re, -mul_rn(a.im, b.im)), fma_rn(a.re, b.im, mul_rn(a.im, b.re)));
}
template <typename R>
__device__ __forceinline__ void eliminate(cx<R>& x, cx<R> f, cx<R> p, bool other) {
  x.re = sub_rn(x.re, fma_rn(f.re, p.re, -mul_rn(f.im, p.im)));
  // (a product has the same rounding whichever factor comes first)
  const R a = other ? f.re : f.im, b = other ? p.im : p.re;
  const R c = other ? f.im : f.re, d = other ? p.re : p.im;
  x.im = sub_rn(x.im, fma_rn(a, b, mul_rn(c, d)));
}

// One CTA per matrix, the whole matrix in shared memory.  A step's chain (largest entry of the
// column, reciprocal) is as long as its update: FP64 issues two lanes per clock and SM, and a
// division is some twenty operations one after another.  So the first warp updates the next column
// ahead of the rest and finds that column's pivot and reciprocal while the other warps update the
// remaining columns.  128 blocks of 40: 284 -> 230 us, 16 of 64: 682 -> 588, 30 of 106: 2436 -> 2225.
// (Padded rows and a scheduler kept free for the chain gave nothing more.  FP32 has no such pipe: there
// the single warp's column is what a step waits for, 8 blocks of 100 680 -> 946 us, so it keeps the
// form above.)
__global__ void __launch_bounds__(kThreads) k_gj_small64(int n, BM<double> Mm, BM<double> X,
                                                         int32_t* status, const int32_t* active) {
  const int p = blockIdx.x;
  if (active && !active[p]) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  z64* A = reinterpret_cast<z64*>(smem_raw);
  z64* f = A + (size_t)n * n;  // the pivot column
  z64* prow = f + n;            // the scaled pivot row
  int* perm = reinterpret_cast<int*>(prow + n);
  int* src = perm + n;
  __shared__ unsigned char other[kThreads];  // n <= kThreads (gj_fits_small)
  __shared__ z64 recip;
  __shared__ int pivot;
  int32_t* st = status ? status + p : nullptr;
  const z64* m = bat(Mm, p);
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const z64 zero = mkc(0.0, 0.0);
  for (int r = 0; r < n; ++r)
    for (int c = tid; c < n; c += kThreads) A[r * n + c] = m[(long long)r * Mm.ld + c];
  const int old = kThreads / n;  // rows per step of the elimination unrolled by four
  if (tid < n) other[tid] = tid % old + (tid / (4 * old) * 4 + 3) * old >= n;
  __syncthreads();
  // the pivot of column j among rows [j, n) and its reciprocal (first warp)
  auto search = [&](int j) {
    Mag<double> best{-1.0, 0.0};
    int bi = n;
    for (int r = lane; r < n; r += 32) {
      if (r < j) continue;
      const Mag<double> v = mag2(A[r * n + j]);
      if (better(v, r, best, bi)) {
        best = v;
        bi = r;
      }
    }
    for (int off = 16; off > 0; off >>= 1) {
      const Mag<double> ov{__shfl_down_sync(0xffffffffu, best.hi, off),
                      __shfl_down_sync(0xffffffffu, best.lo, off)};
      const int oi = __shfl_down_sync(0xffffffffu, bi, off);
      if (better(ov, oi, best, bi)) {
        best = ov;
        bi = oi;
      }
    }
    if (lane == 0) {
      const int pr = bi >= n ? j : bi;
      pivot = perm[j] = pr;
      recip = pivot_recip(A[pr * n + j], st);
    }
  };
  if (wid == 0) search(0);
  constexpr int kWorkers = kThreads - 32;
  const int dr = kWorkers / n, dc = kWorkers - dr * n;
  __syncthreads();
  for (int j = 0; j < n; ++j) {
    const int pr = pivot;
    // row pr receives row j; the pivot row is kept scaled, row j itself is written with it below
    if (tid < n) {
      const z64 a = A[j * n + tid], v = A[pr * n + tid];
      A[pr * n + tid] = a;
      prow[tid] = tid == j ? recip : cmul(v, recip);
      if (tid == j)
        f[pr] = a;
      else if (tid != pr)
        f[tid] = A[tid * n + j];
    }
    __syncthreads();
    if (wid == 0) {
      const int c = j + 1;
      if (c < n) {
        const z64 pc = prow[c];
        for (int r = lane; r < n; r += 32) {
          z64 x = A[r * n + c];
          eliminate(x, f[r], pc, other[r]);
          A[r * n + c] = r == j ? pc : x;
        }
        __syncwarp();
        search(c);
      }
    } else {
      int r = (tid - 32) / n, c = tid - 32 - r * n;
      while (r < n) {
        if (c != j + 1) {
          z64 x = c == j ? zero : A[r * n + c];
          eliminate(x, f[r], prow[c], other[r]);
          A[r * n + c] = r == j ? prow[c] : x;
        }
        r += dr;
        c += dc;
        if (c >= n) {
          c -= n;
          ++r;
        }
      }
    }
    __syncthreads();
  }
  if (tid == 0) {
    for (int c = 0; c < n; ++c) src[c] = c;
    for (int j = n - 1; j >= 0; --j) {
      int t = src[j];
      src[j] = src[perm[j]];
      src[perm[j]] = t;
    }
  }
  __syncthreads();
  z64* x = bat(X, p);
  for (int r = 0; r < n; ++r)
    for (int c = tid; c < n; c += kThreads) x[(long long)r * X.ld + c] = A[r * n + src[c]];
}

// Panel step of the blocked form: columns [k0, k0 + w) of A (n x n, in global memory).
// The panel is eliminated in shared memory; then, for the columns outside the panel, one pass
// per column (each column owned by one thread, so no barrier) moves the swapped rows to their
// final place, copies the pivot rows into T and zeroes them in A.  The row swaps of the panel
// only ever move a panel row's content to an outside row, so reading all sources before any
// panel row is cleared is enough to apply them at once.
template <typename R>
__global__ void __launch_bounds__(kThreads) k_gj_panel(int n, int k0, int w, int nb, BM<R> Am,
                                                       cx<R>* U, cx<R>* T, int32_t* piv,
                                                       int32_t* status, const int32_t* active) {
  chain_next();
  chain_wait();
  const int p = blockIdx.x;
  if (active && !active[p]) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cx<R>* P = reinterpret_cast<cx<R>*>(smem_raw);
  cx<R>* f = P + (size_t)n * w;
  cx<R>* prow = f + n;
  int* cont = reinterpret_cast<int*>(prow + w);  // [n] source row of each row's final content
  int* spv = cont + n;                           // [w] pivot rows of this panel
  __shared__ GjScratch<R> sc;
  int32_t* st = status ? status + p : nullptr;
  cx<R>* a = bat(Am, p);
  const long long ld = Am.ld;
  int32_t* pv = piv + (long long)p * n;
  {
    // the panel columns, eight rows per batch with the loads ahead of the stores
    const int c = threadIdx.x % w, r0 = threadIdx.x / w, rs = blockDim.x / w;
    if (r0 < rs)
      for (int rb = r0; rb < n; rb += 8 * rs) {
        cx<R> v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u)
          if (rb + u * rs < n) v[u] = a[(long long)(rb + u * rs) * ld + k0 + c];
#pragma unroll
        for (int u = 0; u < 8; ++u)
          if (rb + u * rs < n) P[(long long)(rb + u * rs) * w + c] = v[u];
      }
  }
  for (int r = threadIdx.x; r < n; r += blockDim.x) cont[r] = r;
  __syncthreads();
  for (int jj = 0; jj < w; ++jj) {
    const int j = k0 + jj;
    const int pr = gj_column(P, n, w, j, jj, f, prow, sc, st);
    if (threadIdx.x == 0) {
      pv[j] = pr;
      spv[jj] = pr;
      const int t = cont[j];
      cont[j] = cont[pr];
      cont[pr] = t;
    }
  }
  __syncthreads();
  cx<R>* Tp = T + (long long)p * nb * n;
  const cx<R> zero = mkc<R>(R(0), R(0));
  for (int c = threadIdx.x; c < n; c += blockDim.x) {
    if (c >= k0 && c < k0 + w) {
      for (int jj = 0; jj < w; ++jj) Tp[(long long)jj * n + c] = zero;
      continue;
    }
    // (1) final pivot rows -> T, read before anything of this column is written
    for (int j0 = 0; j0 < w; j0 += 8) {
      cx<R> v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (j0 + u < w) v[u] = a[(long long)cont[k0 + j0 + u] * ld + c];
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (j0 + u < w) Tp[(long long)(j0 + u) * n + c] = v[u];
    }
    // (2) rows below the panel that took part in a swap receive a panel row's content (all
    // sources are panel rows, read before any is cleared; loads batched ahead of the stores)
    for (int j0 = 0; j0 < w; j0 += 8) {
      cx<R> v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (j0 + u < w && spv[j0 + u] >= k0 + w)
          v[u] = a[(long long)cont[spv[j0 + u]] * ld + c];
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (j0 + u < w && spv[j0 + u] >= k0 + w) a[(long long)spv[j0 + u] * ld + c] = v[u];
    }
    // (3) the pivot rows are cleared outside the panel
    for (int jj = 0; jj < w; ++jj) a[(long long)(k0 + jj) * ld + c] = zero;
  }
  cx<R>* Up = U + (long long)p * n * nb;
  for (int r = threadIdx.x / w; r < n; r += blockDim.x / w) {
    const int c = threadIdx.x % w;
    if (threadIdx.x / w < (int)blockDim.x / w) {
      const cx<R> v = P[(long long)r * w + c];
      a[r * ld + k0 + c] = v;
      Up[(long long)r * nb + c] = v;
    }
  }
}

// Pivot candidates.  hi + lo of mag2 is brought to h = RN(hi + lo) and the exact rest l, so that the
// larger sum has the larger h, then the larger l; equal sums go to the lower row.  Keys order like
// unsigned integers (a candidate's h key is at least 1), so a warp finds its winner with reductions
// of the integer unit.
struct Cand {
  uint32_t h, l;
  int row;
};
__device__ __forceinline__ Cand candidate(cx<float> a, int row) {
  const Mag<float> m = mag2(a);
  const float h = __fadd_rn(m.hi, m.lo);
  const uint32_t l = __float_as_uint(__fsub_rn(m.lo, __fsub_rn(h, m.hi)));
  return Cand{__float_as_uint(h) + 1u, l & 0x80000000u ? ~l : l | 0x80000000u, row};
}
__device__ __forceinline__ bool wins(const Cand& a, const Cand& b) {
  return a.h > b.h || (a.h == b.h && (a.l > b.l || (a.l == b.l && a.row < b.row)));
}
__device__ __forceinline__ Cand warp_winner(Cand c) {
  const uint32_t full = 0xffffffffu;
  const uint32_t h = __reduce_max_sync(full, c.h);
  const uint32_t tied = __ballot_sync(full, c.h == h);
  int src = __ffs((int)tied) - 1;
  if (tied & (tied - 1)) {
    const uint32_t l = __reduce_max_sync(full, c.h == h ? c.l : 0u);
    const bool in = c.h == h && c.l == l;
    const int row = (int)__reduce_min_sync(full, in ? (uint32_t)c.row : 0xffffffffu);
    src = __ffs((int)__ballot_sync(full, in && c.row == row)) - 1;
  }
  return Cand{h, __shfl_sync(full, c.l, src), __shfl_sync(full, c.row, src)};
}
// pivot_recip with the scaling by powers of two done on the exponent field; far exponents take the
// general form (the same numbers, rounded at the same places)
__device__ __forceinline__ cx<float> pivot_recip32(cx<float> a, int32_t* st) {
  const uint32_t ex = __float_as_uint(fmaxf(fabsf(a.re), fabsf(a.im))) >> 23;  // no sign bit
  if (ex < 64u || ex > 190u) return pivot_recip(a, st);
  const float down = __uint_as_float((253u - ex) << 23);  // 2^(126 - ex): the larger part in [0.5, 1)
  const float ar = __fmul_rn(a.re, down), ai = __fmul_rn(a.im, down);
  const float inv = __fmul_rn(__frcp_rn(__fmaf_rn(ar, ar, __fmul_rn(ai, ai))), down);
  return mkc<float>(__fmul_rn(ar, inv), __fmul_rn(-ai, inv));
}

// FP32 form of the blocked elimination.  A panel is eliminated in registers, and the trailing
// update reads the matrix through the panel's row exchanges and writes it to a second buffer, so no
// pass over the matrix moves rows: src and dst alternate from panel to panel.
//
// Panel step: columns [k0, k0 + w) of src (w = W, the panel width, but for a matrix's LAST panel,
// which may be narrower).  Thread (g, c) keeps rows g, g + kG, ... of column c in registers for all
// steps; a step exchanges only the pivot column f, the two rows of the exchange and the pivot
// through shared memory.  Writes the eliminated panel to U and to its columns of dst, the pivot
// rows, and for every row the source row of its content after the panel's exchanges (cont).
//
// Bound by the chain of W steps (pivot search, exchange, update, a barrier between each) on one SM
// per item: 65 us for 64 items of n = 400, W = 32, where a panel in shared memory on 256 threads
// that also moved the rows of the whole matrix took 110 us.  512 threads: 1024 spend more on the
// part of a step that every warp repeats, and a test per slot (instead of filler rows) parted the
// slots' loads and took 140 us.
constexpr int kPanelThreads = 512, kPanelWarps = kPanelThreads / 32;
template <int W, int NR, bool LAST>
__global__ void __launch_bounds__(kPanelThreads)
    k_gj_panel32(int n, int k0, int w, int nb, const cx<float>* srcs, cx<float>* dsts,
                 cx<float>* U, int32_t* piv, int32_t* conts, int32_t* status,
                 const int32_t* active) {
  chain_next();
  chain_wait();
  const int p = blockIdx.x;
  if (active && !active[p]) return;
  constexpr int kG = kPanelThreads / W;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  // slot NR - 1 holds the last rows: slot i of group g has row g + i kG - off, and the rows outside
  // [0, n) are zeros that only fill the threads (every slot of every thread then does the same work,
  // with no test that would part the slots' instructions)
  const int off = (NR - 1 - n / kG) * kG;
  cx<float>* fbuf = reinterpret_cast<cx<float>*>(smem_raw);  // [2][NR kG] pivot columns in turn
  int* cont = reinterpret_cast<int*>(fbuf + 2 * NR * kG);    // [n]
  const cx<float> zero = mkc<float>(0.0f, 0.0f);
  __shared__ Cand best_of[kPanelWarps];
  __shared__ cx<float> rowj[W], rowp[W], recip;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int c = tid % W, g = tid / W;
  int32_t* st = status ? status + p : nullptr;
  const long long nn = (long long)n * n;
  const cx<float>* a = srcs + p * nn;
  auto row_of = [&](int i) { return g + i * kG - off; };
  // rows that an unrolling by four of steps of `old` rows leaves over: in a full panel such rows
  // are in the last four slots
  const int old = 256 / w;
  auto left_over = [&](int r) { return r % old + (r / (4 * old) * 4 + 3) * old >= n; };
  constexpr int kTail = LAST ? 0 : NR - 4;
  unsigned long long other = 0;
#pragma unroll
  for (int i = kTail; i < NR; ++i)
    if (row_of(i) >= 0 && left_over(row_of(i))) other |= 1ull << i;
  cx<float> v[NR];
#pragma unroll
  for (int i = 0; i < NR; ++i) {
    const int r = row_of(i);
    v[i] = (r >= 0 && r < n && c < w) ? a[(long long)r * n + k0 + c] : zero;
  }
  for (int r = tid; r < n; r += kPanelThreads) cont[r] = r;
  for (int jj = 0; jj < w; ++jj) {
    const int j = k0 + jj;
    cx<float>* slots = fbuf + (jj & 1) * NR * kG;  // the last step's column may still be read
    cx<float>* f = slots + off;                    // by row
    // the pivot column, and its largest entry in rows [j, n).  Its registers start the update from 0
    if (c == jj) {
#pragma unroll
      for (int i = 0; i < NR; ++i) {
        slots[g + i * kG] = v[i];
        v[i] = zero;
      }
    }
    __syncthreads();
    const int w0 = n > kPanelThreads ? 0 : j / 32;  // first warp with a candidate
    const int w1 = min(kPanelWarps, (n + 31) / 32);
    if (wid >= w0 && wid < w1) {
      Cand best{0u, 0u, n};
      for (int r = tid; r < n; r += kPanelThreads) {
        if (r < j) continue;
        const Cand cand = candidate(f[r], r);
        if (wins(cand, best)) best = cand;
      }
      best = warp_winner(best);
      if (lane == 0) best_of[wid] = best;
    }
    __syncthreads();
    // every warp combines the winners
    const bool mine = lane >= w0 && lane < w1;
    const Cand top = warp_winner(mine ? best_of[lane] : Cand{0u, 0u, n});
    const int pr = top.row >= n ? j : top.row;
    // rows j and pr go to shared memory
    const int ij = (j + off) / kG, ip = (pr + off) / kG;
    const bool own_j = j % kG == g, own_p = pr % kG == g;
    if (own_j || own_p) {
#pragma unroll
      for (int i = 0; i < NR; ++i) {
        if (own_j && i == ij) rowj[c] = v[i];
        if (own_p && i == ip) rowp[c] = v[i];
      }
    }
    if (tid == 0) {
      recip = pivot_recip32(f[pr], st);
      f[pr] = f[j];  // after the exchange row pr holds row j's old content
      piv[(long long)p * n + j] = pr;
      const int t = cont[j];
      cont[j] = cont[pr];
      cont[pr] = t;
    }
    __syncthreads();
    const cx<float> d = recip;
    const cx<float> pj = c == jj ? d : cmul(rowp[c], d);
    if (own_p) {
      const cx<float> moved = rowj[c];
#pragma unroll
      for (int i = 0; i < NR; ++i)
        if (i == ip) v[i] = moved;
    }
#pragma unroll
    for (int i = 0; i < NR; ++i)
      eliminate(v[i], slots[g + i * kG], pj, i >= kTail && (other >> i & 1ull));
    if (own_j) {
#pragma unroll
      for (int i = 0; i < NR; ++i)
        if (i == ij) v[i] = pj;
    }
  }
  __syncthreads();
  cx<float>* o = dsts + p * nn;
  cx<float>* u = U + (long long)p * n * nb;
#pragma unroll
  for (int i = 0; i < NR; ++i) {
    const int r = row_of(i);
    if (r >= 0 && r < n && c < w) {
      o[(long long)r * n + k0 + c] = v[i];
      u[(long long)r * nb + c] = v[i];
    }
  }
  for (int r = tid; r < n; r += kPanelThreads) conts[(long long)p * n + r] = cont[r];
}

// Trailing update of a panel step: dst = E src + U T outside the panel's columns, where E applies
// the panel's row exchanges (row r of the result starts from row cont[r] of src) and clears the
// pivot rows, U is the eliminated panel (n x w, row stride nb) and T the pivot rows
// src[cont[k0 + k]].  An 80 x 80 block per CTA (n = 400 is 5 x 5 blocks with no padding; 64 x 64
// blocks would pad it to 448^2, 25 % more work), each thread 5 x 5 complex accumulators: rows
// ty + 16 i, columns tx + 16 j.  The whole U and T blocks are staged in shared memory at once (one
// barrier), and src is read into the accumulators before the multiply-adds so that its latency
// overlaps the staging.
constexpr int kMaxPanel = 32;
constexpr int kUpdTile = 80;
__global__ void __launch_bounds__(256) k_gj_update32(int n, int k0, int w, int nb,
                                                     const cx<float>* U, const cx<float>* srcs,
                                                     cx<float>* dsts, const int32_t* conts,
                                                     const int32_t* active) {
  chain_next();
  chain_wait();
  const int p = blockIdx.z;
  if (active && !active[p]) return;
  __shared__ cx<float> Us[kUpdTile][kMaxPanel + 1];  // row-major like U; padded rows
  __shared__ cx<float> Ts[kMaxPanel][kUpdTile];
  const int m0 = blockIdx.y * kUpdTile, n0 = blockIdx.x * kUpdTile;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const long long nn = (long long)n * n;
  const cx<float>* u = U + (long long)p * n * nb;
  const cx<float>* src = srcs + p * nn;
  cx<float>* dst = dsts + p * nn;
  const int32_t* cont = conts + (long long)p * n;
  const cx<float> zero = mkc<float>(0.0f, 0.0f);
  cx<float> acc[5][5];
#pragma unroll
  for (int i = 0; i < 5; ++i) {
    const int r = m0 + ty + 16 * i;
    const bool keep = r < n && (r < k0 || r >= k0 + w);
    const cx<float>* row = src + (long long)(keep ? cont[r] : 0) * n;
#pragma unroll
    for (int j = 0; j < 5; ++j) {
      const int col = n0 + tx + 16 * j;
      acc[i][j] = (keep && col < n) ? row[col] : zero;
    }
  }
  // staging: slot e of U is (row e / 32, column e % 32), of T (row e / 80, column e % 80); all
  // loads are issued before the first shared-memory store
  constexpr int kPer = kMaxPanel * kUpdTile / 256;  // 10
  cx<float> us[kPer], ts[kPer];
#pragma unroll
  for (int q = 0; q < kPer; ++q) {
    const int e = threadIdx.x + 256 * q;
    const int r = e >> 5, k = e & 31;
    us[q] = (k < w && m0 + r < n) ? u[(long long)(m0 + r) * nb + k] : zero;
  }
#pragma unroll
  for (int q = 0; q < kPer; ++q) {
    const int e = threadIdx.x + 256 * q;
    const int k = e / kUpdTile, col = e % kUpdTile;
    ts[q] = (k < w && n0 + col < n) ? src[(long long)cont[k0 + k] * n + n0 + col] : zero;
  }
#pragma unroll
  for (int q = 0; q < kPer; ++q) {
    const int e = threadIdx.x + 256 * q;
    Us[e >> 5][e & 31] = us[q];
    Ts[e / kUpdTile][e % kUpdTile] = ts[q];
  }
  __syncthreads();
  for (int k = 0; k < w; ++k) {
    cx<float> av[5], bv[5];
#pragma unroll
    for (int i = 0; i < 5; ++i) av[i] = Us[ty + 16 * i][k];
#pragma unroll
    for (int j = 0; j < 5; ++j) bv[j] = Ts[k][tx + 16 * j];
#pragma unroll
    for (int i = 0; i < 5; ++i)
#pragma unroll
      for (int j = 0; j < 5; ++j) cfma(acc[i][j], av[i], bv[j]);
  }
#pragma unroll
  for (int i = 0; i < 5; ++i)
#pragma unroll
    for (int j = 0; j < 5; ++j) {
      const int r = m0 + ty + 16 * i, col = n0 + tx + 16 * j;
      if (r < n && col < n && (col < k0 || col >= k0 + w)) dst[(long long)r * n + col] = acc[i][j];
    }
}

// The same update for panels of at most four columns (blocks beyond 2425), which memory bounds: one
// read and one write of the matrix for four complex multiply-adds per element.  No tile is worth
// staging there; a thread keeps its 2 x 8 elements (rows of a warp, columns 32 apart) and the pivot
// rows of its columns in registers, so that 16 loads per thread are under way.  The sums are those of
// k_gj_update32, in its order.  n = 3430: two slabs solved in 345 ms with the tiles, 325 with this kernel (the tiles
// took 48 us per update, 3.9 TB/s); at n = 2400, eight columns, the tiles are faster (31.6 ms against
// 32.3 for an inverse).
constexpr int kThinPanel = 4, kThinRows = 8, kThinCols = 64, kThinWarps = 8;
__global__ void __launch_bounds__(32 * kThinWarps)
    k_gj_update_thin(int n, int k0, int w, int nb, const cx<float>* U, const cx<float>* srcs,
                     cx<float>* dsts, const int32_t* conts, const int32_t* active) {
  chain_next();
  chain_wait();
  const int p = blockIdx.z;
  if (active && !active[p]) return;
  __shared__ cx<float> Us[kThinWarps * kThinRows][kThinPanel];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int m0 = blockIdx.y * kThinWarps * kThinRows, n0 = blockIdx.x * kThinCols + lane;
  const long long nn = (long long)n * n;
  const cx<float>* u = U + (long long)p * n * nb;
  const cx<float>* src = srcs + p * nn;
  cx<float>* dst = dsts + p * nn;
  const int32_t* cont = conts + (long long)p * n;
  const cx<float> zero = mkc<float>(0.0f, 0.0f);
  cx<float> acc[kThinRows][2], t[kThinPanel][2];
#pragma unroll
  for (int i = 0; i < kThinRows; ++i) {
    const int r = m0 + wid * kThinRows + i;
    const bool keep = r < n && (r < k0 || r >= k0 + w);
    const cx<float>* row = src + (long long)(keep ? cont[r] : 0) * n;
#pragma unroll
    for (int j = 0; j < 2; ++j) acc[i][j] = keep && n0 + 32 * j < n ? row[n0 + 32 * j] : zero;
  }
#pragma unroll
  for (int k = 0; k < kThinPanel; ++k) {
    const cx<float>* row = src + (long long)(k < w ? cont[k0 + k] : 0) * n;
#pragma unroll
    for (int j = 0; j < 2; ++j) t[k][j] = k < w && n0 + 32 * j < n ? row[n0 + 32 * j] : zero;
  }
  for (int e = threadIdx.x; e < kThinWarps * kThinRows * kThinPanel; e += 32 * kThinWarps) {
    const int r = m0 + e / kThinPanel, k = e % kThinPanel;
    Us[e / kThinPanel][k] = r < n && k < w ? u[(long long)r * nb + k] : zero;
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < kThinPanel; ++k) {
    if (k >= w) break;
#pragma unroll
    for (int i = 0; i < kThinRows; ++i)
#pragma unroll
      for (int j = 0; j < 2; ++j) cfma(acc[i][j], Us[wid * kThinRows + i][k], t[k][j]);
  }
#pragma unroll
  for (int i = 0; i < kThinRows; ++i)
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int r = m0 + wid * kThinRows + i, col = n0 + 32 * j;
      if (r < n && col < n && (col < k0 || col >= k0 + w)) dst[(long long)r * n + col] = acc[i][j];
    }
}

// Column permutation that the pivoting left: column c of the inverse is column map[c] of the
// eliminated matrix.  A chain of exchanges, so one thread per item follows it in shared memory.
__global__ void __launch_bounds__(kThreads) k_gj_perm(int n, const int32_t* piv, int32_t* map,
                                                      const int32_t* active) {
  const int p = blockIdx.x;
  if (active && !active[p]) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  int* src = reinterpret_cast<int*>(smem_raw);
  int* pv = src + n;
  for (int c = threadIdx.x; c < n; c += blockDim.x) {
    src[c] = c;
    pv[c] = piv[(long long)p * n + c];
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int j = n - 1; j >= 0; --j) {
      const int q = pv[j], t = src[j];
      src[j] = src[q];
      src[q] = t;
    }
  }
  __syncthreads();
  for (int c = threadIdx.x; c < n; c += blockDim.x) map[(long long)p * n + c] = src[c];
}

// X = the columns of A in their final order (A and X may differ in precision), one row at a time
// per CTA through all CTAs of an item.
template <typename RA, typename RX>
__global__ void __launch_bounds__(kThreads) k_gj_columns(int n, BMc<RA> Am, BM<RX> Xm,
                                                         const int32_t* map,
                                                         const int32_t* active) {
  const int p = blockIdx.y;
  if (active && !active[p]) return;
  const cx<RA>* a = bat(Am, p);
  cx<RX>* x = bat(Xm, p);
  const int32_t* m = map + (long long)p * n;
  for (int r = blockIdx.x; r < n; r += gridDim.x)
    for (int c = threadIdx.x; c < n; c += blockDim.x) {
      const cx<RA> v = a[(long long)r * Am.ld + m[c]];
      x[(long long)r * Xm.ld + c] = mkc<RX>((RX)v.re, (RX)v.im);
    }
}

// X = A and a change of precision (the one-CTA form's input and output)
template <typename RA, typename RX>
__global__ void __launch_bounds__(kThreads) k_convert(long long n, const cx<RA>* a, cx<RX>* x,
                                                      const int32_t* active, long long per) {
  for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < n;
       k += (long long)gridDim.x * blockDim.x) {
    if (active && !active[k / per]) continue;
    x[k] = mkc<RX>((RX)a[k].re, (RX)a[k].im);
  }
}
inline unsigned convert_blocks(long long n) {
  const long long b = (n + kThreads - 1) / kThreads;
  return (unsigned)(b > 152 * 32 ? 152 * 32 : (b < 1 ? 1 : b));
}

}  // namespace

static size_t small_smem(int n, int elem_bytes) {
  return (size_t)n * n * elem_bytes + 2 * (size_t)n * elem_bytes + 2 * n * sizeof(int);
}
static size_t panel_smem(int n, int w, int elem_bytes) {
  return (size_t)n * w * elem_bytes + (size_t)n * elem_bytes + (size_t)w * elem_bytes +
         (size_t)(n + w) * sizeof(int);
}

bool gj_fits_small(int n, int elem_bytes) { return small_smem(n, elem_bytes) <= kSmemBudget; }

bool gj_supports(int n, int elem_bytes) {
  // the panel kernel holds n x nb panel values, the pivot column and the row map in shared
  // memory (nb = 1 at worst), and the final unpermutation n row indices
  if (n < 1) return false;
  if (gj_fits_small(n, elem_bytes)) return true;
  return panel_smem(n, gj_panel_width(n, elem_bytes), elem_bytes) <= kSmemBudget + 1024 &&
         (size_t)n * sizeof(int) <= 48 * 1024;
}


int gj_panel_width(int n, int elem_bytes) {
  size_t per_col = (size_t)n * elem_bytes + elem_bytes + sizeof(int);
  size_t fixed = (size_t)n * (elem_bytes + sizeof(int));
  int w = fixed >= kSmemBudget ? 1 : (int)std::min<size_t>(32, (kSmemBudget - fixed) / per_col);
  int p2 = 1;
  while (p2 * 2 <= w) p2 *= 2;
  return std::max(1, p2);
}

namespace {
template <typename RA, typename RX>
cudaError_t columns(cudaStream_t s, int P, int n, BMc<RA> A, BM<RX> X, const int32_t* piv,
                    int32_t* map, const int32_t* active) {
  static std::atomic<unsigned> attr{0};
  cudaError_t e = set_smem_once(attr, reinterpret_cast<const void*>(&k_gj_perm), 96 * 1024);
  if (e != cudaSuccess) return e;
  k_gj_perm<<<P, kThreads, 2 * (size_t)n * sizeof(int), s>>>(n, piv, map, active);
  k_gj_columns<RA, RX><<<dim3(std::min(n, 128), P), kThreads, 0, s>>>(n, A, X, map, active);
  count_launch(2);
  return cudaGetLastError();
}

template <int W, int NR, bool LAST>
cudaError_t panel32(cudaStream_t s, int P, int n, int k0, int w, int nb, const cx<float>* src,
                    cx<float>* dst, cx<float>* U, int32_t* piv, int32_t* cont, int32_t* status,
                    const int32_t* active) {
  static std::atomic<unsigned> attr{0};
  auto* fn = &k_gj_panel32<W, NR, LAST>;
  cudaError_t e = set_smem_once(attr, reinterpret_cast<const void*>(fn), 220 * 1024);
  if (e != cudaSuccess) return e;
  const size_t smem = 2 * (size_t)NR * (kPanelThreads / W) * sizeof(cx<float>) + n * sizeof(int);
  count_launch();
  return launch_chained(fn, dim3(P), dim3(kPanelThreads), smem, s, n, k0, w, nb, src, dst, U, piv,
                        cont, status, active);
}

// The panel kernel of width nb, by the rows a thread holds (gj_panel_width keeps n nb <= 22528, so
// n / kG + 1 <= 45; at nb = 1, n <= 9266 and 19).
cudaError_t panel32(cudaStream_t s, int P, int n, int k0, int w, int nb, const cx<float>* src,
                    cx<float>* dst, cx<float>* U, int32_t* piv, int32_t* cont, int32_t* status,
                    const int32_t* active) {
#define NEGF_PANEL_ARGS s, P, n, k0, w, nb, src, dst, U, piv, cont, status, active
#define NEGF_PANEL(W_)                                                              \
  case W_:                                                                          \
    if (w < W_) return panel32<W_, 45, true>(NEGF_PANEL_ARGS);                      \
    if (n * nb < 14 * kPanelThreads) return panel32<W_, 14, false>(NEGF_PANEL_ARGS); \
    if (n * nb < 28 * kPanelThreads) return panel32<W_, 28, false>(NEGF_PANEL_ARGS); \
    return panel32<W_, 45, false>(NEGF_PANEL_ARGS)
  switch (nb) {
    NEGF_PANEL(32);
    NEGF_PANEL(16);
    NEGF_PANEL(8);
    NEGF_PANEL(4);
    NEGF_PANEL(2);
    case 1: return panel32<1, 19, false>(NEGF_PANEL_ARGS);
  }
#undef NEGF_PANEL
#undef NEGF_PANEL_ARGS
  return cudaErrorInvalidValue;
}
}  // namespace

// Both eliminations are chains of two short kernels per panel, and the mixed form's FP64 fallback runs
// its whole chain without an item in nearly every call: the kernels are launched chained, which took
// the inverse of one 400 block (mixed) from 1782 to 1586 us, of one 2400 block from 39.5 to 31.6 ms, of 64
// blocks of 400 from 5.57 to 5.44 ms.  The update is a chained product by strips there; with items to
// work on it is one by tiles, not chained (64 FP64 blocks of 400: 45.0 ms, 48.7 chained, 50.5 by strips).
cudaError_t gj_inverse64(cudaStream_t s, int P, int n, BM<double> M, BM<double> X, z64* U, z64* T,
                         int32_t* piv, int32_t* status, const int32_t* active, bool mostly_idle) {
  if (P <= 0 || n <= 0) return cudaSuccess;
  const int eb = (int)sizeof(z64);
  if (gj_fits_small(n, eb)) {
    cudaError_t e = cudaFuncSetAttribute(
        k_gj_small64, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemBudget + 1024);
    if (e != cudaSuccess) return e;
    k_gj_small64<<<P, kThreads, small_smem(n, eb), s>>>(n, M, X, status, active);
    count_launch();
    return cudaGetLastError();
  }
  const int nb = gj_panel_width(n, eb);
  cudaError_t e = cudaFuncSetAttribute(k_gj_panel<double>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)kSmemBudget + 1024);
  if (e != cudaSuccess) return e;
  for (int k0 = 0; k0 < n; k0 += nb) {
    const int w = std::min(nb, n - k0);
    size_t smem = panel_smem(n, w, eb);
    prof_begin(s, PROF_GJ_PANEL);
    e = launch_chained(&k_gj_panel<double>, dim3(P), dim3(kThreads), smem, s, n, k0, w, nb, M, U, T,
                       piv, status, active);
    prof_end(s, PROF_GJ_PANEL);
    count_launch();
    if (e != cudaSuccess) return e;
    BMc<double> Ua{U, (long long)n * nb, nullptr, nb};
    BMc<double> Ta{T, (long long)nb * n, nullptr, n};
    BMc<double> none{nullptr, 0, nullptr, 0};
    e = gemm_simt(s, P, n, n, w, mkc<double>(1.0, 0.0), Ua, OP_N, Ta, OP_N, mkc<double>(1.0, 0.0),
                  M, mkc<double>(0.0, 0.0), none, active, mostly_idle ? GEMM_STRIPS : GEMM_TILES);
    if (e != cudaSuccess) return e;
  }
  // T is free again
  return columns<double, double>(s, P, n, cst(M), X, piv, reinterpret_cast<int32_t*>(T), active);
}

cudaError_t gj_inverse32(cudaStream_t s, int P, int n, BM<double> M, BM<double> X, cx<float>* m32,
                         cx<float>* x32, cx<float>* U, int32_t* piv, int32_t* map, int32_t* status,
                         const int32_t* active) {
  if (P <= 0 || n <= 0) return cudaSuccess;
  const int eb = (int)sizeof(cx<float>);
  const long long nn = (long long)n * n, tot = P * nn;
  k_convert<double, float><<<convert_blocks(tot), kThreads, 0, s>>>(tot, M.p, m32, active, nn);
  count_launch();
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  if (gj_fits_small(n, eb)) {
    e = cudaFuncSetAttribute(k_gj_small<float>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)kSmemBudget + 1024);
    if (e != cudaSuccess) return e;
    k_gj_small<float><<<P, kThreads, small_smem(n, eb), s>>>(
        n, BM<float>{m32, nn, nullptr, n}, BM<float>{x32, nn, nullptr, n}, status, active);
    k_convert<float, double><<<convert_blocks(tot), kThreads, 0, s>>>(tot, x32, X.p, active, nn);
    count_launch(2);
    return cudaGetLastError();
  }
  const int nb = gj_panel_width(n, eb);
  cx<float>*src = m32, *dst = x32;
  const dim3 grid((n + kUpdTile - 1) / kUpdTile, (n + kUpdTile - 1) / kUpdTile, P);
  for (int k0 = 0; k0 < n; k0 += nb) {
    const int w = std::min(nb, n - k0);
    prof_begin(s, PROF_GJ_PANEL);
    e = panel32(s, P, n, k0, w, nb, src, dst, U, piv, map, status, active);
    prof_end(s, PROF_GJ_PANEL);
    if (e != cudaSuccess) return e;
    if (nb <= kThinPanel) {
      constexpr int kRows = kThinWarps * kThinRows;
      const dim3 thin((n + kThinCols - 1) / kThinCols, (n + kRows - 1) / kRows, P);
      e = launch_chained(&k_gj_update_thin, thin, dim3(32 * kThinWarps), 0, s, n, k0, w, nb, U,
                         src, dst, map, active);
    } else {
      e = launch_chained(&k_gj_update32, grid, dim3(256), 0, s, n, k0, w, nb, U, src, dst, map,
                         active);
    }
    count_launch();
    if (e != cudaSuccess) return e;
    std::swap(src, dst);
  }
  return columns<float, double>(s, P, n, BMc<float>{src, nn, nullptr, n}, X, piv, map, active);
}

}  // namespace negf
