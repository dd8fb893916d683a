// Shared device/host helpers of the RGF library: complex arithmetic, batched operand
// descriptors and the internal launcher declarations.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "negf.h"

namespace negf {

template <typename R>
struct cx {
  R re, im;
};
using z64 = cx<double>;

template <typename R>
__host__ __device__ __forceinline__ cx<R> mkc(R a, R b) {
  cx<R> z;
  z.re = a;
  z.im = b;
  return z;
}
template <typename R>
__host__ __device__ __forceinline__ cx<R> operator+(cx<R> a, cx<R> b) {
  return mkc<R>(a.re + b.re, a.im + b.im);
}
template <typename R>
__host__ __device__ __forceinline__ cx<R> operator-(cx<R> a, cx<R> b) {
  return mkc<R>(a.re - b.re, a.im - b.im);
}
template <typename R>
__host__ __device__ __forceinline__ cx<R> operator*(cx<R> a, cx<R> b) {
  return mkc<R>(a.re * b.re - a.im * b.im, a.re * b.im + a.im * b.re);
}
template <typename R>
__host__ __device__ __forceinline__ cx<R> operator*(R s, cx<R> a) {
  return mkc<R>(s * a.re, s * a.im);
}
template <typename R>
__host__ __device__ __forceinline__ cx<R> conjc(cx<R> a) {
  return mkc<R>(a.re, -a.im);
}
// acc += a * b with fused multiply-adds
template <typename R>
__device__ __forceinline__ void cfma(cx<R>& acc, cx<R> a, cx<R> b) {
  acc.re = fma(a.re, b.re, acc.re);
  acc.re = fma(-a.im, b.im, acc.re);
  acc.im = fma(a.re, b.im, acc.im);
  acc.im = fma(a.im, b.re, acc.im);
}
// 1 / a in double precision (Smith's method avoids overflow of |a|^2)
__host__ __device__ __forceinline__ z64 crecip(z64 a) {
  double r, d;
  if (fabs(a.re) >= fabs(a.im)) {
    r = a.im / a.re;
    d = a.re + a.im * r;
    return mkc<double>(1.0 / d, -r / d);
  }
  r = a.re / a.im;
  d = a.re * r + a.im;
  return mkc<double>(r / d, -1.0 / d);
}

enum Op { OP_N = 0, OP_T = 1, OP_C = 2 };

// Batched matrix operand: batch item p lives at p_base + (idx ? idx[p] : p) * stride, and
// element (r, c) at + r * ld + c (row-major).  stride 0 with idx NULL means "shared".
template <typename R>
struct BM {
  cx<R>* p;
  long long stride;
  const int32_t* idx;
  int ld;
};
template <typename R>
struct BMc {
  const cx<R>* p;
  long long stride;
  const int32_t* idx;
  int ld;
};
template <typename R>
__host__ __device__ __forceinline__ BMc<R> cst(BM<R> a) {
  BMc<R> b;
  b.p = a.p;
  b.stride = a.stride;
  b.idx = a.idx;
  b.ld = a.ld;
  return b;
}
template <typename R>
__device__ __forceinline__ const cx<R>* bat(BMc<R> a, int p) {
  return a.p + (a.idx ? (long long)a.idx[p] : (long long)p) * a.stride;
}
template <typename R>
__device__ __forceinline__ cx<R>* bat(BM<R> a, int p) {
  return a.p + (a.idx ? (long long)a.idx[p] : (long long)p) * a.stride;
}

// Chains of short kernels: a kernel launched by launch_chained may be set up while the one before it
// on the stream still runs (once all of that one's CTAs have started and called chain_next), and
// waits in chain_wait, first thing, until it has finished with its writes visible.
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void chain_next() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
template <class... P, class... A>
inline cudaError_t launch_chained(void (*fn)(P...), dim3 grid, dim3 block, size_t smem,
                                  cudaStream_t s, A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, fn, static_cast<P>(args)...);
  return e != cudaSuccess ? e : cudaGetLastError();
}

// ---- launchers (all asynchronous on `s`) ----------------------------------------------

// Form of an FP64 product: chosen by size, or given.
enum GemmForm { GEMM_AUTO = 0, GEMM_TILES = 1, GEMM_STRIPS = 2 };
// C[p] = alpha op(A[p]) op(B[p]) + beta C[p] + gamma D[p] on the CUDA cores (FP64 form).
// beta == 0 does not read C; D.p == NULL skips the D term.  Batch items with
// active[p] == 0 are skipped (active may be NULL).
cudaError_t gemm_simt(cudaStream_t s, int P, int M, int N, int K, z64 alpha, BMc<double> A,
                      int opA, BMc<double> B, int opB, z64 beta, BM<double> C, z64 gamma,
                      BMc<double> D, const int32_t* active, int form = GEMM_AUTO);

// X[p] = M[p]^-1 by Gauss-Jordan elimination with partial pivoting (largest |m|, lowest row
// on ties, pivots compared in FP64).  A zero pivot sets NEGF_PT_SINGULAR in status[p] and is
// replaced by a tiny number so the sweep continues.  Scratch: piv (P x n).
// FP64: mostly_idle: active is expected to select no item.  M is destroyed; scratch U (P x n x nb), T (P x nb x n), nb = gj_panel_width(n, 16).
// FP32: elimination in FP32 (m32 and x32: P x n x n, U: P x n x nb, nb = gj_panel_width(n, 8), map:
// P x n), M is kept; M and X are contiguous n x n blocks.
cudaError_t gj_inverse64(cudaStream_t s, int P, int n, BM<double> M, BM<double> X, z64* U, z64* T,
                         int32_t* piv, int32_t* status, const int32_t* active,
                         bool mostly_idle = false);
cudaError_t gj_inverse32(cudaStream_t s, int P, int n, BM<double> M, BM<double> X, cx<float>* m32,
                         cx<float>* x32, cx<float>* U, int32_t* piv, int32_t* map, int32_t* status,
                         const int32_t* active);
int gj_panel_width(int n, int elem_bytes);
bool gj_fits_small(int n, int elem_bytes);
// Whether the batched Gauss-Jordan inverse launches for n x n blocks of elem_bytes complex
// elements (shared-memory limits: n <= 9266 for FP32, n <= 5147 for FP64 elements).
bool gj_supports(int n, int elem_bytes);

}  // namespace negf
