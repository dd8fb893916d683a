// Batched complex GEMM on the CUDA cores.  This is the arithmetic of the plain FP64 form of
// the recursive Green's function sweeps (Eqs. 1-2 evaluated block by block): every product
// of two b x b blocks of G, g, H or Sigma goes through here when precision == FP64.
#include <algorithm>

#include "common.cuh"
#include "profile.cuh"

namespace negf {

namespace {
constexpr int BMT = 64;  // tile rows
constexpr int BNT = 64;  // tile cols
constexpr int BKT = 8;   // k chunk
constexpr int TY = 16, TX = 16;  // 256 threads, 4 x 4 outputs each

__device__ __forceinline__ z64 load_op(const z64* a, int ld, int op, int r, int c, int rows,
                                         int cols) {
  // element (r, c) of op(A) where op(A) has shape rows x cols
  if (r >= rows || c >= cols) return mkc(0.0, 0.0);
  if (op == OP_N) return a[(long long)r * ld + c];
  z64 v = a[(long long)c * ld + r];
  if (op == OP_C) v.im = -v.im;
  return v;
}

__global__ void __launch_bounds__(256) k_gemm_simt(int M, int N, int K, z64 alpha, BMc<double> A,
                                                   int opA, BMc<double> B, int opB, z64 beta, BM<double> C,
                                                   z64 gamma, BMc<double> D,
                                                   const int32_t* active) {
  const int p = blockIdx.z;
  if (active && !active[p]) return;
  __shared__ z64 As[BKT][BMT];
  __shared__ z64 Bs[BKT][BNT];
  const z64* a = bat(A, p);
  const z64* b = bat(B, p);
  const int m0 = blockIdx.y * BMT, n0 = blockIdx.x * BNT;
  const int tx = threadIdx.x % TX, ty = threadIdx.x / TX;
  z64 acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = mkc(0.0, 0.0);

  for (int k0 = 0; k0 < K; k0 += BKT) {
    // 512 elements of each tile, 2 per thread
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      int id = threadIdx.x + e * 256;
      // A tile: (m, k) -> As[k][m]; walk m fastest for op T/C coalescing, k fastest for N
      int mm, kk;
      if (opA == OP_N) {
        kk = id % BKT;
        mm = id / BKT;
      } else {
        mm = id % BMT;
        kk = id / BMT;
      }
      As[kk][mm] = load_op(a, A.ld, opA, m0 + mm, k0 + kk, M, K);
      int nn, kb;
      if (opB == OP_N) {
        nn = id % BNT;
        kb = id / BNT;
      } else {
        kb = id % BKT;
        nn = id / BKT;
      }
      Bs[kb][nn] = load_op(b, B.ld, opB, k0 + kb, n0 + nn, K, N);
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < BKT; ++kk) {
      z64 av[4], bv[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) av[i] = As[kk][ty + TY * i];
#pragma unroll
      for (int j = 0; j < 4; ++j) bv[j] = Bs[kk][tx + TX * j];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) cfma(acc[i][j], av[i], bv[j]);
    }
    __syncthreads();
  }
  z64* c = bat(C, p);
  const z64* d = D.p ? bat(D, p) : nullptr;
  const bool use_beta = (beta.re != 0.0 || beta.im != 0.0);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    int r = m0 + ty + TY * i;
    if (r >= M) continue;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      int col = n0 + tx + TX * j;
      if (col >= N) continue;
      z64 v = alpha * acc[i][j];
      z64* cp = c + (long long)r * C.ld + col;
      if (use_beta) v = v + beta * (*cp);
      if (d) v = v + gamma * d[(long long)r * D.ld + col];
      *cp = v;
    }
  }
}

// Products by strips: one warp per 4 rows x 8 columns, lane (y, x) holding row y and column x.  FP64
// issues two lanes per clock and SM here, so the four multiply-adds per lane and k step that a warp
// does take 256 clocks of its scheduler while their operands are 192 bytes: the caches serve them
// without staging, at any size, and what counts is that the work is split evenly and that loads are
// on their way kStripAhead steps before.  128 x 128 x 128, 512 items: 7.18 ms, 1.95 FP64
// multiply-adds per clock and SM at 1.9 GHz, like the tiles above.  Larger pieces per warp (1 x 2,
// 2 x 1 to 4 x 2 elements per lane) took 1.2 to 1.4 times as long at every size.
constexpr int kStripRows = 4, kStripCols = 8, kStripWarps = 4, kStripAhead = 4;
__global__ void __launch_bounds__(32 * kStripWarps)
    k_gemm_strip(int M, int N, int K, z64 alpha, BMc<double> A, int opA, BMc<double> B, int opB,
                 z64 beta, BM<double> C, z64 gamma, BMc<double> D, const int32_t* active) {
  chain_next();
  chain_wait();
  const int p = blockIdx.y;
  if (active && !active[p]) return;
  const int lane = threadIdx.x & 31;
  const long long cols = (N + kStripCols - 1) / kStripCols;
  const long long strips = (M + kStripRows - 1) / kStripRows * cols;
  const z64 *ap = bat(A, p), *bp = bat(B, p);
  // op(A)[r][k] and op(B)[k][c] as base + k * step
  const long long sa = opA == OP_N ? 1 : A.ld, sb = opB == OP_N ? B.ld : 1;
  const bool use_beta = (beta.re != 0.0 || beta.im != 0.0);
  for (long long strip = blockIdx.x * kStripWarps + (threadIdx.x >> 5); strip < strips;
       strip += gridDim.x * kStripWarps) {
    const int r = (int)(strip / cols) * kStripRows + (lane >> 3);
    const int c = (int)(strip % cols) * kStripCols + (lane & 7);
    // rows and columns beyond the edge read the last one
    const long long ra = r < M ? r : M - 1, cb = c < N ? c : N - 1;
    const z64* a = ap + (opA == OP_N ? ra * A.ld : ra);
    const z64* b = bp + (opB == OP_N ? cb : cb * B.ld);
    z64 acc = mkc(0.0, 0.0);
    struct Step {
      z64 a, b;
    };
    auto load = [&](Step (&t)[kStripAhead], int k0) {
#pragma unroll
      for (int u = 0; u < kStripAhead; ++u) {
        const long long k = k0 + u < K ? k0 + u : K - 1;
        t[u].a = a[k * sa];
        t[u].b = b[k * sb];
      }
    };
    auto step = [&](Step (&t)[kStripAhead], int k0) {
#pragma unroll
      for (int u = 0; u < kStripAhead; ++u) {
        if (k0 + u >= K) break;
        t[u].a.im = opA == OP_C ? -t[u].a.im : t[u].a.im;
        t[u].b.im = opB == OP_C ? -t[u].b.im : t[u].b.im;
        cfma(acc, t[u].a, t[u].b);
      }
    };
    Step t0[kStripAhead], t1[kStripAhead];  // one being used, one on its way
    load(t0, 0);
    for (int k = 0; k < K; k += 2 * kStripAhead) {
      load(t1, k + kStripAhead);
      step(t0, k);
      if (k + kStripAhead >= K) break;
      load(t0, k + 2 * kStripAhead);
      step(t1, k + kStripAhead);
    }
    if (r >= M || c >= N) continue;
    z64* out = bat(C, p) + (long long)r * C.ld + c;
    z64 v = alpha * acc;
    if (use_beta) v = v + beta * *out;
    if (D.p) v = v + gamma * bat(D, p)[(long long)r * D.ld + c];
    *out = v;
  }
}

}  // namespace

cudaError_t gemm_simt(cudaStream_t s, int P, int M, int N, int K, z64 alpha, BMc<double> A,
                      int opA, BMc<double> B, int opB, z64 beta, BM<double> C, z64 gamma,
                      BMc<double> D, const int32_t* active, int form) {
  if (P <= 0 || M <= 0 || N <= 0) return cudaSuccess;
  // Tiles run at the FP64 rate of an SM each, 64 x 64 x 4 multiply-adds per k step at two per clock, in
  // waves of one per SM: 8192 clocks per k and wave.  Strips split evenly but reach 72 % of the rate.
  // Measured, us, strips / tiles: 64 items of 40 36 / 166, 1 of 400 673 / 1686, 64 of 200 3380 / 5602, 3
  // of 64 x 1000 x 500 1078 / 2107, 200 of 64 x 64 x 300 2245 / 2519; 64 of 128 1248 / 1090, 64 of 256
  // 9503 / 7226, 64 of 400 36089 / 33482, 1 of 1200 15365 / 14448.  Both form the same sums.
  // Strips write their output while others still read: an output that starts on an operand goes to
  // the tiles (right for it up to one tile), as does K = 0.
  constexpr long long kSms = 152;
  const long long tiles = (long long)((M + BMT - 1) / BMT) * ((N + BNT - 1) / BNT) * P;
  const double tile_clocks = 8192.0 * ((tiles + kSms - 1) / kSms);
  const double strip_clocks = 2.0 / 0.72 / kSms * P * ((M + kStripRows - 1) / kStripRows * kStripRows) *
                              ((N + kStripCols - 1) / kStripCols * kStripCols);
  const bool strips = form == GEMM_AUTO ? strip_clocks < tile_clocks : form == GEMM_STRIPS;
  if (strips && K > 0 && C.p != A.p && C.p != B.p) {
    const long long strips =
        (long long)((M + kStripRows - 1) / kStripRows) * ((N + kStripCols - 1) / kStripCols);
    // CTAs per item: enough to fill the chip, few enough that masked items cost little
    const long long most = std::max(64ll, 152ll * 8 / P);
    const unsigned ctas = (unsigned)std::min(most, (strips + kStripWarps - 1) / kStripWarps);
    count_launch();
    return launch_chained(&k_gemm_strip, dim3(ctas, P), dim3(32 * kStripWarps), 0, s, M, N, K,
                          alpha, A, opA, B, opB, beta, C, gamma, D, active);
  }
  const dim3 grid((N + BNT - 1) / BNT, (M + BMT - 1) / BMT, P);
  k_gemm_simt<<<grid, 256, 0, s>>>(M, N, K, alpha, A, opA, B, opB, beta, C, gamma, D, active);
  count_launch();
  return cudaGetLastError();
}

}  // namespace negf
