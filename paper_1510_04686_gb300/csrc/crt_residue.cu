// Operand residue kernels of the tensor-core complex GEMM (see crt_residue.cuh, crt_plan.cuh).
#include <cmath>

#include "f32x2.cuh"
#include "crt_residue.cuh"

namespace negf {
namespace {

// ------------------------------------------------------------------ line norm
// Sum of squares of |x| relative to 2^ex, ex the largest biased exponent so far.  The leading 20
// mantissa bits are used (truncated; scale_of allows for it), a subnormal value counts as the next
// larger number with an implicit bit.
struct Norm {
  int ex;
  float s;
};
__device__ __forceinline__ float pow2m(int d) {  // 2^-d, 0 <= d; 0 beyond FP32's range
  return d > 126 ? 0.0f : __int_as_float((127 - d) << 23);
}
// n complex values at once: one test for a larger exponent, and the FP32 value of each mantissa and
// relative exponent by a shift and a subtraction of the high word.
template <int n>
__device__ __forceinline__ void norm_add(Norm& nm, const z64* v) {
  int h[2 * n], top = 1 << 20;
#pragma unroll
  for (int i = 0; i < 2 * n; ++i) {
    const double x = i & 1 ? v[i / 2].im : v[i / 2].re;
    h[i] = (__double2hiint(x) & 0x7FFFFFFF) | (int)min((unsigned)__double2loint(x), 1u);
    top = max(top, h[i]);
  }
  top >>= 20;
  if (top > nm.ex) {
    nm.s *= pow2m(2 * (top - nm.ex));
    nm.ex = top;
  }
  const int low = max((nm.ex - 126) << 20, 1);  // below: zero, or nothing next to 2^ex
  const unsigned off = (unsigned)(nm.ex - 127) << 23;
#pragma unroll
  for (int i = 0; i < 2 * n; ++i) {
    const float f = h[i] >= low ? __uint_as_float(((unsigned)h[i] << 3) - off) : 0.0f;
    nm.s = fmaf(f, f, nm.s);
  }
}
__device__ __forceinline__ void norm_merge(Norm& n, int oe, float os) {
  const int e = max(n.ex, oe);
  n.s = n.s * pow2m(2 * (e - n.ex)) + os * pow2m(2 * (e - oe));
  n.ex = e;
}
__device__ __forceinline__ Norm norm_warp(Norm n) {
  for (int o = 16; o > 0; o >>= 1)
    norm_merge(n, __shfl_xor_sync(0xffffffffu, n.ex, o), __shfl_xor_sync(0xffffffffu, n.s, o));
  return n;
}
// Exponent e with sigma 2-norm 2^e < 2^alpha for the line; kNonFinite when it holds an infinity or
// NaN.
__device__ __forceinline__ int scale_of(Norm n, int alpha, float sigma2) {
  if (n.ex >= 0x7FF) return kNonFinite;
  if (!(n.s > 0.0f)) return 0;
  // truncated mantissas and the FP32 sum make s at most 2^-8 too small in relative terms
  int x;
  frexpf(n.s * sigma2 * 1.00390625f, &x);  // norm < 2^(x / 2 + ex - 1023)
  return alpha - ((x + 1) >> 1) - (n.ex - 1023);
}

// ------------------------------------------------------------------ residues
// round(sigma x 2^e) plus 128 in every digit position, so that byte i of the result is the balanced
// digit i plus 128.  sig = sigma 2^64 (0: sigma is one).  flip: 0x80000000 changes the sign of x.
// The scaled line's norm is below 2^alpha, alpha <= 60, so |sigma x 2^e| is the mantissa, aligned to
// the top of 64 bits, shifted right by three or more; 64 and beyond leave nothing.
__device__ __forceinline__ unsigned long long biased(double x, int e, unsigned flip,
                                                     unsigned long long sig) {
  constexpr unsigned long long kBias = 0x8080808080808080ull;
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const int ex = (int)((hi >> 20) & 0x7FF);
  const unsigned mh = (hi & 0xFFFFFu) | (ex ? 0x100000u : 0u);
  unsigned long long m =
      (unsigned long long)__funnelshift_l(lo, mh, 11) << 32 | (unsigned long long)(lo << 11);
  if (sig) m = __umul64hi(m, sig);
  unsigned long long r;  // a shift by 64 or more gives zero
  asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(m), "r"((unsigned)(1085 - max(ex, 1) - e)));
  r = (r + 1) >> 1;
  const long long neg = (long long)((int)(hi ^ flip) >> 31);  // 0 or -1
  return (r ^ (unsigned long long)neg) + (kBias - (unsigned long long)neg);
}
// Digits 2 t and 2 t + 1 of a biased value as a BF16 pair; sel = the byte selector of t.  A byte b
// is (128 + its low seven bits, exact with the exponent of 128) - (128 or 256 by its top bit).
__device__ __forceinline__ uint32_t digit_pair(unsigned long long v, uint32_t sel) {
  const uint32_t w = __byte_perm((uint32_t)v, (uint32_t)(v >> 32), sel);
  const uint32_t a = (w & 0x007F007Fu) | 0x43004300u;
  const uint32_t o = (w & 0x00800080u) ^ 0xC380C380u;
  const __nv_bfloat162 r = __hadd2(*reinterpret_cast<const __nv_bfloat162*>(&a),
                                   *reinterpret_cast<const __nv_bfloat162*>(&o));
  return *reinterpret_cast<const uint32_t*>(&r);
}
// D = A B for one 16 x 8 tile, K = 16 (all BF16 integers, FP32 sums exact)
__device__ __forceinline__ void mma_16x8x16(float* d, const uint32_t* a, uint32_t b0,
                                            uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9},"
      " {%10,%10,%10,%10};"
      : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(0.0f));
}
// Two integers below 2^24 modulo p (balanced to within one unit).  x / p rounds to the nearest
// integer in the single rounding of the FMA.
__device__ __forceinline__ f2 residues(f2 x, f2 invp, f2 negp) {
  const f2 magic = pack2(12582912.0f, 12582912.0f), unmagic = pack2(-12582912.0f, -12582912.0f);
  return fma2(add2(fma2(x, invp, magic), unmagic), negp, x);
}
__device__ __forceinline__ uint32_t bf16_pair(float lo, float hi) {
  const __nv_bfloat162 w = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&w);
}

constexpr int kThreads = 256, kWarps = kThreads / 32;
// a pad of one entry after every eight keeps the digit loads free of bank conflicts
__host__ __device__ constexpr int padded(int k) { return k + (k >> 3); }
// The constants in shared memory (a lane-dependent index into the kernel's parameters is served
// one lane at a time, once per CTA instead of once per warp); padded rows.
typedef uint32_t Coef[2 * kMaxMod][kDigits + 1];
__device__ __forceinline__ void load_coef(const ResidueConst& rc, Coef& coef) {
  for (int i = threadIdx.x; i < 2 * kMaxMod * kDigits; i += blockDim.x)
    coef[i / kDigits][i % kDigits] = reinterpret_cast<const uint32_t*>(&rc.coef[0][0])[i];
}

// The residue planes of lines l0 .. l0 + LINES - 1, elements k0 .. k0 + len - 1 (multiples of 8),
// from their biased integers in shared memory.
template <int LINES, int NB>
__device__ __forceinline__ void write_planes(const ResidueConst& rc, const Coef& coef, int n,
                                             const ulonglong2* ints,
                                             int lds, int l0, int n_lines, int k0, int len, int L,
                                             __nv_bfloat16* base) {
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // lane (g, t) holds columns 2 t, 2 t + 1 of a digit matrix and, of every eight results, the
  // pair (u, v) of modulus 4 b + t
  const int g = lane >> 2, t = lane & 3;
  const uint32_t sel = (uint32_t)(2 * t) | (uint32_t)(2 * t + 1) << 8;
  uint32_t b0[NB], b1[NB];
  f2 invp[NB], negp[NB];
#pragma unroll
  for (int b = 0; b < NB; ++b) {
    const int col = 8 * b + g, l = min(4 * b + t, n - 1);
    b0[b] = coef[col][t];
    b1[b] = coef[col][t + 4];
    invp[b] = pack2(rc.invp[l], rc.invp[l]);
    negp[b] = pack2(rc.negp[l], rc.negp[l]);
  }
  const long long plane = (long long)n_lines * L;  // one residue plane of an item
  const int blocks = (len + 63) / 64;
  for (int job = w; job < LINES * blocks; job += kWarps) {
    const int line = job / blocks, kb = (job - line * blocks) * 64 + 8 * g;
    if (l0 + line >= n_lines) break;
    const bool in = kb < len;
    const ulonglong2* row = ints + line * lds + padded(in ? kb : 0);
    uint32_t u[NB][4], v[NB][4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const ulonglong2 e0 = row[2 * i], e1 = row[2 * i + 1];
      const uint32_t a[4] = {digit_pair(e0.x, sel), digit_pair(e1.x, sel),
                             digit_pair(e0.y, sel), digit_pair(e1.y, sel)};
#pragma unroll
      for (int b = 0; b < NB; ++b) {
        float d[4];
        mma_16x8x16(d, a, b0[b], b1[b]);
        // neighbouring accumulators (u and v of one value) form the pairs without moves
        float u0, v0, u1, v1;
        unpack2(residues(pack2(d[0], d[1]), invp[b], negp[b]), u0, v0);
        unpack2(residues(pack2(d[2], d[3]), invp[b], negp[b]), u1, v1);
        u[b][i] = bf16_pair(u0, u1);
        v[b][i] = bf16_pair(v0, v1);
      }
    }
    if (!in) continue;
#pragma unroll
    for (int b = 0; b < NB; ++b) {
      const int l = 4 * b + t;
      if (l < n) {
        __nv_bfloat16* o = base + 2 * l * plane + (long long)(l0 + line) * L + k0 + kb;
        *reinterpret_cast<uint4*>(o) = make_uint4(u[b][0], u[b][1], u[b][2], u[b][3]);
        *reinterpret_cast<uint4*>(o + plane) = make_uint4(v[b][0], v[b][1], v[b][2], v[b][3]);
      }
    }
  }
}

// Residues of LINES lines per CTA.  The strip (LINES lines of K complex values) is read once,
// coalesced along the operand's memory layout, with the norms taken on the way; its values become
// biased 64-bit integers in shared memory.  A warp then takes 64 values of a line at a time: four
// 16 x 16 digit matrices (rows: values, columns: the digits of Re and Im) times the 16 x 2 n
// constants, whose results are reduced modulo p in registers; a lane ends up with eight
// neighbouring values of a residue plane and stores them as 16 bytes, 128 contiguous bytes per
// plane and warp.  Bound by instruction issue, so that what counts is instructions per value: norms
// take the FP32 value of a mantissa by a shift and a subtraction, sigma is a 64-bit integer
// multiplication (as an FP64 one it held the two-lane FP64 pipe for a fifth of the kernel), and u and
// v of a value are reduced as the neighbouring accumulators that they are.  The two conversions of 64
// products of 400^3 take 314 us (about 360 before these).
template <int LINES, int NB>
__global__ void __launch_bounds__(kThreads)
    k_residue_strip(const __grid_constant__ ResidueConst rc, int n, int alpha, unsigned long long sig,
                    float sigma2, int n_lines, int K, int L, BMc<double> X, int op, bool line_is_col,
                    __nv_bfloat16* out, int32_t* eo, const int32_t* active) {
  static_assert(kWarps % LINES == 0 && 32 % LINES == 0, "warps and lanes per line");
  const int p = blockIdx.y;
  if (active && !active[p]) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int lds = padded(L);
  z64* strip = reinterpret_cast<z64*>(smem_raw);  // [LINES][padded(L)]
  ulonglong2* ints = reinterpret_cast<ulonglong2*>(smem_raw);
  __shared__ Norm part[kWarps][LINES];
  __shared__ int sexp[LINES];
  __shared__ Coef coef;
  load_coef(rc, coef);
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int l0 = blockIdx.x * LINES;
  const z64* x = bat(X, p);
  // line and first element of this thread, and the step between its elements
  constexpr int kPerLine = kWarps / LINES;
  const int li = line_is_col ? lane % LINES : w / kPerLine;
  const int k0 = line_is_col ? w * (32 / LINES) + lane / LINES : (w % kPerLine) * 32 + lane;
  constexpr int kStep = kThreads / LINES, kLoads = 4;
  const bool have = l0 + li < n_lines;
  const long long estride = line_is_col ? X.ld : 1;
  const z64* src = x + (line_is_col ? (long long)(l0 + li) : (long long)(l0 + li) * X.ld);
  Norm nm{1, 0.0f};
  for (int kb = k0; kb < L; kb += kLoads * kStep) {
    z64 v[kLoads];
#pragma unroll
    for (int u = 0; u < kLoads; ++u) {
      const int k = kb + u * kStep;
      v[u] = have && k < K ? src[k * estride] : mkc(0.0, 0.0);
    }
#pragma unroll
    for (int u = 0; u < kLoads; u += 2) {
      const int k = kb + u * kStep;
      if (k >= L) break;
      norm_add<2>(nm, v + u);
      strip[li * lds + padded(k)] = v[u];
      if (k + kStep < L) strip[li * lds + padded(k + kStep)] = v[u + 1];
    }
  }
  if (line_is_col) {
#pragma unroll
    for (int o = 16; o >= LINES; o >>= 1)
      norm_merge(nm, __shfl_xor_sync(0xffffffffu, nm.ex, o), __shfl_xor_sync(0xffffffffu, nm.s, o));
    if (lane < LINES) part[w][lane] = nm;
  } else {
    nm = norm_warp(nm);
    if (lane == 0) part[w][li] = nm;
  }
  __syncthreads();
  if (threadIdx.x < LINES) {
    const int line = threadIdx.x;
    const int first = line_is_col ? 0 : line * kPerLine, count = line_is_col ? kWarps : kPerLine;
    Norm t = part[first][line];
    for (int i = 1; i < count; ++i) norm_merge(t, part[first + i][line].ex, part[first + i][line].s);
    const int e = scale_of(t, alpha, sigma2);
    sexp[line] = e;
    if (l0 + line < n_lines)
      eo[(long long)p * n_lines + l0 + line] = e == kNonFinite ? kNonFinite : -e;
  }
  __syncthreads();
  {  // each thread converts the elements that it loaded
    const bool fine = sexp[li] != kNonFinite;
    const unsigned conj = op == OP_C ? 0x80000000u : 0u;
    const int e = fine ? sexp[li] : 0;
#pragma unroll 2
    for (int k = k0; k < L; k += kStep) {
      const int at = li * lds + padded(k);
      const z64 v = fine ? strip[at] : mkc(0.0, 0.0);
      ints[at] = make_ulonglong2(biased(v.re, e, 0u, sig), biased(v.im, e, conj, sig));
    }
  }
  __syncthreads();
  write_planes<LINES, NB>(rc, coef, n, ints, lds, l0, n_lines, 0, L, L,
                          out + (long long)p * 2 * n * n_lines * L);
}

// Lines too long for a strip in shared memory: one line per CTA, its norm in a first pass over it,
// then its residues kSegment elements at a time.
constexpr int kSegment = 4096;
template <int NB>
__global__ void __launch_bounds__(kThreads)
    k_residue_long(const __grid_constant__ ResidueConst rc, int n, int alpha, unsigned long long sig,
                   float sigma2, int n_lines, int K, int L, BMc<double> X, int op, bool line_is_col,
                   __nv_bfloat16* out, int32_t* eo, const int32_t* active) {
  const int p = blockIdx.y;
  if (active && !active[p]) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  ulonglong2* ints = reinterpret_cast<ulonglong2*>(smem_raw);
  __shared__ Norm part[kWarps];
  __shared__ int sexp;
  __shared__ Coef coef;
  load_coef(rc, coef);
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, line = blockIdx.x;
  const long long estride = line_is_col ? X.ld : 1;
  const z64* src = bat(X, p) + (line_is_col ? (long long)line : (long long)line * X.ld);
  Norm nm{1, 0.0f};
  for (int k = threadIdx.x; k < K; k += kThreads) {
    const z64 v = src[k * estride];
    norm_add<1>(nm, &v);
  }
  nm = norm_warp(nm);
  if (lane == 0) part[w] = nm;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int i = 1; i < kWarps; ++i) norm_merge(nm, part[i].ex, part[i].s);
    sexp = scale_of(nm, alpha, sigma2);
    eo[(long long)p * n_lines + line] = sexp == kNonFinite ? kNonFinite : -sexp;
  }
  __syncthreads();
  const bool fine = sexp != kNonFinite;
  const unsigned conj = op == OP_C ? 0x80000000u : 0u;
  const int e = fine ? sexp : 0;
  for (int s0 = 0; s0 < L; s0 += kSegment) {
    const int len = min(kSegment, L - s0);
    for (int k = threadIdx.x; k < len; k += kThreads) {
      const z64 v = fine && s0 + k < K ? src[(s0 + k) * estride] : mkc(0.0, 0.0);
      ints[padded(k)] = make_ulonglong2(biased(v.re, e, 0u, sig), biased(v.im, e, conj, sig));
    }
    __syncthreads();
    write_planes<1, NB>(rc, coef, n, ints, 0, line, n_lines, s0, len, L,
                        out + (long long)p * 2 * n * n_lines * L);
    __syncthreads();
  }
}

// Largest strip of `lines` lines.
constexpr int kStripBytes = 200 * 1024;
__host__ constexpr size_t strip_bytes(int lines, int L) {
  return (size_t)lines * padded(L) * sizeof(z64);
}

}  // namespace

namespace {
template <int LINES, int NB>
cudaError_t launch_strip(cudaStream_t s, const CrtPlan& pl, int alpha, unsigned long long sig,
                         float sigma2, int items, int n_lines, int K, int L, BMc<double> X, int op, bool line_is_col,
                         __nv_bfloat16* out, int32_t* eo, const int32_t* active) {
  static std::atomic<unsigned> attr{0};
  cudaError_t e = set_smem_once(attr, reinterpret_cast<const void*>(&k_residue_strip<LINES, NB>),
                                kStripBytes);
  if (e != cudaSuccess) return e;
  const dim3 grid((n_lines + LINES - 1) / LINES, items);
  k_residue_strip<LINES, NB><<<grid, kThreads, strip_bytes(LINES, L), s>>>(
      residue_const(pl), pl.n, alpha, sig, sigma2, n_lines, K, L, X, op, line_is_col, out, eo, active);
  return cudaGetLastError();
}
template <int LINES>
cudaError_t launch_strip(cudaStream_t s, const CrtPlan& pl, int alpha, unsigned long long sig,
                         float sigma2, int items, int n_lines, int K, int L, BMc<double> X, int op, bool line_is_col,
                         __nv_bfloat16* out, int32_t* eo, const int32_t* active) {
  if (pl.n <= 12)
    return launch_strip<LINES, 3>(s, pl, alpha, sig, sigma2, items, n_lines, K, L, X, op, line_is_col,
                                  out, eo, active);
  return launch_strip<LINES, 4>(s, pl, alpha, sig, sigma2, items, n_lines, K, L, X, op, line_is_col,
                                out, eo, active);
}
}  // namespace

namespace {
cudaError_t launch_long(cudaStream_t s, const CrtPlan& pl, int alpha, unsigned long long sig,
                        float sigma2, int items, int n_lines, int K, int L, BMc<double> X, int op, bool line_is_col,
                        __nv_bfloat16* out, int32_t* eo, const int32_t* active) {
  auto* fn = pl.n <= 12 ? &k_residue_long<3> : &k_residue_long<4>;
  static std::atomic<unsigned> attr[2];
  const size_t smem = strip_bytes(1, kSegment);
  cudaError_t e = set_smem_once(attr[pl.n <= 12 ? 0 : 1], reinterpret_cast<const void*>(fn),
                                (int)smem);
  if (e != cudaSuccess) return e;
  fn<<<dim3(n_lines, items), kThreads, smem, s>>>(residue_const(pl), pl.n, alpha, sig, sigma2, n_lines, K,
                                                  L, X, op, line_is_col, out, eo, active);
  return cudaGetLastError();
}
}  // namespace

cudaError_t launch_residues(cudaStream_t s, const CrtPlan& pl, int alpha, double sigma, int items,
                            int n_lines, int K, int L, BMc<double> X, int op, bool line_is_col,
                            __nv_bfloat16* out, int32_t* eo, const int32_t* active) {
  const unsigned long long sig = sigma < 1.0 ? (unsigned long long)ldexp(sigma, 64) : 0ull;
  const float sigma2 = (float)(sigma * sigma);
  // eight lines per CTA while three CTAs fit an SM (the constants and the reductions are then a
  // small part of a CTA's work), fewer for longer lines
  constexpr size_t kThree = 74 * 1024;
  if (strip_bytes(8, L) <= kThree)
    return launch_strip<8>(s, pl, alpha, sig, sigma2, items, n_lines, K, L, X, op, line_is_col, out, eo,
                           active);
  if (strip_bytes(4, L) <= kThree)
    return launch_strip<4>(s, pl, alpha, sig, sigma2, items, n_lines, K, L, X, op, line_is_col, out, eo,
                           active);
  if (strip_bytes(2, L) <= kThree)
    return launch_strip<2>(s, pl, alpha, sig, sigma2, items, n_lines, K, L, X, op, line_is_col, out, eo,
                           active);
  if (strip_bytes(1, L) <= kStripBytes)
    return launch_strip<1>(s, pl, alpha, sig, sigma2, items, n_lines, K, L, X, op, line_is_col, out, eo,
                           active);
  return launch_long(s, pl, alpha, sig, sigma2, items, n_lines, K, L, X, op, line_is_col, out, eo,
                     active);
}

}  // namespace negf
