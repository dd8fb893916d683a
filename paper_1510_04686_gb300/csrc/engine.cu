// Engine dispatch: FP64 reference form and the mixed-precision tensor-core form.
#include <atomic>

#include "crt_gemm.cuh"
#include "engine.cuh"
#include "profile.cuh"
#include "tc_gemm.cuh"

namespace negf {

namespace {
template <class T>
T* take(char* base, size_t& off, size_t n) {
  size_t a = (off + 255) & ~size_t(255);
  off = a + n * sizeof(T);
  return base ? reinterpret_cast<T*>(base + a) : nullptr;
}

}  // namespace

__device__ unsigned long long g_fp64_fallbacks;  // items recomputed by the FP64 fallback

// Newton-Schulz gating: act[p] = (active ? active[p] : 1) && (force || rmax[p] > tol); rmax[p]
// is reset to 0 for the next residual product.  With count set, the selected items are added
// to g_fp64_fallbacks.  act may alias active (each thread reads its own entry first).
__global__ void k_refine_gate(int P, const int32_t* active, int force, float* rmax, float tol,
                              int32_t* act, int count) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= P) return;
  const bool base = active ? active[p] != 0 : true;
  const bool on = base && (force || rmax[p] > tol);
  act[p] = on ? 1 : 0;
  rmax[p] = 0.0f;
  if (on && count) atomicAdd(&g_fp64_fallbacks, 1ull);
}

// Residual target of the mixed-form inverse: after a step with max |R| <= 2^-24 the next
// residual R^2 is at the rounding floor of the products.
constexpr float kRefineTol = 5.9604644775390625e-8f;
void carve_engine(char* base, size_t& off, int P, int b, int precision, bool residues,
                  EngineWs& w) {
  const size_t bb = (size_t)b * b;
  const int nb64 = gj_panel_width(b, (int)sizeof(z64));
  w.invU = take<z64>(base, off, (size_t)P * b * nb64);
  w.invT = take<z64>(base, off, (size_t)P * b * nb64);
  w.piv = take<int32_t>(base, off, (size_t)P * b);
  w.map = nullptr;
  w.m32 = w.x32 = w.invU32 = nullptr;
  w.r64 = nullptr;
  w.act = nullptr;
  w.rmax = nullptr;
  w.tc = nullptr;
  w.residues = residues;
  if (prec_mixed(precision)) {
    const int nb32 = gj_panel_width(b, (int)sizeof(cx<float>));
    w.map = take<int32_t>(base, off, (size_t)P * b);
    w.m32 = take<cx<float>>(base, off, (size_t)P * bb);
    w.x32 = take<cx<float>>(base, off, (size_t)P * bb);
    w.invU32 = take<cx<float>>(base, off, (size_t)P * b * nb32);
    w.r64 = take<z64>(base, off, (size_t)P * bb);
    w.act = take<int32_t>(base, off, (size_t)P);
    w.rmax = take<float>(base, off, (size_t)P);
    size_t a = (off + 1023) & ~size_t(1023);
    w.tc = base ? base + a : nullptr;
    off = a;
    if (residues) {
      CrtWs cw;
      crt_ws_carve(base, off, P, b, b, b, prec_bits(precision), true, cw);
    } else {
      TcWs tw;
      tc_ws_carve(base, off, P, b, b, b, prec_bits(precision), tw);
    }
  }
}

bool engine_supports(int precision, int b) {
  if (precision == NEGF_PREC_FP64) return gj_supports(b, 16);
  return prec_mixed(precision) && tc_supports_k(b, prec_bits(precision)) && gj_supports(b, 8);
}

int lead_precision(const negf_options* o, int b) {
  if (o->lead_precision != NEGF_PREC_AUTO) return o->lead_precision;
  if (o->precision == NEGF_PREC_FP64) return NEGF_PREC_FP64;
  return engine_supports(NEGF_PREC_MIXED_56, b) ? NEGF_PREC_MIXED_56 : NEGF_PREC_MIXED;
}

int lead_step_precision(const negf_options* o, int b, int it) {
  const int p = lead_precision(o, b);
  if (o->lead_precision != NEGF_PREC_AUTO || p != NEGF_PREC_MIXED_56) return p;
  if (it == 0) return NEGF_PREC_MIXED;
  if (it <= 8) return NEGF_PREC_MIXED_56;
  return it <= 14 ? NEGF_PREC_MIXED : NEGF_PREC_MIXED_40;
}

long long engine_fp64_fallbacks() {
  unsigned long long v = 0;
  if (cudaMemcpyFromSymbol(&v, g_fp64_fallbacks, sizeof(v)) != cudaSuccess) return -1;
  return (long long)v;
}

static TcWs tc_view(const EngineWs& w, int P, int b, int bits) {
  TcWs t;
  size_t off = 0;
  tc_ws_carve(static_cast<char*>(w.tc), off, P, b, b, b, bits, t);
  return t;
}
static CrtWs crt_view(const EngineWs& w, int P, int b, int bits) {
  CrtWs t;
  size_t off = 0;
  crt_ws_carve(static_cast<char*>(w.tc), off, P, b, b, b, bits, true, t);
  return t;
}
// The device error word, first in the operand scratch of either form.
static int32_t* err_word(const EngineWs& w) {
  return static_cast<int32_t*>(w.tc);
}

cudaError_t Engine::gemm(int P, int M, int N, int K, z64 alpha, BMc<double> A, int opA,
                         BMc<double> B, int opB, z64 beta, BM<double> C, z64 gamma,
                         BMc<double> D, const int32_t* active, int reuse) {
  kept.reuse = reuse;
  if (prec_mixed(prec) && w.residues)
    return crt_gemm(s, P, M, N, K, alpha, A, opA, B, opB, beta, C, gamma, D, false, active,
                    crt_view(w, P, b, prec_bits(prec)), prec_bits(prec), n_sys, nullptr, &kept);
  if (prec_mixed(prec))
    return tc_gemm(s, P, M, N, K, alpha, A, opA, B, opB, beta, C, gamma, D, false, active,
                   tc_view(w, P, b, prec_bits(prec)), prec_bits(prec), n_sys, false, nullptr,
                   &kept);
  return gemm_simt(s, P, M, N, K, alpha, A, opA, B, opB, beta, C, gamma, D, active);
}

cudaError_t Engine::timeout_reset() {
  if (!prec_mixed(prec)) return cudaSuccess;
  return tc_timeout_reset(s, err_word(w));
}

namespace {
std::atomic<int> g_fail_waits{0};
}

cudaError_t Engine::timeout_flag(int P, int32_t* status) {
  if (!prec_mixed(prec)) return cudaSuccess;
  if (g_fail_waits.load()) {  // test hook: report as if a bounded wait had given up
    cudaError_t e = cudaMemsetAsync(err_word(w), 1, sizeof(int32_t), s);
    if (e != cudaSuccess) return e;
  }
  return tc_timeout_flag(s, err_word(w), P, status);
}

void engine_fail_waits(int on) { g_fail_waits.store(on ? 1 : 0); }

cudaError_t Engine::inv(int P, BM<double> Mm, BM<double> X, int32_t* status,
                        const int32_t* active) {
  if (!prec_mixed(prec)) {
    prof_begin(s, PROF_INV);
    cudaError_t e = gj_inverse64(s, P, b, Mm, X, w.invU, w.invT, w.piv, status, active);
    prof_end(s, PROF_INV);
    return e;
  }
  kept = Kept{};  // the products below use the same scratch
  // FP32 Gauss-Jordan start X0, then X <- X + X (I - M X) with tensor-core products
  const long long bb = (long long)b * b;
  if (Mm.idx || X.idx || Mm.stride != bb || X.stride != bb || Mm.ld != b || X.ld != b)
    return cudaErrorInvalidValue;
  prof_begin(s, PROF_INV);
  cudaError_t e = gj_inverse32(s, P, b, Mm, X, w.m32, w.x32, w.invU32, w.piv, w.map, status, active);
  prof_end(s, PROF_INV);
  if (e != cudaSuccess) return e;
  if (refine_max <= 0) return cudaSuccess;
  const int bits = prec_bits(prec);
  const BMc<double> none{nullptr, 0, nullptr, 0};
  const unsigned gb = (unsigned)((P + 255) / 256);
  BM<double> R{w.r64, bb, nullptr, b};
  const BMc<double> Mc = cst(Mm);
  const BMc<double> Xc{X.p, bb, nullptr, b};
  for (int it = 0; it < refine_max; ++it) {
    // items refined by this step: all of them for the first refine_min steps, afterwards those
    // whose previous residual stayed above the target
    k_refine_gate<<<gb, 256, 0, s>>>(P, active, (it == 0 || it < refine_min) ? 1 : 0, w.rmax,
                                     kRefineTol, w.act, 0);
    count_launch();
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    const z64 zero = mkc(0.0, 0.0), one = mkc(1.0, 0.0), mone = mkc(-1.0, 0.0);
    if (w.residues) {
      // A step that every item follows with another one does not need its residual in the tier's
      // precision: the error of kCorrectionBits, 2^-40 |M| |X| in R, is the next step's to remove,
      // as is R^2 (an FP32 start leaves R = 2^-24 |M| |X| or more, so no item takes a step more for
      // it).  The correction X R needs no more at any step: an item is done when |R| <= 2^-24, where
      // they put the error of X R below 2^-58 of |X|.
      const CrtWs cw = crt_view(w, P, b, bits);
      const int rbits = it + 1 < refine_min ? kCorrectionBits : bits;
      e = crt_gemm(s, P, b, b, b, mone, Mc, OP_N, Xc, OP_N, zero, R, zero, none, true, w.act, cw,
                   rbits, 0, w.rmax);
      if (e != cudaSuccess) return e;
      e = crt_gemm(s, P, b, b, b, one, Xc, OP_N, cst(R), OP_N, zero, X, one, Xc, false, w.act, cw,
                   kCorrectionBits);
      if (e != cudaSuccess) return e;
      continue;
    }
    const TcWs tw = tc_view(w, P, b, bits);
    e = tc_gemm(s, P, b, b, b, mone, Mc, OP_N, Xc, OP_N, zero, R, zero, none, true, w.act, tw,
                bits, 0, false, w.rmax);
    if (e != cudaSuccess) return e;
    // X <- X + X R in place (each output element reads only its own X entry; the product reads
    // the slices of X made before it).  With |R| << 1 only accuracy relative to |X| matters.
    e = tc_gemm(s, P, b, b, b, one, Xc, OP_N, cst(R), OP_N, zero, X, one, Xc, false, w.act, tw,
                bits, 0, true);
    if (e != cudaSuccess) return e;
  }
  // items whose last residual was still above the target: FP64 Gauss-Jordan (M is intact)
  k_refine_gate<<<gb, 256, 0, s>>>(P, w.act, 0, w.rmax, kRefineTol, w.act, 1);
  count_launch();
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  prof_begin(s, PROF_INV);
  e = gj_inverse64(s, P, b, Mm, X, w.invU, w.invT, w.piv, status, w.act, true);
  prof_end(s, PROF_INV);
  return e;
}

}  // namespace negf
