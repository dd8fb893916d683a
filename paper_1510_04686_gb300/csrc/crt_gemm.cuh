// Tensor-core complex GEMM with FP64-class accuracy from exact residue products.
//
//   C = alpha op(A) op(B) + beta C + gamma D (+ I)       (complex128 in and out)
//
// Each operand row (A) / column (B) is scaled by a power of two so that its 2-norm lies below
// 2^alpha_a (2^alpha_b) and rounded once to integers.  The integer product is computed exactly
// modulo n pairwise coprime integers p of up to 9 bits: balanced residues are exact in BF16, a
// sum of K products of them stays below 2^24 and is exact in the FP32 accumulator of the tensor
// core (K is cut into parts where it is too long), and by Cauchy-Schwarz every result is below
// P / 2, P the product of the moduli, so its residues determine it (Chinese remainder theorem).
// (Products by residues of scaled integers are the method of Ozaki, Uchino and Imamura, "Ozaki scheme
// II: a GEMM-oriented emulation of floating-point matrix multiplication using an integer modular
// technique"; the form below is this library's own.)
// The moduli split over the Gaussian integers, so a complex product takes two real products per
// modulus (crt_plan.cuh): 24 of b x b x b for 48-bit values at b = 400, where fixed-point digit
// products take 84 (21 digit pairs in the four-product real embedding).  The only rounding is
// that of the scaled operands and of the FP64 result.
#pragma once
#include "common.cuh"
#include "crt_plan.cuh"
#include "tc_gemm.cuh"

namespace negf {

struct CrtWs {
  void* resA;           // bf16 [P][2 n][M][L]
  void* resB;           // bf16 [P][2 n][N][L]
  int32_t* expA;        // [P][M]
  int32_t* expB;        // [P][N]
  int32_t* err;         // device error word (bounded waits that gave up)
  size_t elemsA, elemsB;  // what resA and resB hold, and the lines of expA and expB: a product
  size_t linesA, linesB;  // that needs more is refused
};

// CrtWs scratch for P items of an M x N x K product at `bits` bits per value; with `shorter`, for
// every product of up to K terms at these bits or fewer, as the sweeps of b x b blocks need it.
void crt_ws_carve(char* base, size_t& off, int P, int M, int N, int K, int bits, bool shorter,
                  CrtWs& w);
// Bytes of the scratch of one product.
size_t crt_ws_bytes(int P, int M, int N, int K, int bits);

// Flops of the tensor-core GEMM launches made while profiling was on, counted on the device
// for the items that ran (the current device; both calls synchronise it): algorithmic complex
// 8 M N K, and the BF16 MMA flops issued over the padded tiles.
cudaError_t crt_prof_flops(double* alg, double* hw);
cudaError_t crt_prof_reset();

// n_distinct: number of different matrices an indexed operand (idx != NULL) selects from
// (0 = unknown: convert every item).  bits: a tier's (tc_bits_ok) or kCorrectionBits; the
// workspace must have been carved for such a product (else cudaErrorInvalidValue).  rmax (nullable, float [P], zeroed by the
// caller): rmax[p] is raised to the largest |Re| or |Im| of item p's outputs (the Newton-Schulz
// residual norm when C = I - M X).  kept (nullable): what the scratch of `ws` holds, see Kept.
cudaError_t crt_gemm(cudaStream_t s, int P, int M, int N, int K, z64 alpha, BMc<double> A,
                    int opA, BMc<double> B, int opB, z64 beta, BM<double> C, z64 gamma,
                    BMc<double> D, bool add_identity, const int32_t* active, const CrtWs& ws,
                    int bits, int n_distinct = 0, float* rmax = nullptr, Kept* kept = nullptr);

}  // namespace negf
