// Operand residues of the tensor-core complex GEMM (internal): every row of op(A) and column of
// op(B) is scaled by a power of two so that its 2-norm lies below 2^alpha, rounded once to
// integers, and written modulo p_1 .. p_n as the pairs (u, v) = (a + j b, a - j b) of crt_plan.cuh,
// balanced residues that BF16 holds exactly.
#pragma once
#include <cuda_bf16.h>

#include "common.cuh"
#include "crt_plan.cuh"
#include "tc_slice.cuh"

namespace negf {

// Exponent of a line that holds an infinity or NaN: its products are NaN.
constexpr int kNonFinite = 1 << 20;

// Residues of n_lines lines of `items` matrices, K complex values each (element k of a line is
// op(X)[line][k] when the lines are rows of op(A), op(X)[k][line] when they are columns of op(B);
// line_is_col: whether a line is a column of X in memory), multiplied by sigma.  out[item][2 l + h][line][L] (h = 0:
// u, 1: v; l < n), zero from K to L; eo[item][line]: the line is 2^eo times its integers.
// Items with active[item] == 0 are skipped.
cudaError_t launch_residues(cudaStream_t s, const CrtPlan& pl, int alpha, double sigma,
                            int items, int n_lines, int K, int L, BMc<double> X, int op, bool line_is_col,
                            __nv_bfloat16* out, int32_t* eo, const int32_t* active);

}  // namespace negf
