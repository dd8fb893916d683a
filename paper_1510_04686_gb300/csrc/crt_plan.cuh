// Residue plan of the tensor-core complex GEMM (internal): the moduli, the precision they carry
// and the constants of the residue and reconstruction kernels.
//
// A product of integer matrices whose entries stay below P / 2 in magnitude is determined by its
// residues modulo pairwise coprime p_1 .. p_n with product P (Chinese remainder theorem).  Every
// p here has only prime factors = 1 mod 4, so -1 has a square root j modulo p and the Gaussian
// integers modulo p split into two independent rings: a + i b -> (u, v) = (a + j b, a - j b).
// One complex product modulo p is then two real products u u', v v' (instead of the four of a
// real embedding), and Re = (u + v) / 2, Im = (u - v) / (2 j).
#pragma once
#include <stddef.h>
#include <stdint.h>

namespace negf {

constexpr int kMaxMod = 16;  // most moduli of a plan
constexpr int kDigits = 8;   // balanced base-256 digits of a scaled operand value

// Residue kernels: a value is written in balanced digits, x = sum_i x_i 2^(8 i) with
// -128 <= x_i <= 127; then a + j b and a - j b modulo p_l are sums of sixteen digits (those of a,
// then those of b) times the constants coef[2 l + h], h = 0 (u) and 1 (v): balanced residues of
// 2^(8 i) and +- j 2^(8 i).  Digits and constants are exact in BF16 and the sums, below
// 16 * 128 * 256, in FP32, so they are small matrix products.
struct ResidueConst {
  uint16_t coef[2 * kMaxMod][2 * kDigits];  // BF16 bit patterns
  float invp[kMaxMod];
  float negp[kMaxMod];
};

// Reconstruction: with s = u + v and t = u - v modulo p_l, Re x / P = sum_l s_l re[l] and
// Im x / P = sum_l t_l im[l] modulo 1, both as 64-bit binary fractions (the wrap-around of the
// integer sum is the reduction modulo 1).  hre, him: what the rounding of re[l], im[l] to 64 bits
// left, in units of the last place; their sums correct the fraction where its own rounding would
// show (CrtPlan::hp; in the 56-bit tier it is 2^-56.6 of P, the operands' rounding 2^-60).  P = sigma 2^expo with sigma in (1/2, 1): the values of
// op(A) are multiplied by sigma before they are rounded to integers, so that the product itself is
// simply fraction * 2^expo (a multiplication per operand value instead of one per result, which
// would stand at the end of every tile).  Where the fractions are corrected the results are multiplied
// by mant instead: the 56-bit tier's operands would feel the rounding of that multiplication.
struct CrtConst {
  float invp[kMaxMod];
  float negp[kMaxMod];
  unsigned long long re[kMaxMod];
  unsigned long long im[kMaxMod];
  float hre[kMaxMod], him[kMaxMod];
  double sigma;
  unsigned long long mant;  // sigma 2^64, truncated
  int expo;
};

struct CrtPlan {
  int cls;         // modulus class (kClasses of crt_plan.cu)
  int n;           // moduli
  int parts;       // K parts, each exact in one FP32 accumulator
  int k16;         // 16-wide K steps per part (the last part may be shorter)
  int alpha_a;     // line norms of op(A) are scaled below 2^alpha_a,
  int alpha_b;     // those of op(B) below 2^alpha_b; 2^(alpha_a + alpha_b) < P / 2
  bool hp;         // the fractions need their correction sums (56-bit tier, long contractions)
};

// Products inside the refinement of an inverse (engine.cu), which need no tier's precision.
constexpr int kCorrectionBits = 36;
// The plan for a contraction of K complex terms at `bits` bits per value (a tier's, or
// kCorrectionBits); false where the tier does not cover K (tc_supports_k).
bool crt_plan(int K, int bits, CrtPlan* out);
// Row length of the residue planes: K rounded up to 8 (rows of whole 16-byte units for the TMA).
inline int residue_ld(int K) { return (K + 7) / 8 * 8; }
// Elements of one operand line in all residue planes of a contraction of K terms (2 n rows); with
// `shorter`, the most that any contraction of up to K terms takes in this tier or a narrower one.
// The number of moduli does not grow with K: 513 to 560 terms in the 48-bit tier take 13 in one K
// part, 561 to 600 take 12 in two, so the longest contraction is not always the one that needs most.
size_t crt_line_elements(int K, int bits, bool shorter);
// Constants of a plan's modulus set (its first n moduli).
const ResidueConst& residue_const(const CrtPlan& pl);
const CrtConst& crt_const(const CrtPlan& pl);

}  // namespace negf
