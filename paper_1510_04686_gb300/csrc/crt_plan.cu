// Moduli and constants of the residue GEMM (see crt_plan.cuh).  Host code only.
#include "crt_plan.cuh"

#include <algorithm>
#include <cmath>
#include <cstring>
#include <mutex>
#include <vector>

#include "tc_gemm.cuh"

namespace negf {
namespace {

using u128 = unsigned __int128;

// Modulus classes.  Residues are at most (p + 1) / 2 in magnitude (exact in BF16 up to 256), so
// a sum of K products stays below 2^24, exact in an FP32 accumulator, when
// K ((p + 1) / 2)^2 <= 2^24.  Larger moduli carry more bits per product but fewer terms: each
// class is the set of the largest usable moduli for contractions (or parts of them) of up to the length
// that it names.  The lengths rise by 1.25 from 256 to 1024; one of 320 is left out because it takes
// as many moduli as 400 in every tier.
constexpr int kClasses = 6;
constexpr int kClassK[kClasses] = {256, 400, 512, 640, 800, 1024};
constexpr int kMaxAlpha = 60;  // scaled values stay below 2^61 (64-bit fixed point, eight digits)

struct Class {
  int count;
  int p[kMaxMod];
  ResidueConst rc;
  double log2P[kMaxMod + 1];
  int alpha[kMaxMod + 1];  // largest a with 2^a < P / 2
  CrtConst cc[kMaxMod + 1];
};
Class g_class[kClasses];
std::once_flag g_once;

int balanced(long long x, int p) {
  long long r = x % p;
  if (r < 0) r += p;
  return (int)(2 * r > p ? r - p : r);
}
int inverse_mod(long long a, int p) {
  a %= p;
  if (a < 0) a += p;
  for (int x = 1; x < p; ++x)
    if (a * x % p == 1) return x;
  return 0;
}
bool splits(int m) {  // every prime factor of m is 1 mod 4
  for (int d = 2; d * d <= m; ++d)
    while (m % d == 0) {
      if (d % 4 != 1) return false;
      m /= d;
    }
  return m == 1 || m % 4 == 1;
}
int gcd(int a, int b) { return b ? gcd(b, a % b) : a; }
// BF16 bit pattern of an integer of at most 256 in magnitude (exact)
uint16_t bf16_bits(int x) {
  const float f = (float)x;
  uint32_t u;
  std::memcpy(&u, &f, sizeof(u));
  return (uint16_t)(u >> 16);
}
// round(2^64 g / p) modulo 2^64
unsigned long long fraction(int g, int p) {
  return (unsigned long long)((((u128)g << 64) + (unsigned)p / 2) / (unsigned)p);
}
// 2^64 g / p - fraction(g, p)
float fraction_rest(int g, int p) {
  const int r = (int)(((u128)g << 64) % (unsigned)p);
  return (float)((double)balanced(r, p) / p);
}

void build() {
  for (int c = 0; c < kClasses; ++c) {
    Class& k = g_class[c];
    const int half = std::min(256, (int)std::floor(std::sqrt(16777216.0 / kClassK[c])));
    k.count = 0;
    for (int m = 2 * half - 1; m > 4 && k.count < kMaxMod; m -= 2) {
      if (!splits(m)) continue;
      bool ok = true;
      for (int i = 0; i < k.count; ++i) ok = ok && gcd(m, k.p[i]) == 1;
      if (ok) k.p[k.count++] = m;
    }
    int j[kMaxMod];
    for (int l = 0; l < k.count; ++l) {
      const int p = k.p[l];
      j[l] = 1;
      while ((j[l] * j[l] + 1) % p != 0) ++j[l];
      long long w = 1;
      for (int i = 0; i < kDigits; ++i) {
        const int c = balanced(w, p), d = balanced(w * j[l], p);
        k.rc.coef[2 * l][i] = k.rc.coef[2 * l + 1][i] = bf16_bits(c);
        k.rc.coef[2 * l][kDigits + i] = bf16_bits(d);
        k.rc.coef[2 * l + 1][kDigits + i] = bf16_bits(-d);
        w = w * 256 % p;
      }
      k.rc.invp[l] = 1.0f / (float)p;
      k.rc.negp[l] = -(float)p;
    }
    k.log2P[0] = 0.0;
    k.alpha[0] = 0;
    u128 P = 1;
    bool fits = true;
    for (int n = 1; n <= k.count; ++n) {
      // P stays below 2^126: longer prefixes are not offered
      fits = fits && k.log2P[n - 1] + std::log2((double)k.p[n - 1]) < 126.0;
      if (!fits) {
        k.count = n - 1;
        break;
      }
      P *= (unsigned)k.p[n - 1];
      k.log2P[n] = k.log2P[n - 1] + std::log2((double)k.p[n - 1]);
      int bits = 0;  // 2^(bits - 1) < P < 2^bits
      while ((P >> bits) != 0) ++bits;
      // 2^(bits - 2) < P / 2; the margin covers the rounding of the scaled lines
      int a = bits - 2;
      const u128 top = (u128)1 << (bits - 1);
      if ((P - top) < (top >> 20)) --a;
      k.alpha[n] = a;
      CrtConst& cc = k.cc[n];
      for (int l = 0; l < n; ++l) {
        const int p = k.p[l];
        const int m = (int)((P / (unsigned)p) % (unsigned)p);  // P / p_l modulo p_l
        const int mi = inverse_mod(m, p);
        cc.invp[l] = 1.0f / (float)p;
        cc.negp[l] = -(float)p;
        const int gr = (int)((long long)mi * inverse_mod(2, p) % p);
        const int gi = (int)((long long)mi * inverse_mod(2LL * j[l], p) % p);
        cc.re[l] = fraction(gr, p);
        cc.im[l] = fraction(gi, p);
        cc.hre[l] = fraction_rest(gr, p);
        cc.him[l] = fraction_rest(gi, p);
      }
      cc.expo = bits;
      cc.mant = bits >= 64 ? (unsigned long long)(P >> (bits - 64))
                           : (unsigned long long)P << (64 - bits);
      cc.sigma = std::ldexp((double)(unsigned long long)(bits > 64 ? P >> (bits - 64) : P),
                            bits > 64 ? -64 : -bits);
    }
  }
}

void ready() { std::call_once(g_once, build); }

// Least alpha_a + alpha_b of a tier of w-bit values (tc_value_bits, those of the digit products).  A
// line is scaled so that its 2-norm lies in [2^(alpha - 1), 2^alpha); the roundings of both operands
// then put a result off by 1.2 * 2^-alpha |A line| |B line| (rms) at most, and alpha = w + 2 holds
// nearly all results within 2^-w |A line| |B line|.  Digit products, whose values are rounded relative
// to the largest entry of a line, are stated to 2^-w K max|A line| max|B line|, which is never less.
// Error against 64 bits, relative to the result, here / digits: normally distributed entries, 48 bits,
// K = 400 1.4e-14 / 4.9e-14, 512 3.8e-15 / 5.1e-14, 1024 2.8e-14 / 6.2e-14; 40 bits, K = 512
// 9.1e-13 / 1.2e-11.  Entries of one size, the most favourable to digits: 48 bits, K = 400 1.4e-14 /
// 6.9e-15, 512 3.8e-15 / 6.9e-15, 1024 2.8e-14 / 7.1e-15; one modulus more would bring these level too,
// for 733 -> 857 us of 64 products of 400^3.
// The 56-bit tier is at the level of FP64 arithmetic, below its digit products.  Corrections: 2^-40 of
// |A line| |B line| (2^-43 for the longest), so that a product with |B| <= 2^-24 everywhere is good to
// 2^-58 of |A line|.  (40-bit contractions beyond 1024 terms take nearly what the wider digits of the
// longest ones, 42 bits, ask for.)
int need_alpha(int K, int bits) {
  if (bits == 56) return 113;
  if (bits == kCorrectionBits) return K <= 1024 ? 80 : 87;
  const int need = 2 * tc_value_bits(K, bits) + 4;
  return bits == 40 && K > 1024 ? std::max(need, 87) : need;
}
// Whether the rounding of the reconstruction's fractions to 64 bits would show: it is about 2^-67 p
// sqrt(n parts) of P, half of what the 48-bit tier allows at some 5000 terms.
bool need_corrections(int K, int bits) { return bits == 56 || (bits == 48 && K > 4096); }

}  // namespace

bool crt_plan(int K, int bits, CrtPlan* out) {
  if (!tc_supports_k(K, std::max(bits, 40))) return false;
  ready();
  // Cost of a plan in K terms of one real product per output: n moduli, each with one
  // accumulator flush per part that is worth kFlush terms (the flush of one part overlaps the
  // products of the next), plus the residues of both operands.
  constexpr double kFlush = 320.0, kResidue = 0.5;
  const int k16 = (K + 15) / 16;
  const int need = need_alpha(K, bits);
  double best = -1.0;
  for (int c = 0; c < kClasses; ++c) {
    const Class& k = g_class[c];
    int n = 1;
    while (n <= k.count && std::min(k.alpha[n], 2 * kMaxAlpha) < need) ++n;
    if (n > k.count) continue;
    const int most = kClassK[c] / 16;
    const int parts = (k16 + most - 1) / most;
    const int per = (k16 + parts - 1) / parts;
    const double cost = n * (parts * std::max(16.0 * per, kFlush) + kResidue * K);
    if (best >= 0.0 && cost >= best) continue;
    best = cost;
    const int sum = std::min(k.alpha[n], 2 * kMaxAlpha);
    *out = CrtPlan{c, n, parts, per, (sum + 1) / 2, sum / 2, need_corrections(K, bits)};
  }
  return best >= 0.0;
}

size_t crt_line_elements(int K, int bits, bool shorter) {
  if (!shorter) {
    CrtPlan pl;
    return crt_plan(K, bits, &pl) ? 2 * (size_t)pl.n * residue_ld(K) : 0;
  }
  // running maxima over k, extended as far as they have been asked for
  static std::mutex mu;
  static std::vector<size_t> most[4];
  constexpr int kTiers[4] = {kCorrectionBits, 40, 48, 56};
  std::lock_guard<std::mutex> lk(mu);
  size_t need = 0;
  for (int t = 0; t < 4 && kTiers[t] <= bits; ++t) {
    std::vector<size_t>& m = most[t];
    for (int k = (int)m.size() + 1; k <= K; ++k)
      m.push_back(std::max(m.empty() ? 0 : m.back(), crt_line_elements(k, kTiers[t], false)));
    need = std::max(need, m[K - 1]);
  }
  return need;
}

const ResidueConst& residue_const(const CrtPlan& pl) {
  ready();
  return g_class[pl.cls].rc;
}
const CrtConst& crt_const(const CrtPlan& pl) {
  ready();
  return g_class[pl.cls].cc[pl.n];
}

}  // namespace negf
