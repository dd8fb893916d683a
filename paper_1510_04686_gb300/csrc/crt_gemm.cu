// Tensor-core complex GEMM (tcgen05 + TMA + TMEM) on residues modulo small integers.
// See crt_gemm.cuh for the arithmetic; this file holds the MMA kernel and its host launcher.
#include <cuda_bf16.h>

#include <algorithm>
#include <atomic>

#include "crt_gemm.cuh"
#include "crt_residue.cuh"
#include "f32x2.cuh"
#include "profile.cuh"
#include "tc_common.cuh"

namespace negf {
namespace {

// warps 0-15 epilogue (four per scheduler hide each other's latencies), warp 16 TMA producer, warp
// 17 MMA issuer, warps 18-19 idle (they complete the warpgroup that gives its registers to the
// epilogue)
constexpr int kThreads = 640;
constexpr int kEpiWarps = 16;
constexpr int kRegsLaunch = 96;  // 65536 / 640, rounded down to a multiple of 8
constexpr int kRegsEpi = 112, kRegsIssue = 32;
static_assert(4 * kRegsEpi + kRegsIssue <= 5 * kRegsLaunch, "register split of the warpgroups");

// Flops of the launches made while profiling is on: [0] algorithmic complex 8 M N K of the
// active items, [1] issued BF16 MMA flops (padded tiles, computed slice products).
__device__ double g_crt_prof[2];

// ------------------------------------------------------------------ reconstruction
constexpr float kMagic = 12582912.0f;           // 1.5 * 2^23
constexpr uint32_t kMagicBits = 0x4B400000u;    // its bit pattern; x + kMagic has kMagicBits + x
// x modulo p, balanced to within one unit, for two integers |x| <= 2^24
__device__ __forceinline__ f2 residue2(f2 x, f2 invp, f2 negp) {
  const f2 magic = pack2(kMagic, kMagic), unmagic = pack2(-kMagic, -kMagic);
  return fma2(add2(fma2(x, invp, magic), unmagic), negp, x);
}
// (signed 64-bit binary fraction) * 2^eo as FP64, rounded once, with 32-bit integer operations only
// (FP64 arithmetic is scarce on this GPU).  Results below the normal range become 0, above it
// infinite; eo at kNonFinite / 2 or more marks a line that held an infinity or NaN.
__device__ __forceinline__ double from_fraction(unsigned long long f, int eo) {
  const uint32_t sign = (uint32_t)(f >> 32) & 0x80000000u;
  const unsigned long long a = sign ? 0ull - f : f;
  uint32_t hi = (uint32_t)(a >> 32), lo = (uint32_t)a;
  int e = eo + 1021;
  if (hi == 0) {
    hi = lo;
    lo = 0;
    e -= 32;
  }
  const int lz = __clz((int)hi) & 31;
  e -= lz;  // biased exponent less one: the mantissa below carries the implicit bit
  hi = __funnelshift_l(lo, hi, lz);
  lo <<= lz;
  const uint32_t up = (lo >> 10) & 1u;  // round to nearest at bit 10
  uint32_t mlo = __funnelshift_r(lo, hi, 11);
  uint32_t mhi = (hi >> 11) + ((uint32_t)e << 20);
  const unsigned long long m = ((unsigned long long)mhi << 32 | mlo) + up;
  mhi = (uint32_t)(m >> 32) | sign;
  mlo = (uint32_t)m;
  if ((uint32_t)e >= 2046u || hi == 0) {  // outside the normal range, or zero
    mlo = 0;
    if (eo >= kNonFinite / 2)
      mhi = 0x7FF80000u;
    else
      mhi = (e < 0 || hi == 0) ? 0u : (sign | 0x7FF00000u);
  }
  return __hiloint2double((int)mhi, (int)mlo);
}
// A signed fraction times m 2^-64
__device__ __forceinline__ unsigned long long mul_fraction(unsigned long long f,
                                                           unsigned long long m) {
  const unsigned long long h = __umul64hi((long long)f < 0 ? 0ull - f : f, m);
  return (long long)f < 0 ? 0ull - h : h;
}
// Two complex entries (32 bytes) of a row at once, for 32-byte aligned addresses.
__device__ __forceinline__ void load2(const z64* p, z64* v) {
  asm volatile("ld.global.v4.f64 {%0, %1, %2, %3}, [%4];"
               : "=d"(v[0].re), "=d"(v[0].im), "=d"(v[1].re), "=d"(v[1].im)
               : "l"(p));
}
__device__ __forceinline__ void store2(z64* p, const z64* v) {
  asm volatile("st.global.v4.f64 [%0], {%1, %2, %3, %4};" ::"l"(p), "d"(v[0].re), "d"(v[0].im),
               "d"(v[1].re), "d"(v[1].im)
               : "memory");
}
// Whether both rows' entries at even columns are 32-byte aligned for every item.
__device__ __forceinline__ bool pairs_aligned(const void* p, long long stride, int ld) {
  return ((reinterpret_cast<uintptr_t>(p) & 31) | (uintptr_t)((stride | ld) & 1)) == 0;
}

// ------------------------------------------------------------------ MMA kernel
// One tile: 128 rows x NT columns of complex outputs.  For every modulus and K part two real
// products u and v (kind::f16, exact in the FP32 accumulators, TMEM columns [0, NT) and
// [NT, 2 NT)); the epilogue reduces both modulo p and adds s re[l], t im[l] to the 64-bit
// fractions of Re and Im.  Real fractions live in registers, imaginary ones in TMEM columns
// [2 NT, 4 NT) as (low, high) pairs.  While the epilogue works on one accumulator the MMAs fill the other.
//
// Persistent: CTAs walk the tiles of all items in turn, the K chunks of all products and
// tiles run through one ring of stages without draining it, so the next tile's first products
// overlap this tile's final pass.
//
// What bounds it (64 items of 400^3, 48-bit): 421 us, where digit slices took 1204 us.  A
// 128 x 128 tile takes 50 us for its 24 products, of which the tensor core is busy 20; with the
// epilogue switched off the loads and MMAs alone take 45 (25 KB per 64-wide K chunk, 95 KB/us
// into each SM), so the tile is as large as the fractions' 16 bytes per output allow: registers
// hold Re, TMEM holds Im and both accumulators.  One CTA per tile: CTA pairs (cta_group::2) load
// half of B each, but their hand-overs cross SMs and cost more (499 us).  Sixteen epilogue warps
// instead of eight keep the integer multiply-adds of the reconstruction (the busiest pipe of the
// epilogue) behind the MMAs; one elected lane issues TMA and MMA (elect.sync instead of a test of
// the lane number took the MMA issue from 479 to 360 us per 76 items).
template <int NT, bool HP>
struct Cfg {
  static constexpr int kABox = kBM * kKC * 2;
  static constexpr int kBBox = NT * kKC * 2;
  static constexpr int kChunk = kABox + kBBox;
  // K chunks per stage.  Narrow tiles have little to do between a stage's barriers: two chunks per
  // stage take 3.5 % less time for 37 items of 333 x 217 x 591 (418 us now).  Wide ones need the stages
  // (64 items of 400^3, 731 us now, 3 % more with two chunks); nor do the correction sums leave the
  // issuer waiting (2 % more).
  static constexpr int kPer = NT <= 64 && !HP ? 2 : 1;
  static constexpr int kStage = kPer * kChunk;
  static constexpr int kStages = std::min(10, (227 * 1024 - 1280) / kStage);
  static_assert(kBBox % 1024 == 0, "stages keep the 1024-byte alignment of the swizzle");
  static constexpr int kSmem = kStages * kStage + 1024 + 256;  // + align + barriers
  static_assert((2 * kStages + 4) * 8 + 16 <= 256, "barrier space");
  static_assert(kSmem <= 227 * 1024, "shared memory of one CTA");
};

// The tiles of a launch.  An item's rows are dealt out evenly to its row tiles and its columns to
// its column tiles: all CTAs then load the same amount, which is what bounds them, instead of most
// loading full tiles and the last ones a remainder.
struct Tiles {
  int m, n, items;  // row tiles and column tiles of an item, items
  int rows;         // rows per tile (<= 128)
  int cols;         // columns per tile (<= NT)
};

template <int NT, bool HP>
__global__ void __launch_bounds__(kThreads, 1)
    k_crt_gemm(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB,
              const __grid_constant__ CrtConst crt, int n_mod, int parts, int part_k16, int k16,
              Tiles tiles, int M, int N, int Kc, const int32_t* __restrict__ eA,
              const int32_t* __restrict__ eB, const int32_t* __restrict__ zidxA, int zmodeA,
              const int32_t* __restrict__ zidxB, int zmodeB, z64 alpha, z64 beta, z64 gamma,
              BM<double> C, BMc<double> D, int add_identity, const int32_t* active, int32_t* err,
              float* rmax, int count_flops) {
  using CF = Cfg<NT, HP>;
  constexpr int kStages = CF::kStages;
  constexpr int kCols = NT / 4;            // columns per epilogue warp
  constexpr int kFin = 4;                  // columns per round of the final pass
  static_assert(kCols % 8 == 0, "epilogue chunks");
  constexpr uint32_t kTmemCols = 512;      // 4 NT <= 512
  static_assert(4 * NT <= 512 && NT % 32 == 0, "TMEM budget, MMA shapes");
  static_assert(!HP || NT <= 64, "registers of the correction sums");
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem = reinterpret_cast<unsigned char*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + kStages * CF::kStage);
  uint64_t* empty = full + kStages;
  uint64_t* accfull = empty + kStages;
  uint64_t* accempty = accfull + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(accempty + 2);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int per_item = tiles.m * tiles.n;
  const int n_tiles = per_item * tiles.items;
  const int n_steps = n_mod * parts;  // (modulus, K part) pairs, the parts of a modulus in turn

  if (threadIdx.x == 0) {
    for (int i = 0; i < kStages; ++i) mbar_init(&full[i], 1);
    for (int i = 0; i < kStages; ++i) mbar_init(&empty[i], 1);
    for (int i = 0; i < 2; ++i) {
      mbar_init(&accfull[i], 1);
      mbar_init(&accempty[i], kEpiWarps);  // one arrival per epilogue warp
    }
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == kEpiWarps + 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tmem_slot)), "r"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    tc_fence_before();
  }
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  if (warp >= kEpiWarps) {
  asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsIssue));
  if (warp == kEpiWarps) {
    // ---------------- TMA producer: the K chunks of u and v of every step of every tile
    if (elect_one()) {
      const uint32_t bytes = (uint32_t)((tiles.rows + tiles.cols) * kKC * 2);
      int stage = 0;
      uint32_t phase = 0;
      for (int t = blockIdx.x; t < n_tiles && !*abort_flag; t += gridDim.x) {
        const int p = t / per_item, r = t - p * per_item;
        if (active && !active[p]) continue;
        const int m0 = (r % tiles.m) * tiles.rows, n0 = (r / tiles.m) * tiles.cols;
        // residue set of this batch item: its own (mode 0), the indexed one (1) or the shared (2)
        const int zA = (zmodeA == 0 ? p : (zmodeA == 1 ? zidxA[p] : 0)) * 2 * n_mod;
        const int zB = (zmodeB == 0 ? p : (zmodeB == 1 ? zidxB[p] : 0)) * 2 * n_mod;
        bool ok = true;
        for (int h = 0; ok && h < 2 * n_mod * parts; ++h) {
          // product h: modulus h / (2 parts), part, then u or v
          const int step = h >> 1, mod = step / parts, part = step - mod * parts;
          const int z = 2 * mod + (h & 1);
          const int lo = part * part_k16, hi = min(k16, lo + part_k16);
          for (int kc = lo; kc < hi; kc += CF::kPer * kKC / 16) {
            if (!mbar_wait(&empty[stage], phase ^ 1, abort_flag)) {
              ok = false;
              break;
            }
            unsigned char* st = smem + stage * CF::kStage;
            const bool two = CF::kPer == 2 && hi - kc > kKC / 16;
            mbar_expect_tx(&full[stage], two ? 2 * bytes : bytes);
            tma_load_3d(st, &mapA, &full[stage], kc * 16, m0, zA + z);
            tma_load_3d(st + CF::kABox, &mapB, &full[stage], kc * 16, n0, zB + z);
            if (two) {
              st += CF::kChunk;
              tma_load_3d(st, &mapA, &full[stage], kc * 16 + kKC, m0, zA + z);
              tma_load_3d(st + CF::kABox, &mapB, &full[stage], kc * 16 + kKC, n0, zB + z);
            }
            if (++stage == kStages) {
              stage = 0;
              phase ^= 1;
            }
          }
        }
      }
    }
  } else if (warp == kEpiWarps + 1) {
    // ---------------- MMA issuer 
    if (elect_one()) {
      constexpr uint32_t idesc = idesc_bf16(kBM, NT);
      int stage = 0;
      uint32_t phase = 0;
      uint32_t use = 0;  // products issued so far: buffer use & 1
      for (int t = blockIdx.x; t < n_tiles && !*abort_flag; t += gridDim.x) {
        const int p = t / per_item;
        if (active && !active[p]) continue;
        bool ok = true;
        for (int h = 0; ok && h < 2 * n_steps; ++h, ++use) {
          const int buf = use & 1;
          // the buffer's previous product must have been read out
          if (use >= 2 && !mbar_wait(&accempty[buf], ((use >> 1) - 1) & 1, abort_flag)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t dcol = tmem + (uint32_t)(buf * NT);
          const int part = (h >> 1) % parts;
          const int lo = part * part_k16, hi = min(k16, lo + part_k16);
          uint32_t acc_on = 0;
          for (int kc = lo; kc < hi; kc += CF::kPer * kKC / 16) {
            if (!mbar_wait(&full[stage], phase, abort_flag)) {
              ok = false;
              break;
            }
            tc_fence_after();
            const uint32_t a = smem_u32(smem + stage * CF::kStage), b = a + CF::kABox;
            const uint64_t da = sw128_desc(a), db = sw128_desc(b);
            const int nk = hi - kc;  // K steps left in this part
#pragma unroll
            for (int k = 0; k < CF::kPer * kKC / 16; ++k) {
              // one K step is 32 bytes along the swizzled row of its chunk
              constexpr int kPerChunk = kKC / 16;
              const uint64_t at = k / kPerChunk * (CF::kChunk >> 4) + k % kPerChunk * 2;
              if (k < nk) mma_bf16(dcol, da + at, db + at, idesc, k == 0 ? acc_on : 1u);
            }
            acc_on = 1;
            mma_commit(&empty[stage]);
            if (++stage == kStages) {
              stage = 0;
              phase ^= 1;
            }
          }
          if (!ok) break;
          mma_commit(&accfull[buf]);
        }
      }
    }
  }
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kRegsEpi));
    // ---------------- epilogue: warp w owns TMEM lanes 32 (w % 4) .. + 31 (tile rows) and the
    // NT / 4 columns from (NT / 4) (w / 4)
    const int q = warp & 3;
    const int cbase = (warp >> 2) * kCols;
    const uint32_t lane_off = (uint32_t)(q * 32) << 16;
    const uint32_t t_u = tmem + lane_off + (uint32_t)cbase, t_v = t_u + NT;
    const uint32_t t_im = tmem + lane_off + 2 * NT + 2 * (uint32_t)cbase;  // (low, high) pairs
    const int cls_alpha = coef_class(alpha), cls_beta = coef_class(beta);
    const int cls_gamma = D.p ? coef_class(gamma) : 0;
    const bool want_max = rmax != nullptr;
    // alpha A B alone, and C (and D) addressable as 32-byte pairs of columns
    const bool plain = cls_alpha == 1 && !cls_beta && !cls_gamma && !add_identity;
    const bool wide = pairs_aligned(C.p, C.stride, C.ld) &&
                      (!cls_gamma || pairs_aligned(D.p, D.stride, D.ld));
    // the fractions start from minus what the magic bias of every step's s and t adds
    unsigned long long re0 = 0, im0 = 0;
    for (int l = 0; l < n_mod; ++l) {
      re0 -= (unsigned long long)kMagicBits * crt.re[l];
      im0 -= (unsigned long long)kMagicBits * crt.im[l];
    }
    re0 *= (unsigned long long)parts;
    im0 *= (unsigned long long)parts;
    uint32_t use = 0;  // steps done: parity of both accumulators' barriers
    auto release = [&](int buf) {
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&accempty[buf]);
    };
    for (int t = blockIdx.x; t < n_tiles; t += gridDim.x) {
      const int p = t / per_item, r = t - p * per_item;
      if (active && !active[p]) continue;
      // rows and columns of this warp
      const int m0 = (r % tiles.m) * tiles.rows + q * 32;
      const int m_end = min(M, m0 - q * 32 + tiles.rows);
      const int nb = (r / tiles.m) * tiles.cols, n0 = nb + cbase;
      const int n_end = min(N, nb + tiles.cols);
      if (count_flops && warp == 0 && lane == 0) {
        // this CTA's share of the launch: algorithmic complex flops of its outputs and the
        // issued BF16 MMA flops of its 128 rows
        const int rows = max(0, m_end - m0), cols = max(0, min(tiles.cols, N - n0));
        atomicAdd(&g_crt_prof[0], 8.0 * rows * cols * (double)Kc);
        atomicAdd(&g_crt_prof[1], 2.0 * kBM * NT * 16.0 * k16 * 2.0 * n_mod);
      }
      // line exponents of this lane's row and of column n0 + lane, fetched ahead of their use
      const int zA = zmodeA == 0 ? p : (zmodeA == 1 ? zidxA[p] : 0);
      const int zB = zmodeB == 0 ? p : (zmodeB == 1 ? zidxB[p] : 0);
      const int em = m0 + lane < m_end ? crt.expo + eA[(long long)zA * M + m0 + lane] : 0;
      const int en = n0 + lane < n_end ? eB[(long long)zB * N + n0 + lane] : 0;
      unsigned long long re[kCols];
      float cre[kCols], cim[kCols];  // HP only
#pragma unroll
      for (int j = 0; j < kCols; ++j) {
        re[j] = re0;
        if constexpr (HP) cre[j] = cim[j] = 0.0f;
      }
#pragma unroll 1
      for (int c0 = 0; c0 < kCols; c0 += 8) {
        uint32_t im[16];
#pragma unroll
        for (int j = 0; j < 16; ++j) im[j] = (uint32_t)(j & 1 ? im0 >> 32 : im0);
        tmem_st16(t_im + 2 * c0, im);
      }
      tmem_st_wait();
      bool ok = __all_sync(0xffffffffu, !*abort_flag);
      int part = 0, mod = 0;
#pragma unroll 1
      for (int step = 0; step < n_steps; ++step, ++use) {
        const f2 invp = pack2(crt.invp[mod], crt.invp[mod]);
        const f2 negp = pack2(crt.negp[mod], crt.negp[mod]);
        const unsigned long long gre = crt.re[mod], gim = crt.im[mod];
        const float hre = crt.hre[mod], him = crt.him[mod];
        if (++part == parts) {
          part = 0;
          ++mod;
        }
        // u modulo p, packed as BF16 pairs (integers up to 256 are exact)
        if (!ok || !mbar_wait_warp(&accfull[0], use & 1, abort_flag)) {
          ok = false;
          break;
        }
        tc_fence_after();
        uint32_t up[kCols / 2];
#pragma unroll
        for (int c0 = 0; c0 < kCols; c0 += 8) {
          uint32_t x[8];
          tmem_ld8(t_u + c0, x);
          tmem_ld_wait();
#pragma unroll
          for (int j = 0; j < 8; j += 2) {
            float a, b;
            unpack2(residue2(pack2(__uint_as_float(x[j]), __uint_as_float(x[j + 1])), invp, negp),
                    a, b);
            const __nv_bfloat162 w = __floats2bfloat162_rn(a, b);
            up[(c0 + j) / 2] = *reinterpret_cast<const uint32_t*>(&w);
          }
        }
        release(0);
        // v modulo p, and the step's contribution to both fractions
        if (!mbar_wait_warp(&accfull[1], use & 1, abort_flag)) {
          ok = false;
          break;
        }
        tc_fence_after();
#pragma unroll
        for (int c0 = 0; c0 < kCols; c0 += 8) {
          uint32_t x[8], im[16];
          tmem_ld8(t_v + c0, x);
          tmem_ld16(t_im + 2 * c0, im);
          tmem_ld_wait();
#pragma unroll
          for (int j = 0; j < 8; j += 2) {
            const f2 v = residue2(pack2(__uint_as_float(x[j]), __uint_as_float(x[j + 1])), invp,
                                  negp);
            const uint32_t pk = up[(c0 + j) / 2];
            const f2 um = add2(pack2(__uint_as_float(pk << 16), __uint_as_float(pk & 0xFFFF0000u)),
                               pack2(kMagic, kMagic));
            float s0, s1, d0, d1;
            unpack2(add2(um, v), s0, s1);
            unpack2(fma2(v, pack2(-1.0f, -1.0f), um), d0, d1);
            re[c0 + j] += __float_as_uint(s0) * gre;
            re[c0 + j + 1] += __float_as_uint(s1) * gre;
            const unsigned long long i0 =
                ((unsigned long long)im[2 * j + 1] << 32 | im[2 * j]) + __float_as_uint(d0) * gim;
            const unsigned long long i1 =
                ((unsigned long long)im[2 * j + 3] << 32 | im[2 * j + 2]) +
                __float_as_uint(d1) * gim;
            im[2 * j] = (uint32_t)i0;
            im[2 * j + 1] = (uint32_t)(i0 >> 32);
            im[2 * j + 2] = (uint32_t)i1;
            im[2 * j + 3] = (uint32_t)(i1 >> 32);
            if constexpr (HP) {
              cre[c0 + j] = fmaf(s0 - kMagic, hre, cre[c0 + j]);
              cre[c0 + j + 1] = fmaf(s1 - kMagic, hre, cre[c0 + j + 1]);
              cim[c0 + j] = fmaf(d0 - kMagic, him, cim[c0 + j]);
              cim[c0 + j + 1] = fmaf(d1 - kMagic, him, cim[c0 + j + 1]);
            }
          }
          tmem_st16(t_im + 2 * c0, im);
        }
        tmem_st_wait();
        release(1);
      }
      if (!ok) {
        // a bounded wait gave up: this tile's outputs are NaN, so that the caller's finite checks
        // see the failure instead of stale values
        const double qnan = __longlong_as_double(0x7FF8000000000000LL);
        const int m = m0 + lane;
        if (m < m_end) {
          z64* crow = bat(C, p) + (long long)m * C.ld;
          for (int n = n0; n < n0 + kCols && n < n_end; ++n) crow[n] = mkc(qnan, qnan);
        }
        continue;
      }
      // ---- final pass: each lane converts its row's outputs to FP64, four columns per round,
      // and writes them as 32-byte sectors where the layout allows.  re[] moves down by four per
      // round, so that one copy of the code serves them all.
      unsigned long long omax = 0ull;  // largest |Re|, |Im| this thread stores, as bits
      const int m = m0 + lane;
      z64* crow = bat(C, p) + (long long)m * C.ld;
      const z64* drow = cls_gamma ? bat(D, p) + (long long)m * D.ld : nullptr;
      const bool pairs = wide && ((n0 & 1) == 0);
#pragma unroll 1
      for (int c0 = 0; c0 < kCols; c0 += kFin) {
        if (n0 + c0 >= n_end) break;
        uint32_t im[2 * kFin];
        tmem_ld8(t_im + 2 * c0, im);
        tmem_ld_wait();
#pragma unroll
        for (int j = 0; j < kFin; j += 2) {
          const int n = n0 + c0 + j;
          const int sh0 = em + __shfl_sync(0xffffffffu, en, c0 + j);
          const int sh1 = em + __shfl_sync(0xffffffffu, en, c0 + j + 1);
          if (m < m_end && n < n_end) {
            const bool two = n + 1 < n_end;
            z64 o[2];
            unsigned long long i0 = (unsigned long long)im[2 * j + 1] << 32 | im[2 * j];
            unsigned long long i1 = (unsigned long long)im[2 * j + 3] << 32 | im[2 * j + 2];
            if constexpr (HP) {  // the corrections, in units of the last place
              re[j] += (long long)__float2int_rn(cre[j]);
              re[j + 1] += (long long)__float2int_rn(cre[j + 1]);
              i0 += (long long)__float2int_rn(cim[j]);
              i1 += (long long)__float2int_rn(cim[j + 1]);
              re[j] = mul_fraction(re[j], crt.mant);
              re[j + 1] = mul_fraction(re[j + 1], crt.mant);
              i0 = mul_fraction(i0, crt.mant);
              i1 = mul_fraction(i1, crt.mant);
            }
            o[0] = mkc(from_fraction(re[j], sh0), from_fraction(i0, sh0));
            o[1] = mkc(from_fraction(re[j + 1], sh1), from_fraction(i1, sh1));
            if (!plain) {
              z64 c[2], d[2];
              c[0] = c[1] = d[0] = d[1] = mkc(0.0, 0.0);
              if (pairs && two) {
                if (cls_beta) load2(crow + n, c);
                if (cls_gamma) load2(drow + n, d);
              } else {
                if (cls_beta) {
                  c[0] = crow[n];
                  if (two) c[1] = crow[n + 1];
                }
                if (cls_gamma) {
                  d[0] = drow[n];
                  if (two) d[1] = drow[n + 1];
                }
              }
#pragma unroll
              for (int i = 0; i < 2; ++i) {
                o[i] = coef_mul(cls_alpha, alpha, o[i]);
                if (cls_beta) o[i] = o[i] + coef_mul(cls_beta, beta, c[i]);
                if (cls_gamma) o[i] = o[i] + coef_mul(cls_gamma, gamma, d[i]);
                if (add_identity && n + i == m) o[i].re += 1.0;
              }
            }
            if (pairs && two) {
              store2(crow + n, o);
            } else {
              crow[n] = o[0];
              if (two) crow[n + 1] = o[1];
            }
            if (want_max) {
              omax = max(omax, max(abs_bits(o[0].re), abs_bits(o[0].im)));
              if (two) omax = max(omax, max(abs_bits(o[1].re), abs_bits(o[1].im)));
            }
          }
        }
#pragma unroll
        for (int j = 0; j + kFin < kCols; ++j) {
          re[j] = re[j + kFin];
          if constexpr (HP) {
            cre[j] = cre[j + kFin];
            cim[j] = cim[j + kFin];
          }
        }
      }
      if (want_max) {  // per-item max |output| (non-negative floats order like their bit patterns)
        const float wm = warp_max_f((float)__longlong_as_double((long long)omax));
        if (lane == 0 && wm > 0.0f)
          atomicMax(reinterpret_cast<unsigned int*>(rmax + p), __float_as_uint(wm));
      }
    }
  }
  __syncthreads();
  land_in_flight(abort_flag);
  if (warp == kEpiWarps + 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                 "r"(kTmemCols)
                 : "memory");
  }
  if (threadIdx.x == 0 && *abort_flag && err) atomicExch(err, 1);
}

// ------------------------------------------------------------------ host side
inline int ceil_div(int x, int m) { return (x + m - 1) / m; }

struct GemmArgs {
  int P, M, N, K;
  CrtPlan plan;
  void *resA, *resB;             // residue planes and their numbers, L: row length
  long long planesA, planesB;
  int L;
  const int32_t *expA, *expB, *zA, *zB;
  int zmA, zmB;
  z64 alpha, beta, gamma;
  BM<double> C;
  BMc<double> D;
  bool add_identity;
  const int32_t* active;
  int32_t* err;
  float* rmax;
};

// SMs of the current device (the persistent grid: one CTA per SM).
int sm_count() {
  static std::atomic<int> cached[32];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 152;
  int n = cached[dev & 31].load();
  if (n == 0) {
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 152;
    cached[dev & 31].store(n);
  }
  return n;
}

template <int NT, bool HP>
cudaError_t launch_crt(cudaStream_t s, const GemmArgs& a) {
  using CF = Cfg<NT, HP>;
  static std::atomic<unsigned> attr{0};
  cudaError_t e =
      set_smem_once(attr, reinterpret_cast<const void*>(&k_crt_gemm<NT, HP>), CF::kSmem);
  if (e != cudaSuccess) return e;
  Tiles tiles{ceil_div(a.M, kBM), ceil_div(a.N, NT), a.P, 0, 0};
  tiles.rows = ceil_div(a.M, tiles.m);
  tiles.cols = ceil_div(a.N, tiles.n);
  const long long n_tiles = (long long)tiles.m * tiles.n * tiles.items;
  if (n_tiles > 0x7FFFFFFFll - 4096) return cudaErrorInvalidValue;
  CUtensorMap mA, mB;
  if (!make_map(&mA, a.resA, a.L, a.M, a.planesA, tiles.rows) ||
      !make_map(&mB, a.resB, a.L, a.N, a.planesB, tiles.cols))
    return cudaErrorInvalidValue;
  const unsigned grid = (unsigned)std::min<long long>(n_tiles, sm_count());
  prof_begin(s, PROF_TC_GEMM);
  k_crt_gemm<NT, HP><<<grid, kThreads, CF::kSmem, s>>>(
      mA, mB, crt_const(a.plan), a.plan.n, a.plan.parts, a.plan.k16, ceil_div(a.K, 16), tiles, a.M,
      a.N, a.K, a.expA, a.expB, a.zA, a.zmA, a.zB, a.zmB, a.alpha, a.beta, a.gamma, a.C, a.D,
      a.add_identity ? 1 : 0, a.active, a.err, a.rmax, profiling_on() ? 1 : 0);
  prof_end(s, PROF_TC_GEMM);
  count_launch();
  return cudaGetLastError();
}

// Tile widths.  A tile's time at K = 400 is a fixed part (its rows of A, the hand-overs between
// the roles) plus a part per column, measured as 2.50, 2.02 and 1.63 us per product for 128, 96
// and 64 columns: about 57 + NT.  The width with the least time over the waves of one tile per SM
// is taken, so wide tiles serve the batches and narrow ones keep a small product on all SMs.
constexpr int kWidths[] = {128, 96, 64, 32};

int pick_width(int P, int M, int N, bool hp) {
  int best = 64;
  long long cost = -1;
  for (int nt : kWidths) {
    if (hp && nt > 64) continue;
    const long long tiles = (long long)ceil_div(M, kBM) * ceil_div(N, nt) * P;
    const long long sms = sm_count();
    const long long c = (tiles + sms - 1) / sms * (57 + nt);
    if (cost < 0 || c < cost) {
      cost = c;
      best = nt;
    }
  }
  return best;
}

}  // namespace

cudaError_t crt_prof_flops(double* alg, double* hw) {
  double v[2] = {0.0, 0.0};
  cudaError_t e = cudaMemcpyFromSymbol(v, g_crt_prof, sizeof(v));
  *alg = v[0];
  *hw = v[1];
  return e;
}

cudaError_t crt_prof_reset() {
  const double z[2] = {0.0, 0.0};
  return cudaMemcpyToSymbol(g_crt_prof, z, sizeof(z));
}

size_t crt_ws_bytes(int P, int M, int N, int K, int bits) {
  size_t off = 0;
  CrtWs w;
  crt_ws_carve(nullptr, off, P, M, N, K, bits, false, w);
  return off;
}

void crt_ws_carve(char* base, size_t& off, int P, int M, int N, int K, int bits, bool shorter,
                  CrtWs& w) {
  const size_t line = crt_line_elements(K, bits, shorter);
  auto take = [&](size_t bytes) -> void* {
    size_t a = (off + 1023) & ~size_t(1023);
    off = a + bytes;
    return base ? base + a : nullptr;
  };
  w.linesA = (size_t)P * M;
  w.linesB = (size_t)P * N;
  w.elemsA = w.linesA * line;
  w.elemsB = w.linesB * line;
  w.err = static_cast<int32_t*>(take(256));  // first, so that its place does not depend on P
  w.resA = take(w.elemsA * 2);
  w.resB = take(w.elemsB * 2);
  w.expA = static_cast<int32_t*>(take(w.linesA * 4));
  w.expB = static_cast<int32_t*>(take(w.linesB * 4));
}

cudaError_t crt_gemm(cudaStream_t s, int P, int M, int N, int K, z64 alpha, BMc<double> A,
                    int opA, BMc<double> B, int opB, z64 beta, BM<double> C, z64 gamma,
                    BMc<double> D, bool add_identity, const int32_t* active, const CrtWs& ws,
                    int bits, int n_distinct, float* rmax, Kept* kept) {
  if (P <= 0 || M <= 0 || N <= 0 || K <= 0) return cudaSuccess;
  // Operands shared by all items (stride 0) or selected per item from n_distinct matrices are
  // converted once per distinct matrix; the kernel maps each item to its residue set.
  auto plan_op = [&](BMc<double>& X, const int32_t*& z, int& mode, int& items) {
    z = nullptr;
    mode = 0;
    items = P;
    if (!X.idx && X.stride == 0) {
      mode = 2;
      items = 1;
    } else if (X.idx && n_distinct > 0 && n_distinct <= P) {
      mode = 1;
      z = X.idx;
      items = n_distinct;
      X.idx = nullptr;
    }
  };
  GemmArgs g;
  int PA = P, PB = P;
  plan_op(A, g.zA, g.zmA, PA);
  plan_op(B, g.zB, g.zmB, PB);
  // with a shared operand the active mask cannot gate the conversion by item
  const int32_t* actA = g.zmA == 0 ? active : nullptr;
  const int32_t* actB = g.zmB == 0 ? active : nullptr;
  if (!crt_plan(K, bits, &g.plan))
    return cudaErrorInvalidValue;  // K beyond the tier's range (callers check tc_supports_k)
  const int L = residue_ld(K);
  const size_t line = 2 * (size_t)g.plan.n * L, linesA = (size_t)PA * M, linesB = (size_t)PB * N;
  if (linesA > ws.linesA || linesB > ws.linesB || linesA * line > ws.elemsA ||
      linesB * line > ws.elemsB)
    return cudaErrorInvalidValue;
  __nv_bfloat16* ra = static_cast<__nv_bfloat16*>(ws.resA);
  __nv_bfloat16* rb = static_cast<__nv_bfloat16*>(ws.resB);
  const KeptOperand ka{A.p,  ra,  g.zA ? g.zA : A.idx, actA, A.stride,   A.ld,
                       opA, M, K, PA, g.plan.cls, 2 * g.plan.n + g.plan.hp};
  const KeptOperand kb{B.p,  rb,  g.zB ? g.zB : B.idx, actB, B.stride,   B.ld,
                       opB, N, K, PB, g.plan.cls, 2 * g.plan.n + g.plan.hp};
  const bool haveA = kept && (kept->reuse & REUSE_A) && kept->a == ka;
  const bool haveB = kept && (kept->reuse & REUSE_B) && kept->b == kb;
  prof_begin(s, PROF_SLICE);
  // a row of op(A) is a column of A in memory for op T/C; a column of op(B) is a column of B for
  // op N
  cudaError_t e = cudaSuccess;
  if (!haveA)
    e = launch_residues(s, g.plan, g.plan.alpha_a, g.plan.hp ? 1.0 : crt_const(g.plan).sigma, PA, M,
                        K, L, A, opA, opA != OP_N, ra, ws.expA, actA);
  if (e != cudaSuccess) return e;
  if (!haveB)
    e = launch_residues(s, g.plan, g.plan.alpha_b, 1.0, PB, N, K, L, B, opB, opB == OP_N, rb,
                        ws.expB, actB);
  prof_end(s, PROF_SLICE);
  count_launch(!haveA + !haveB);
  if (e != cudaSuccess) return e;
  if (kept) *kept = Kept{ka, kb, 0};
  // correction sums of the fractions: their registers limit the tile to 64
  const bool hp = g.plan.hp;
  const int nt = pick_width(P, M, N, hp);
  g.resA = ra;
  g.resB = rb;
  g.planesA = (long long)PA * 2 * g.plan.n;
  g.planesB = (long long)PB * 2 * g.plan.n;
  g.L = L;
  g.P = P;
  g.M = M;
  g.N = N;
  g.K = K;
  g.expA = ws.expA;
  g.expB = ws.expB;
  g.alpha = alpha;
  g.beta = beta;
  g.gamma = gamma;
  g.C = C;
  g.D = D;
  g.add_identity = add_identity;
  g.active = active;
  g.err = ws.err;
  g.rmax = rmax;
  if (hp) return nt == 64 ? launch_crt<64, true>(s, g) : launch_crt<32, true>(s, g);
  switch (nt) {
    case 128: return launch_crt<128, false>(s, g);
    case 96: return launch_crt<96, false>(s, g);
    case 64: return launch_crt<64, false>(s, g);
    default: return launch_crt<32, false>(s, g);
  }
}

}  // namespace negf
