// fv_fxsum.cuh -- sums of a few doubles on the integer pipe, exact with one
// rounding.
//
// GB300 retires two FP64 operations per SM per clock (an FP64 add of a warp
// holds the pipe for 16 clocks) but 64 integer operations on the ALU and as
// many integer multiply-adds on the FMA pipe, and the FP64 kernels leave both
// nearly idle.  The flux differences of a cell, sum_k (G_k+ - G_k-), are
// 2d - 1 FP64 adds per unknown; here they are one fixed-point accumulation:
// every term's 53-bit significand, shifted to the largest exponent of the
// terms with 28 bits to spare below it, is added into two 64-bit words (the
// upper 22 and the lower 31 bits of the significand apart, each by one signed
// 32 x 32 -> 64 multiply-add with +-2^shift, which shifts, applies the sign and
// accumulates at once), and the total is rounded once, to nearest even.
//
// The sum is exact before that rounding: where a term would lose bits (more
// than 28 binary orders below the largest; zeros, and what lies below 2^-1042,
// count as zero), or the exponents are near the ends of the range (infinities
// and NaN included), `ok` is false and the caller adds in FP64.  So the error is at most half an ulp of the result,
// where 2d - 1 roundings were before; the result does not depend on the order
// of the terms, and negating all terms negates it.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define FV_HD __host__ __device__ __forceinline__
#else
#define FV_HD inline
#endif

namespace fv {

// x << n with every n outside 0 .. 31 giving 0 (the shl instruction's rule).
FV_HD int32_t shl_clamped(int32_t x, int32_t n) {
#ifdef __CUDA_ARCH__
  int32_t r;
  asm("shl.b32 %0, %1, %2;" : "=r"(r) : "r"(x), "r"(n));
  return r;
#else
  return (uint32_t)n > 31u ? 0 : (int32_t)((uint32_t)x << n);
#endif
}
FV_HD int clz64(uint64_t x) {  // x != 0
#ifdef __CUDA_ARCH__
  return __clzll((long long)x);
#else
  return __builtin_clzll(x);
#endif
}

// Sum of the N terms, plus the first NP of them and minus the others, given
// as bit patterns (hi, lo).  N <= 8.
template <int N, int NP>
FV_HD void fx_sum(const uint32_t (&hi)[N], const uint32_t (&lo)[N], uint32_t& rhi, uint32_t& rlo,
                  bool& ok) {
  constexpr int kGuard = 28;
  uint32_t x[N];  // without the sign: exponent in the upper 11 bits
  uint32_t xm = 0;
#pragma unroll
  for (int i = 0; i < N; ++i) {
    x[i] = hi[i] + hi[i];
    xm = x[i] > xm ? x[i] : xm;
  }
  const int emax = (int)(xm >> 21);
  // terms below 2^(emax - 28), zeros excepted, would lose bits
  const uint32_t low = ((uint32_t)(emax - kGuard) << 21) - 1u;
  bool exact = true;
  int64_t A = 0, B = 0;
#pragma unroll
  for (int i = 0; i < N; ++i) {
    exact = exact && !(x[i] - 1u < low);
    const int k = (int)(x[i] >> 21) + (kGuard - emax);
    const int32_t sx = (int32_t)hi[i] >> 31;
    const int32_t sg = (i < NP ? sx : ~sx) | 1;
    const int32_t sp = shl_clamped(sg, k);  // +-2^k; 0 for a zero term
    const int32_t h22 = (int32_t)(((x[i] | (lo[i] >> 31)) & 0x1FFFFFu) | 0x200000u);
    const int32_t l31 = (int32_t)(lo[i] & 0x7FFFFFFFu);
    A += (int64_t)l31 * sp;
    B += (int64_t)h22 * sp;
  }
  ok = exact && (uint32_t)(emax - 64) < (uint32_t)(0x7F8 - 64);
  // total = B 2^31 + A  ->  sign and magnitude (b 2^31 + a, 0 <= a < 2^31)
  B += A >> 31;
  uint32_t a = (uint32_t)A & 0x7FFFFFFFu;
  const uint32_t sgn = (uint32_t)((uint64_t)B >> 63);
  const uint64_t m64 = 0ull - (uint64_t)sgn;
  a = ((a ^ (uint32_t)m64) & 0x7FFFFFFFu) + sgn;
  uint64_t b = ((uint64_t)B ^ m64) + (a >> 31);
  a &= 0x7FFFFFFFu;
  ok = ok && (b != 0 || a == 0);  // the sum within 53 bits of the largest term, or 0
  const int lz = b != 0 ? clz64(b) : 63;
  uint64_t w = b << lz;
  w |= ((uint64_t)a << 33) >> (64 - lz);
  // bits of a below w only break ties (lz >= 31: none)
  const bool rest = shl_clamped((int32_t)a, lz + 1) != 0;
  const uint32_t rem = ((uint32_t)w & 0x7FFu) | (rest ? 1u : 0u);
  uint64_t m = w >> 11;
  const uint32_t inc = rem + ((uint32_t)m & 1u) > 0x400u ? 1u : 0u;
  m += inc;
  // the implicit bit of m adds one to the exponent field
  const uint32_t ef = (uint32_t)(emax + 13 - lz);
  uint32_t h = (uint32_t)(m >> 32) + (ef << 20) + (sgn << 31);
  uint32_t l = (uint32_t)m;
  rhi = b != 0 ? h : 0u;
  rlo = b != 0 ? l : 0u;
}

}  // namespace fv
