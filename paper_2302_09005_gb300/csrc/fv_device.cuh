// fv_device.cuh -- device-side building blocks of the Rusanov patch kernels:
// Euler physics (Eq. 2, Eq. 5), bit-level helpers for exact maxima and
// positivity checks, and the compile-time patch geometry.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace fv {

// Status bits of the handle's device status word.
enum : unsigned int {
  ST_BAD_PATCH = 1u,
  ST_NONPHYSICAL = 2u,
  ST_TIMEOUT = 4u,
};

// ---------------------------------------------------------------------------
// Bit-level helpers.  A wave speed |u|+c is >= 0 or NaN.  With the sign bit
// cleared, the IEEE bit pattern orders non-negative values like the values
// themselves and puts every NaN above +inf, so maxima taken on the integer
// patterns are exact, order independent, and propagate NaN.  They run on the
// integer pipe, which keeps the FP64 pipe free.
// ---------------------------------------------------------------------------
// The mask is applied in inline PTX: written as C++, the compiler recognises
// "clear the sign bit" as |x| and spends an FP64 add on it.
__device__ __forceinline__ unsigned long long order_bits(double x) {
  unsigned long long r;
  asm("and.b64 %0, %1, 0x7FFFFFFFFFFFFFFF;" : "=l"(r) : "l"(__double_as_longlong(x)));
  return r;
}
__device__ __forceinline__ unsigned long long order_bits(float x) {
  unsigned int r;
  asm("and.b32 %0, %1, 0x7FFFFFFF;" : "=r"(r) : "r"(__float_as_uint(x)));
  return (unsigned long long)r;
}
// Value of a maximum taken on order_bits of type T, as a double.
template <typename T>
__device__ __forceinline__ double order_value(unsigned long long b);
template <>
__device__ __forceinline__ double order_value<double>(unsigned long long b) {
  return __longlong_as_double((long long)b);
}
template <>
__device__ __forceinline__ double order_value<float>(unsigned long long b) {
  return (double)__uint_as_float((unsigned int)b);
}
template <typename T>
__device__ __forceinline__ T max_by_bits(T a, T b);
template <>
__device__ __forceinline__ double max_by_bits<double>(double a, double b) {
  return order_bits(a) >= order_bits(b) ? a : b;
}
template <>
__device__ __forceinline__ float max_by_bits<float>(float a, float b) {
  return order_bits(a) >= order_bits(b) ? a : b;
}

// 0 < x < +inf (not NaN), tested on the bit pattern with integer ops.
__device__ __forceinline__ bool positive_finite(double x) {
  unsigned long long b = (unsigned long long)__double_as_longlong(x);
  return (b - 1ull) < 0x7FEFFFFFFFFFFFFFull;
}
__device__ __forceinline__ bool positive_finite(float x) {
  unsigned int b = __float_as_uint(x);
  return (b - 1u) < 0x7F7FFFFFu;
}

__device__ __forceinline__ unsigned long long warp_max_u64(unsigned long long v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    unsigned long long w = __shfl_xor_sync(0xFFFFFFFFu, v, o);
    v = w > v ? w : v;
  }
  return v;
}

// ---------------------------------------------------------------------------
// |x| and -x on the sign bit with integer operations: exact, and they keep
// the scarce FP64 pipe out of sign manipulations the compiler does not fold
// into a neighbouring instruction.
// ---------------------------------------------------------------------------
__device__ __forceinline__ double abs_t(double x) {
  return __hiloint2double(__double2hiint(x) & 0x7FFFFFFF, __double2loint(x));
}
__device__ __forceinline__ float abs_t(float x) { return fabsf(x); }
__device__ __forceinline__ double neg_t(double x) {
  return __hiloint2double(__double2hiint(x) ^ (int)0x80000000, __double2loint(x));
}
__device__ __forceinline__ float neg_t(float x) { return -x; }

// Explicitly rounded add, subtract and multiply: never contracted into an
// FMA, so an expression rounds the same way wherever it is inlined.
__device__ __forceinline__ double add_rn(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ float add_rn(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ double sub_rn(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ float sub_rn(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }

// ---------------------------------------------------------------------------
// The adds, subtracts and multiplies of the FP64 kernels as FMAs.  On GB300
// the FP64 pipe retires DFMA about 1.19 times faster than DADD or DMUL
// (measured: 0.60 vs 0.50 T instructions/s), and
//   a + b = fma(a, 1, b),   a - b = fma(b, -1, a),   a * b = fma(a, b, -0)
// hold bitwise (the product is exact, or the addend -0 leaves it as it is,
// and there is one rounding), signed zeros included.  The constants 1, -1
// and -0 come in as kernel arguments: a literal would let the compiler fold
// the FMA back into the slower instruction.  FP32 keeps plain operations
// (FADD and FMUL run at the FFMA rate).
// ---------------------------------------------------------------------------
template <typename T>
struct Arith {
  T one, mone, mzero;
  __device__ __forceinline__ T add(T a, T b) const { return add_rn(a, b); }
  __device__ __forceinline__ T sub(T a, T b) const { return sub_rn(a, b); }
  __device__ __forceinline__ T mul(T a, T b) const { return mul_rn(a, b); }
};
template <>
struct Arith<double> {
  double one, mone, mzero;
  __device__ __forceinline__ double add(double a, double b) const { return fma(a, one, b); }
  __device__ __forceinline__ double sub(double a, double b) const { return fma(b, mone, a); }
  __device__ __forceinline__ double mul(double a, double b) const { return fma(a, b, mzero); }
};
// A float as a double, exactly, with integer operations (sign; exponent
// rebased from 127 to 1023; the 23 fraction bits on top of the 52): the
// conversion instruction would run on the FP64 pipe, the scarce unit of this
// GPU.  Zero and subnormal floats give a signed zero (subnormals, below
// 1.2e-38, are flushed); infinities and NaNs keep their class.
__device__ __forceinline__ double widen_f32(float f) {
  const unsigned u = __float_as_uint(f);
  const unsigned e = (u >> 23) & 0xFFu, sign = u & 0x80000000u, m = u & 0x7FFFFFu;
  unsigned hi = sign | ((e + 896u) << 20) | (m >> 3);
  unsigned lo = u << 29;
  hi = e == 0u ? sign : hi;
  lo = e == 0u ? 0u : lo;
  hi = e == 255u ? (sign | 0x7FF00000u | (m >> 3)) : hi;
  return __hiloint2double((int)hi, (int)lo);
}
__device__ __forceinline__ double to_t(float f, double*) { return widen_f32(f); }
__device__ __forceinline__ float to_t(float f, float*) { return f; }

// The same operations with literal constants (the compiler may use plain
// adds and multiplies; the results are the same bits).
template <typename T>
__device__ __forceinline__ Arith<T> plain_arith() {
  return Arith<T>{T(1), T(-1), T(-0.0)};
}

// ---------------------------------------------------------------------------
// Reciprocal and square root, once per cell of the interior and face halo.
//
// FP64 is the scarce unit on GB300 (two FP64 lanes per SM), so the FP64 forms
// spend two FP64 operations each, on the last Newton step; everything before
// it runs in FP32 and integers, on pipes the FP64 kernels leave idle.  The
// argument's significand is split exactly into two floats fh + fl (fl up to
// bits of relative weight 2^-46); a float seed from the special-function
// unit gets a float correction from its residual, which FP32 fused
// multiply-adds give to all its bits:
//   1/a      y0 ~ 1/fh, e = 1 - fh y0 - fl y0, d = y0 (e + e^2);
//   sqrt(x)  s ~ fh rsqrt(fh), e = fh - s s + fl, d = e rsqrt(fh) / 2;
// and seed + d, added in integers on the double's fraction bits, is good to
// about 2^-42.  The FP64 step squares that:
//   y + y (1 - a y)   and   s + (x - s^2) h,  h = rsqrt(fh)/2 ~ 1/(2s),
// each with one rounding of consequence: within an ulp of the correctly
// rounded result (measured by fv_selftest_math against the IEEE operations).
// The forms they replace refined the bare float seed with three and five FP64
// operations.  Arguments whose result or steps would leave the normal range
// (and zero, negative, non-finite values) take the IEEE operation.  The FP32
// forms are the special-function unit's approximations themselves (one
// instruction each, within about an ulp and two ulps): the FP32 path is bound
// by instruction issue, where the IEEE sequences cost about ten instructions
// per cell each, and its error target (1e-5 after a step) is far above an ulp
// of FP32.
// ---------------------------------------------------------------------------

// x (a float in [1/2, 2], as a double) + n 2^-53 x's binade below 1, 2^-52
// from 1 on: n is added to the double's bit pattern.
__device__ __forceinline__ void add_units(float x, long long n, unsigned& hi, unsigned& lo) {
  const unsigned b = __float_as_uint(x);
  const unsigned long long v =
      (((unsigned long long)((b >> 3) + (896u << 20)) << 32) | (b << 29)) + (unsigned long long)n;
  hi = (unsigned)(v >> 32);
  lo = (unsigned)v;
}

__device__ __forceinline__ double recip(double a, const Arith<double>& ar = plain_arith<double>()) {
  const unsigned hi = (unsigned)__double2hiint(a), lo = (unsigned)__double2loint(a);
  if ((hi >> 20) - 2u > 2042u) return 1.0 / a;  // sign clear, exponent 2 .. 2044
  const float fh = __uint_as_float(0x3F800000u | ((hi & 0xFFFFFu) << 3) | (lo >> 29));
  const float fl = __uint_as_float(0x34000000u | ((lo >> 6) & 0x7FFFFFu)) - 0x1p-23f;
  float y0;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y0) : "f"(fh));
  y0 = fminf(fmaxf(y0, 0.5f), 1.0f);
  const float e = fmaf(-fl, y0, fmaf(-fh, y0, 1.0f));
  const float d = y0 * fmaf(e, e, e);
  unsigned yh, yl;
  add_units(y0, (long long)__float2int_rn(d * 0x1p52f) * 2, yh, yl);
  yh += (1023u << 20) - (hi & 0x7FF00000u);
  const double y = __hiloint2double((int)yh, (int)yl);
  return fma(y, fma(neg_t(a), y, 1.0), y);
}
__device__ __forceinline__ float recip(float a, const Arith<float>& = plain_arith<float>()) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a));
  return r;
}

__device__ __forceinline__ double sqrt_t(double x, const Arith<double>& ar = plain_arith<double>()) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  if ((hi >> 20) - 64u > 1982u) return sqrt(x);  // exponent 64 .. 2046
  // x = f 4^k with f in [1, 4)
  const unsigned odd = ((hi >> 20) & 1u) ^ 1u;
  const int k = ((int)(hi >> 20) - 1023 - (int)odd) >> 1;
  const unsigned ob = odd << 23;
  const float fh = __uint_as_float((0x3F800000u + ob) | ((hi & 0xFFFFFu) << 3) | (lo >> 29));
  const float fl = __uint_as_float((0x34000000u + ob) | ((lo >> 6) & 0x7FFFFFu)) -
                   __uint_as_float(0x34000000u + ob);
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(fh));
  const float s = fminf(fmaxf(fh * r, 1.0f), 2.0f);
  const float d = (fmaf(-s, s, fh) + fl) * (0.5f * r);
  unsigned sh, sl;
  add_units(s, (long long)__float2int_rn(d * 0x1p51f) * 2, sh, sl);
  const double s0 = __hiloint2double((int)(sh + ((unsigned)k << 20)), (int)sl);
  const unsigned rb = __float_as_uint(r);
  const double h = __hiloint2double((int)((rb >> 3) + ((unsigned)(895 - k) << 20)), (int)(rb << 29));
  return fma(fma(neg_t(s0), s0, x), h, s0);
}
__device__ __forceinline__ float sqrt_t(float x, const Arith<float>& = plain_arith<float>()) {
  float r;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// ---------------------------------------------------------------------------
// Euler physics of one cell, Eq. 2: q = (rho, j_1..j_D, E),
// u = j / rho, p = (gamma - 1)(E - j.u / 2), c = sqrt(gamma p / rho).
// ---------------------------------------------------------------------------
template <typename T, int D>
struct Prim {
  T u[D];
  T p;
  T c;
  T ep;  // E + p, shared by the energy flux of every direction
};

template <typename T, int D>
__device__ __forceinline__ Prim<T, D> primitives(const T* q, T gm1, T gamma, bool& bad,
                                                 const Arith<T>& ar = plain_arith<T>()) {
  Prim<T, D> w;
  T inv = recip(q[0], ar);
  T jj = T(0);
#pragma unroll
  for (int k = 0; k < D; ++k) {
    w.u[k] = ar.mul(q[1 + k], inv);
    jj = k == 0 ? ar.mul(q[1], w.u[0]) : fma(q[1 + k], w.u[k], jj);
  }
  w.p = ar.mul(gm1, fma(T(-0.5), jj, q[D + 1]));
  w.ep = ar.add(q[D + 1], w.p);
  T c2 = ar.mul(ar.mul(gamma, w.p), inv);
  w.c = sqrt_t(c2, ar);
  bad |= !(positive_finite(q[0]) && positive_finite(w.p));
  return w;
}

// ---------------------------------------------------------------------------
// FP32 bounds of an FP64 cell's wave speed, for maxima: only cells whose
// upper bound reaches the largest lower bound can hold the maximum, and only
// those need the FP64 primitives (19 operations on the scarce pipe; the
// bounds cost none).  um is |u_k| (kdir = k) or the largest |u_k| (kdir < 0),
// and lo <= um + c <= hi for the FP64 um + c; false (lo = 0, hi = inf) where
// that cannot be told: values outside the floats' range, NaN, a pressure that
// is not certain to be positive, or a squared sound speed next to the ends of
// the floats' range -- the caller evaluates those cells.
//
// With x ~ y (1 +- 2^-23) for every truncated input and 2^-23 for the
// approximate reciprocal, u is within 2^-21 of j / rho, the kinetic energy ke
// within 2^-20, and (gamma - 1)(E - ke) within 2^-20 (E + ke) (gamma - 1) of
// p; kWaveEps = 2^-18 covers these, the square root and the final sums four
// times over.
// ---------------------------------------------------------------------------
constexpr float kWaveEps = 0x1p-18f;

// |x| as a float, truncated; `ok` turns false outside the float range (zero
// stays zero).
__device__ __forceinline__ float mag_f32(double x, bool& ok) {
  const unsigned h = (unsigned)__double2hiint(x) & 0x7FFFFFFFu;
  const unsigned l = (unsigned)__double2loint(x);
  // exponents 2^-125 .. 2^126
  const bool in = h - ((1023u - 125u) << 20) < (252u << 20);
  const bool zero = (h | l) == 0u;
  ok = ok && (in || zero);
  const unsigned f = ((h << 3) | (l >> 29)) - (896u << 23);
  return in ? __uint_as_float(f) : 0.f;
}
template <int D>
__device__ __forceinline__ bool wave_bounds(const double* q, float gm1, float gamma, int kdir,
                                            float& lo, float& hi) {
  bool ok = __double2hiint(q[0]) > 0;  // rho > 0
  const float rho = mag_f32(q[0], ok), E = mag_f32(q[D + 1], ok);
  ok = ok && __double2hiint(q[D + 1]) > 0;
  // far from the ends of the range, so that products neither overflow nor
  // underflow where it matters
  ok = ok && rho > 0x1p-60f && rho < 0x1p60f && E > 0x1p-60f && E < 0x1p60f;
  float inv;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(inv) : "f"(rho));
  float ke = 0.f, um = 0.f;
#pragma unroll
  for (int k = 0; k < D; ++k) {
    const float j = mag_f32(q[1 + k], ok), u = j * inv;
    ke = fmaf(0.5f * j, u, ke);
    um = (kdir < 0 || kdir == k) ? fmaxf(um, u) : um;
  }
  const float th = E - ke, tot = E + ke, g = gamma * gm1 * inv;
  ok = ok && th > tot * kWaveEps;  // p > 0 for certain (false for NaN)
  const float c2 = g * th, e2 = g * tot * kWaveEps;
  // c2 and its margin normal numbers (the square root takes subnormal ones for
  // zero) and finite; um may underflow: it is then far below c
  ok = ok && c2 > 0x1p-100f && c2 < 0x1p100f;
  float ch, cl;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(ch) : "f"(c2 + e2));
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(cl) : "f"(fmaxf(c2 - e2, 0.f)));
  hi = ok ? (um + ch) * (1.f + kWaveEps) : __int_as_float(0x7F800000);
  lo = ok ? (um + cl) * (1.f - kWaveEps) : 0.f;
  return ok;
}
// A float not above the wave speed x (a bit pattern of order_bits); 0 where
// x has no float below it in range.
__device__ __forceinline__ float wave_floor(unsigned long long x) {
  bool ok = true;
  const float f = mag_f32(__longlong_as_double((long long)x), ok);
  return ok ? f : 0.f;
}

// Flux f^k (S = D + 2 values) and wave speed |u_k| + c of one cell (Eq. 2, 5).
template <typename T, int D>
__device__ __forceinline__ void flux_dir(const T* q, const Prim<T, D>& w, int k, T* f, T& lam) {
  T uk = w.u[k];
  f[0] = q[1 + k];
#pragma unroll
  for (int m = 0; m < D; ++m) f[1 + m] = (m == k) ? fma(q[1 + m], uk, w.p) : mul_rn(q[1 + m], uk);
  f[D + 1] = mul_rn(w.ep, uk);
  lam = add_rn(abs_t(uk), w.c);
}

// ---------------------------------------------------------------------------
// Patch geometry with a one-cell halo.  P > 0: compile-time patch size;
// P == 0: runtime size (generic path).
// ---------------------------------------------------------------------------
template <int D, int P>
struct Geom {
  int p;
  __device__ __forceinline__ explicit Geom(int p_rt) : p(P > 0 ? P : p_rt) {}
  __device__ __forceinline__ int ne() const { return p + 2; }
  __device__ __forceinline__ int ncell() const {  // halo-inclusive cells
    return D == 1 ? p + 2 : D == 2 ? (p + 2) * (p + 2) : (p + 2) * (p + 2) * (p + 2);
  }
  __device__ __forceinline__ int ptrans() const {  // p^(D-1)
    return D == 1 ? 1 : D == 2 ? p : p * p;
  }
  __device__ __forceinline__ int nint() const { return ptrans() * p; }     // p^D
  __device__ __forceinline__ int nbox() const { return (p + 2) * ptrans(); }  // cells per dir box
  __device__ __forceinline__ int nface() const { return (p + 1) * ptrans(); }  // faces per dir
  // linear cell index of halo-inclusive coordinates
  __device__ __forceinline__ int cell(const int* c) const {
    int idx = c[D - 1];
#pragma unroll
    for (int m = D - 2; m >= 0; --m) idx = idx * (p + 2) + c[m];
    return idx;
  }
  // transverse index of coordinates c (each interior, 1..p) for direction k:
  // the coordinates other than k, lowest axis fastest, shifted to 0..p-1.
  __device__ __forceinline__ int trans(const int* c, int k) const {
    int t = 0;
#pragma unroll
    for (int m = D - 1; m >= 0; --m)
      if (m != k) t = t * p + (c[m] - 1);
    return t;
  }
  // inverse of trans: fill the coordinates other than k from t
  __device__ __forceinline__ void untrans(int t, int k, int* c) const {
#pragma unroll
    for (int m = 0; m < D; ++m)
      if (m != k) {
        c[m] = 1 + t % p;
        t /= p;
      }
  }
  // Cell index of the cell with coordinate ck along a runtime direction k and
  // transverse index t, built with selects (no dynamically indexed arrays,
  // which would live in local memory).
  __device__ __forceinline__ int cell_kt(int k, int ck, int t) const {
    const int ne = p + 2;
    if constexpr (D == 1) {
      return ck;
    } else if constexpr (D == 2) {
      const int a = 1 + t;
      const int c0 = k == 0 ? ck : a;
      const int c1 = k == 0 ? a : ck;
      return c0 + ne * c1;
    } else {
      const int a = 1 + t % p, b = 1 + t / p;
      const int c0 = k == 0 ? ck : a;
      const int c1 = k == 0 ? a : (k == 1 ? ck : b);
      const int c2 = k == 2 ? ck : b;
      return c0 + ne * (c1 + ne * c2);
    }
  }
  // Interior cell index (0-based coordinates, x fastest, stride p) of the
  // cell with interior coordinate c along direction k and transverse index t.
  __device__ __forceinline__ int icell_kt(int k, int c, int t) const {
    if constexpr (D == 1) {
      return c;
    } else if constexpr (D == 2) {
      return k == 0 ? c + p * t : t + p * c;
    } else {
      const int a = t % p, b = t / p;
      const int c0 = k == 0 ? c : a;
      const int c1 = k == 0 ? a : (k == 1 ? c : b);
      const int c2 = k == 2 ? c : b;
      return c0 + p * (c1 + p * c2);
    }
  }
  // Stride of the cell index along direction k.
  __device__ __forceinline__ int stride(int k) const {
    return k == 0 ? 1 : k == 1 ? (p + 2) : (p + 2) * (p + 2);
  }
};

}  // namespace fv
