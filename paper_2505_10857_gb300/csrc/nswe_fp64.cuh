// FP64 reciprocal, square root and division by a fixed divisor with fewer
// instructions on the FP64 pipe.
//
// On GB300 one FP64 warp instruction holds an SM sub-partition's FP64 unit
// for 64 cycles, whatever its active lanes and however independent the
// instructions of a warp are (measured: 64.3 cycles per DFMA for one warp,
// in one chain or four), so the FP64-bound kernels of this library cost what
// they issue. Measured in units of one DFMA: 1.0/x 5.3, sqrt(x) 8.8, x/a 8.5;
// the forms below 3.15, 6.5 and 3. Each is a power-series iteration from the
// hardware's approximation (PTX rcp.approx.ftz.f64 / rsqrt.approx.ftz.f64,
// relative error below 2^-19):
//   1/x:     e = 1 - x y, 1/x = y / (1 - e) = y (1 + e + e^2 + ...), cut after
//            e^2 (the third-order Householder iteration): relative error
//            before the last rounding below 2^-57;
//   sqrt(x): two steps of Heron's iteration s + (x - s^2) / (2 s) with 1/(2 s)
//            from the seed, the residual x - s^2 formed exactly by an FMA;
//   a / b:   q = a (1/b) and one correction by the exact residual a - b q.
// Against the correctly rounded operations, 2e6 random arguments each: the
// reciprocal differs (by one in the last place) in 0.03 % of cases, the square
// root in 0.04 %, the division in none for exponents near zero and in 0.01 %
// over all exponents (subnormal residuals); the reciprocal square root is
// within 0.99 ulp of the exact value (tests/test_gpu_fp64.py).
//
// Arguments outside the normal range, whose result would not be a normal
// number, take the ordinary operation (an integer test of the exponent), so
// zeros, infinities, NaN, negative and subnormal arguments give what 1.0 / x,
// sqrt(x) and a / b give.
#pragma once

namespace nswe {

__device__ __forceinline__ unsigned fp64_exponent(double x) { return (unsigned)(__double2hiint(x) >> 20) & 0x7ffu; }

__device__ __forceinline__ double fast_rcp(double x) {
  if (fp64_exponent(x) - 2u > 2040u) return 1.0 / x;  // biased exponent outside [2, 2042]
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = fma(-x, y, 1.0);
  return fma(fma(e, e, e), y, y);
}

__device__ __forceinline__ double fast_sqrt(double x) {
  // positive, biased exponent in [128, 1920]: the residual x - s^2 neither overflows nor loses bits
  if ((unsigned)(__double2hiint(x) >> 20) - 128u > 1792u) return sqrt(x);
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double h = 0.5 * y;
  double s = x * y;
  s = fma(fma(-s, s, x), h, s);
  return fma(fma(-s, s, x), h, s);
}

__device__ __forceinline__ bool fp64_zero(double x) { return ((__double2hiint(x) << 1) | __double2loint(x)) == 0; }

// a / b with rb = 1.0 / b given.
__device__ __forceinline__ double fast_div(double a, double b, double rb) {
  const double q = a * rb;
  const unsigned eq = fp64_exponent(q);
  if (eq - 64u > 1919u)  // a quotient that is tiny, huge or not finite; zero over a finite rb is already right
    return fp64_zero(a) && fp64_zero(q) ? q : a / b;
  return fma(fma(-b, q, a), rb, q);
}

// x^(-1/2): e = 1 - x y^2, y (1 - e)^(-1/2) = y (1 + e/2 + 3 e^2/8 + ...), cut
// after e^2: relative error before the last rounding below 2^-54.
__device__ __forceinline__ double fast_rsqrt(double x) {
  if ((unsigned)(__double2hiint(x) >> 20) - 2u > 2040u) return rsqrt(x);  // negative, zero, subnormal, huge, NaN
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = fma(-x * y, y, 1.0);
  return fma(y * e, fma(0.375, e, 0.5), y);
}

// fast_* for FP64 arguments, the plain operation in FP32.
__device__ __forceinline__ double rcp_t(double x) { return fast_rcp(x); }
__device__ __forceinline__ float rcp_t(float x) { return 1.0f / x; }
__device__ __forceinline__ double rsqrt_t(double x) { return fast_rsqrt(x); }
__device__ __forceinline__ float rsqrt_t(float x) { return rsqrtf(x); }

}  // namespace nswe
