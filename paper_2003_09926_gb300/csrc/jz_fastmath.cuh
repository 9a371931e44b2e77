// jz_fastmath.cuh -- elementary-function choices of the FP32 and FP64
// arithmetic, shared by the fused stage kernels and the boundary pass.
#pragma once

#include <cmath>
#include <cstdint>

namespace jz {
namespace stg {

// Elementary functions.  FP32 arithmetic uses the hardware approximations
// (sqrt.approx, rcp.approx, ex2/lg2.approx: a few ulp, far below the FP32
// error of the scheme itself); the FP64 kernels' functions follow it.
template <typename R> struct Fn;
template <> struct Fn<float> {
  static __device__ __forceinline__ float sqrt_(float x) {
    float y;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
  }
  static __device__ __forceinline__ float rcp(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
  }
  static __device__ __forceinline__ float div(float a, float b) { return a * rcp(b); }
  // a product that is never fused into a later addition
  static __device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
  // x^e = 2^(e log2 x) for x > 0 (no library call inside the flux code)
  static __device__ __forceinline__ float powp(float x, float e) {
    float l, y;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(l) : "f"(x));
    l *= e;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(l));
    return y;
  }
  // J^(-2/3) = 2^(-2/3 log2 J), J > 0
  static __device__ __forceinline__ float jm23(float J) {
    float l, y;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(l) : "f"(J));
    l *= -2.0f / 3.0f;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(l));
    return y;
  }
};

// FP64 reciprocal, square root and J^(-2/3) of the FP64 stage kernel and
// time-step reduction, whose FP64 pipe passes two lanes per cycle and SM: from
// the hardware's approximations (relative error e of 2^-19.9 for rcp and
// 2^-19.0 for rsqrt, the largest seen over 2^26 mantissas) and their Taylor
// series to e^3, 4, 7 and 7 FP64 instructions.  What the series leave out is below
// 2^-75, so that reciprocal and square root err by the last rounding alone
// (0.5 units in the last place) and J^(-2/3) by it and two thirds of the one in
// y^3, less than the library's cbrt, product and division (1.01 against 3.2
// units).  Step of a 128x96x96 grid: 6.28 ms, 6.63 with the library's division,
// square root and cbrt, 5.98 with the series to e^2, which err by 0.504, 0.75
// and 2.3 units.

// Zero, infinity and NaN give what IEEE arithmetic gives, told apart by integer
// instructions (0.2% of a step); subnormal numbers count as zero.

// 1/b: with e = 1 - b y, 1/b = y (1 + e + e^2 + e^3 + ...)
__device__ __forceinline__ double rcp_d(double b) {
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(b));
  const double e = fma(-b, y, 1.0);
  const double r = fma(y, fma(fma(e, e, e), e, e), y);
  return (uint32_t)((__double2hiint(y) & 0x7fffffff) - 0x00100000) < 0x7fe00000u ? r : y;  // y = 0, inf or NaN
}

// sqrt(x): y of an approximation to x^(-1/2), t + l = x y exactly; with
// e = 1 - t y, sqrt(x) = t + (t e + l) (1/2 + 3 e/8 + 5 e^2/16 + ...)
__device__ __forceinline__ double sqrt_d(double x) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double t = __dmul_rn(x, y);
  const double l = fma(x, y, -t);
  const double e = fma(-t, y, 1.0);
  const double r = fma(fma(t, e, l), fma(fma(0.3125, e, 0.375), e, 0.5), t);
  const int hi = __double2hiint(x);  // NaN of a negative x comes with y
  if ((hi & 0x7fffffff) < 0x00100000) return 0.0;
  return hi == 0x7ff00000 ? x : r;
}

// J^(-2/3) (of |J|): J = m 2^(3q), 1 <= m < 16; y of an FP32 approximation to
// m^(-1/3) (y^2 is exact in FP64), then with e = 1 - m y^3,
// m^(-2/3) = y^2 (1 + 2 e/3 + 5 e^2/9 + 40 e^3/81 + ...).  The exponents are
// integer arithmetic.
__device__ __forceinline__ double jm23_d(double J) {
  const int hi = __double2hiint(J) & 0x7fffffff, lo = __double2loint(J);
  const int ex = (hi >> 20) - 1023;
  const int q = (ex * 21846) >> 16;  // floor(ex / 3), or one less
  const double m = __hiloint2double(hi - (q * 3 << 20), lo);
  float y, l;
  asm("lg2.approx.ftz.f32 %0, %1;"
      : "=f"(l)
      : "f"(__uint_as_float((((uint32_t)hi & 0xfffffu) << 3 | (uint32_t)lo >> 29) | (uint32_t)(ex - 3 * q + 127) << 23)));
  l *= -1.0f / 3.0f;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(l));
  const uint32_t b = __float_as_uint(y);  // a normal number: widened by its bits
  const double y1 = __hiloint2double((int)((b >> 3) + 0x38000000u), (int)(b << 29));
  const double y2 = __dmul_rn(y1, y1);
  const double e = fma(-m, __dmul_rn(y2, y1), 1.0);
  const double c = fma(fma(40.0 / 81.0, e, 5.0 / 9.0), e, 2.0 / 3.0);
  const double r = fma(__dmul_rn(y2, e), c, y2);
  int rhi = __double2hiint(r) - (q * 2 << 20), rlo = __double2loint(r);
  if ((uint32_t)(hi - 0x00100000) >= 0x7fe00000u) {
    rhi = hi < 0x00100000 ? 0x7ff00000 : ((hi ^ 0x7ff00000) | lo ? 0x7ff80000 : 0);
    rlo = 0;
  }
  return __hiloint2double(rhi, rlo);
}

// Five increments in FP64, exactly.  A conversion instruction runs on the FP64
// pipe, which passes two lanes per cycle on a GB300 SM and which the five
// additions and roundings of an update need too; for normal numbers the
// exponent is re-biased with integer instructions instead (one check for all
// five: separate ones cost what they saved).  160x128x128: 0.826 and 0.750 ms
// per step.
__device__ __forceinline__ void widen5(const float x[5], double y[5]) {
  bool normal = true;
#pragma unroll
  for (int v = 0; v < 5; ++v) normal = normal && (__float_as_uint(x[v]) & 0x7fffffffu) - 0x00800000u < 0x7f000000u;
  if (normal) {
#pragma unroll
    for (int v = 0; v < 5; ++v) {
      const uint32_t b = __float_as_uint(x[v]);
      y[v] = __hiloint2double((int)((((b & 0x7fffffffu) >> 3) + 0x38000000u) | (b & 0x80000000u)), (int)(b << 29));
    }
  } else {
#pragma unroll
    for (int v = 0; v < 5; ++v) y[v] = (double)x[v];
  }
}

}  // namespace stg
}  // namespace jz
