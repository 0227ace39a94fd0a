#pragma once
// tkf_fp64.cuh -- FP64 arithmetic that spares the FP64 pipe, shared by the kernels.

#include <cuda_runtime.h>
#include <stdint.h>

namespace tkf {
namespace {

constexpr double kPi = 3.14159265358979323846;

// Exact FP32 <-> FP64 conversions on the integer pipes. On GB300 the hardware conversion runs
// on the FP64 pipe (a warp instruction occupies it for 16 SM cycles), and the FP64 pipe bounds
// the mixed path; these give the IEEE results (round to nearest even) for every normal number
// and zero with a few integer operations. FP32 denormals become signed zero; out of range
// FP64 values (beyond the FP32 normals, infinities, NaN) become NaN, and FP32 infinities and
// NaN become FP64 NaN, so a non-finite value stays non-finite.
__device__ __forceinline__ double f2d(float x) {
  const uint32_t u = __float_as_uint(x), a = u & 0x7FFFFFFFu;
  const bool tiny = a < 0x00800000u, special = a >= 0x7F800000u;
  const uint32_t hi = tiny ? 0u : (special ? 0x7FF80000u : (a >> 3) + (896u << 20));  // bias 127 -> 1023
  return __hiloint2double(int((u & 0x80000000u) | hi), int(tiny ? 0u : (u << 29)));
}

__device__ __forceinline__ float d2f(double x) {
  const uint32_t hi = uint32_t(__double2hiint(x)), lo = uint32_t(__double2loint(x)), a = hi & 0x7FFFFFFFu;
  uint32_t m = ((a - 0x38000000u) << 3) | (lo >> 29);  // bias 1023 -> 127, top 23 mantissa bits
  // round to nearest even on the 29 dropped bits: up if above half, or at half with m odd
  m += (lo >> 28) & ((lo & 0x0FFFFFFFu ? 1u : 0u) | m) & 1u;
  m = a < 0x38100000u ? 0u : (a >= 0x47F00000u ? 0x7FC00000u : m);
  return __uint_as_float((hi & 0x80000000u) | m);
}

// ------------------------------------------------------------------ FP64 without the FP64 pipe's divides
// A division or square root in FP64 is a sequence of 8 to 12 FP64 instructions, and an FP64 warp
// instruction holds its SM partition for 64 cycles on GB300 (integer, FP32 and special-function
// instructions: 1 to 4). The FP64 path's stepping therefore takes reciprocals and roots by
// Newton-Raphson (or one third-order step, which cubes the relative error) from the special-function
// unit's or an FP32 seed, and compares magnitudes as integers. Products that feed a sum are written
// as fma() or __dmul_rn, or as mul_add and mul_sub below, so that they round alike in every instantiation (register
// caps, lanes a track). Sums of the FP64 path's general code that are left to the compiler have rounded alike in all of
// them so far (tilted and axial fields, the map), which nothing guarantees.

// |x| <= lim and |x| < lim for lim >= 0: the bit patterns of non-negative doubles order like the
// values, NaN above all (so a NaN x is neither).
__device__ __forceinline__ bool abs_le(double x, double lim) {
  return (__double_as_longlong(x) & 0x7fffffffffffffffll) <= __double_as_longlong(lim);
}
__device__ __forceinline__ bool abs_lt(double x, double lim) {
  return (__double_as_longlong(x) & 0x7fffffffffffffffll) < __double_as_longlong(lim);
}

// x > 0, as an integer test in FP64 (false for NaN)
__device__ __forceinline__ bool positive(double x) {
  return (unsigned long long)(__double_as_longlong(x) - 1) < 0x7ff0000000000000ull;
}
__device__ __forceinline__ bool positive(float x) { return x > 0.0f; }

// 1/x of a normal x well inside the exponent range, within an ulp: the special-function seed (2^-20)
// and one third-order step.
__device__ __forceinline__ double rcp_nr(double x) {
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = fma(-x, y, 1.0);
  return fma(y, fma(e, e, e), y);
}

// 1/sqrt(x) of a normal x > 0, within 1.1 ulp, in the same way.
__device__ __forceinline__ double rsqrt_nr(double x) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = fma(__dmul_rn(-x, y), y, 1.0);
  return fma(__dmul_rn(y, e), fma(e, 0.375, 0.5), y);
}

// a b + c d and a b - c d with the first product fused and the second rounded. Which of two products a compiler fuses
// depends on what surrounds the sum: left to it, kernels of the same source round differently.
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
template <class R>
__device__ __forceinline__ R mul_add(R a, R b, R c, R d) {
  return fma(a, b, mul_rn(c, d));
}
template <class R>
__device__ __forceinline__ R mul_sub(R a, R b, R c, R d) {
  return fma(a, b, -mul_rn(c, d));
}

// a . b with a fixed order of roundings
__device__ __forceinline__ double dot3f(const double a[3], const double b[3]) {
  return fma(a[2], b[2], fma(a[1], b[1], __dmul_rn(a[0], b[0])));
}
__device__ __forceinline__ void crossf(const double a[3], const double b[3], double o[3]) {
  o[0] = fma(a[1], b[2], -__dmul_rn(a[2], b[1]));
  o[1] = fma(a[2], b[0], -__dmul_rn(a[0], b[2]));
  o[2] = fma(a[0], b[1], -__dmul_rn(a[1], b[0]));
}

// Natural logarithm of a positive normal x (table-driven, after P. T. P. Tang, ACM TOMS 16, 1990):
// x = 2^e m, c ~ 1/m from the top 7 bits of m, ln x = e ln 2 - ln c + ln(1 + z) with z = m c - 1,
// |z| < 2^-8, by its series through z^7 (truncation below 2^-66). 11 FP64 instructions against about
// 25 of log(). The sum with e ln 2 comes last, so that one rounding is of the result's size: within 1.1 ulp where its
// magnitude is 4 to 40 (e times the rounding of ln 2, the table's and the small sum's 2^-53 in the rest), within 2^-50
// below; with e ln 2 - ln c first and the series last, 1.31 ulp. The callers' results are of magnitude 0 to 40 (the
// scattering's below 4 at steep incidence). Zero, negative, not normal: log().
struct LogTable {
  double c[128], l[128];  // c, -ln c
};
constexpr LogTable make_log_table() {
  LogTable t{};
  for (int j = 0; j < 128; ++j) {
    const double c = 256.0 / (257.0 + 2.0 * j);
    // -ln c = 2 artanh((1 - c) / (1 + c))
    const double u = (1.0 - c) / (1.0 + c), u2 = u * u;
    double sum = 0.0;
    for (int k = 41; k >= 1; k -= 2) sum = sum * u2 + 1.0 / k;
    t.c[j] = c;
    t.l[j] = 2.0 * u * sum;
  }
  return t;
}
__device__ const LogTable kLogTable = make_log_table();

__device__ __forceinline__ double log_nr(double x) {
  const uint32_t hi = uint32_t(__double2hiint(x));
  if (hi - 0x00100000u >= 0x7fe00000u) return log(x);
  const int e = int(hi >> 20) - 1023;
  const uint32_t j = (hi >> 13) & 127u;
  const double m = __hiloint2double(int((hi & 0x000fffffu) | 0x3ff00000u), __double2loint(x));
  const double z = fma(m, __ldg(&kLogTable.c[j]), -1.0);
  double p = fma(z, 1.0 / 7, -1.0 / 6);
  p = fma(z, p, 0.2);
  p = fma(z, p, -0.25);
  p = fma(z, p, 1.0 / 3);
  p = fma(z, p, -0.5);
  p = fma(__dmul_rn(z, z), p, z);
  return fma(f2d(float(e)), 0.693147180559945309417, __ldg(&kLogTable.l[j]) + p);
}

// atan2(y, x) (table-driven, after P. T. P. Tang, ACM TOMS 16, 1990): with t = min / max of |x|, |y| and
// k ~ 16 t, atan t = atan(k / 16) + atan(d), d = (min - k/16 max) / (max + k/16 min), |d| < 2^-4.9, by its
// series through d^11 (truncation below 2^-61 relative). 20 FP64 instructions against more than 50 of
// atan2(), within 1.9 ulp (CUDA's atan2: 2). Outside the FP32 range, and where an argument is not finite: atan2().
__device__ const double kAtan16[17] = {  // atan(k / 16)
    0.0, 0.06241880999595735, 0.12435499454676144, 0.18534794999569476, 0.24497866312686414, 0.3028848683749714,
    0.35877067027057225, 0.4124104415973873, 0.4636476090008061, 0.5123894603107377, 0.5585993153435624,
    0.6022873461349642, 0.6435011087932844, 0.6823165548747481, 0.7188299996216245, 0.7531512809621944,
    0.7853981633974483};

__device__ __forceinline__ double atan2_nr(double y, double x) {
  const float xf = fabsf(d2f(x)), yf = fabsf(d2f(y));
  const float big = fmaxf(xf, yf);
  if (!(xf < 1e30f && yf < 1e30f && big > 1e-30f)) return atan2(y, x);
  const bool steep = abs_lt(x, fabs(y));
  const double mn = steep ? fabs(x) : fabs(y), mx = steep ? fabs(y) : fabs(x);
  const float kf = rintf(__fdividef(fminf(xf, yf), big) * 16.0f);
  const double c = f2d(kf * 0.0625f), num = fma(-c, mx, mn), den = fma(c, mn, mx);
  double inv;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(inv) : "d"(den));
  inv = fma(inv, fma(-den, inv, 1.0), inv);  // 2^-40; the quotient's remainder gives the rest
  double d = __dmul_rn(num, inv);
  d = fma(fma(-d, den, num), inv, d);
  const double e = __dmul_rn(d, d);
  double p = fma(e, -1.0 / 11, 1.0 / 9);
  p = fma(e, p, -1.0 / 7);
  p = fma(e, p, 0.2);
  p = fma(e, p, -1.0 / 3);
  const double t = __ldg(&kAtan16[int(kf)]) + fma(__dmul_rn(d, e), p, d);
  // t, pi/2 - t, pi/2 + t or pi - t, with the part of pi below its double
  constexpr double kPiLo = 1.2246467991473532e-16;
  const bool back = __double2hiint(x) < 0;
  const double base = steep ? 0.5 * kPi : (back ? kPi : 0.0), lo = steep ? 0.5 * kPiLo : (back ? kPiLo : 0.0);
  const double r = base + ((steep != back ? -t : t) + lo);
  return copysign(r, y);
}

}  // namespace
}  // namespace tkf
