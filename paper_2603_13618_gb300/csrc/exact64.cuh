// exact64.cuh -- FP64 results without the FP64 pipe.  An SM of this GPU issues about two
// FP64 operations per clock (conversions to and from FP64 included) against 64 integer and
// 128 FP32 ones, so the boundary kernels, which hand FP32 and FP16 states out as FP64
// arrays, are bound by that pipe and not by memory when they convert, add and divide in FP64.
// Conversions and sums here give the value that the FP64 instructions give.  Quotients and
// reciprocals are rounded once, from a value within 2^-86 of the exact one: they are the IEEE
// result except where the exact value lies within 2^-33 of a unit in the last place from the
// middle of two FP64 numbers (about one in 2^32 of them), where they may be the other of the two.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace kss {

// double(x): a normal number's sign, exponent (rebiased by 1023 - 127 = 896) and fraction
// move to their FP64 places; zero, subnormals, infinities and NaN take the conversion.
__device__ __forceinline__ double widen(float x) {
  const uint32_t b = __float_as_uint(x);
  if (((b + 0x00800000u) & 0x7f000000u) == 0u) return double(x);  // exponent field 0 or 255
  return __hiloint2double(int((b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + (896u << 20))),
                          int(b << 29));
}
__device__ __forceinline__ double widen(double x) { return x; }

// The quotient j / r (rounded as above) of two integers, |j| and 0 < r below 2^53 (jd, rd: the
// magnitudes scaled into [1, 2), yd about 1 / rd): q0 = jd yd, then one correction by the
// remainder (Markstein, "Computation of elementary functions on the IBM RISC System/6000
// processor", 1990).  yd is within 2^-43 of 1 / rd, so the corrected quotient is within
// 2^-86 of the exact one before its only rounding.
__device__ __forceinline__ double quotient(double jd, double rd, double yd) {
  const double q0 = jd * yd;
  return fma(fma(-q0, rd, jd), yd, q0);
}

// About 1 / rd for rd in [1, 2) given by its fraction field, within 2^-43: the FP32
// reciprocal of its first 24 bits, one Newton step in FP32 on what that leaves, and the two
// parts added in fixed point (units of 2^-53).
__device__ __forceinline__ double reciprocal46(uint64_t frac) {
  const float rh = __uint_as_float(0x3f800000u | uint32_t(frac >> 29));
  const float rl =
      (__uint_as_float(0x3f800000u | (uint32_t(frac >> 6) & 0x7fffffu)) - 1.f) * 0x1p-23f;
  float y0;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y0) : "f"(rh));
  const float e = fmaf(-rl, y0, fmaf(-rh, y0, 1.f));
  long long y = (long long)(uint32_t(__float2int_rn(y0 * 0x1p24f))) << 29;
  y += __float2int_rn(y0 * e * 0x1p53f);
  // 1 / rd is in (1/2, 1]: keep the approximation there
  y = max(min(y, (1ll << 53) - 1), 1ll << 52);
  return __longlong_as_double((y & ((1ll << 52) - 1)) | (1022ll << 52));
}

// 1 / x (rounded as above): reciprocal46 and one FP64 Newton step, which leaves 2^-86 before its
// rounding (two operations of the FP64 pipe; the compiler's division takes about ten).
// Exponents near the ends of the range, zero, infinities and NaN take the division.
__device__ __forceinline__ double rcp64(double x) {
  const uint32_t hi = uint32_t(__double2hiint(x)), e = (hi >> 20) & 0x7ffu;
  if (e - 3u > 2040u) return 1.0 / x;
  const uint64_t b = uint64_t(__double_as_longlong(x));
  const double m = __longlong_as_double((long long)((b & ((1ull << 52) - 1)) | (1023ull << 52)));
  const double y0 = reciprocal46(b & ((1ull << 52) - 1));
  const double y = fma(fma(-m, y0, 1.0), y0, y0);
  // times 2^(1023 - e), exact; the sign of x
  return __hiloint2double(int((uint32_t(__double2hiint(y)) + ((1023u - e) << 20)) |
                              (hi & 0x80000000u)),
                          __double2loint(y));
}

// n / d (rounded as above), for d positive and of ordinary size (2^-1000 < d < 2^1000; other d give
// some number or NaN): three operations of the FP64 pipe.
__device__ __forceinline__ double ratio64(double n, double d) {
  const uint64_t b = uint64_t(__double_as_longlong(d));
  const double y = reciprocal46(b & ((1ull << 52) - 1));
  const uint32_t e = uint32_t(b >> 52) & 0x7ffu;
  return quotient(n, d, __hiloint2double(int(uint32_t(__double2hiint(y)) + ((1023u - e) << 20)),
                                         __double2loint(y)));
}

// rho = sum v, ux = jx / rho and uy = jy / rho of nine FP32 populations: the sums of FP64
// arithmetic, and their quotients rounded as above.  Where the populations are positive and
// their exponents span at most 25, the moments are integers below 2^53 in units of the smallest
// population's last place: every FP64 partial sum is exact, and so are these integer sums.
// Other cells return false.
__device__ __forceinline__ bool moments_exact(const float (&v)[9], double& rho, double& ux,
                                              double& uy) {
  uint32_t lo = 0xffffffffu, hi = 0u, b[9];
#pragma unroll
  for (int q = 0; q < 9; ++q) {
    b[q] = __float_as_uint(v[q]);
    lo = min(lo, b[q]);
    hi = max(hi, b[q]);
  }
  const int e0 = int(lo >> 23);
  if (e0 < 1 || hi >= 0x7f800000u || int(hi >> 23) - e0 > 25) return false;
  long long m[9];
#pragma unroll
  for (int q = 0; q < 9; ++q)
    m[q] = (long long)(uint64_t((b[q] & 0x7fffffu) | 0x800000u) *
                       uint64_t(1u << (int(b[q] >> 23) - e0)));
  const long long r = ((m[0] + m[1]) + (m[2] + m[3])) + ((m[4] + m[5]) + (m[6] + m[7])) + m[8];
  const long long j[2] = {(m[1] - m[3]) + (m[5] + m[8]) - (m[6] + m[7]),
                          (m[2] - m[4]) + (m[5] + m[6]) - (m[7] + m[8])};
  constexpr uint64_t kFrac = (1ull << 52) - 1, kOne = 1023ull << 52;
  const int zr = __clzll(r);  // r < 2^53: at least 11
  const uint64_t fr = (uint64_t(r) << (zr - 11)) & kFrac;
  rho = __longlong_as_double((long long)(fr | (uint64_t(63 - zr + e0 - 150 + 1023) << 52)));
  const double rd = __longlong_as_double((long long)(fr | kOne));
  const double yd = reciprocal46(fr);
  double u[2];
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const uint64_t a = uint64_t(j[k] < 0 ? -j[k] : j[k]);
    const int z = __clzll((long long)a);
    const double jd =
        __longlong_as_double((long long)(((a << ((z - 11) & 63)) & kFrac) | kOne));
    const long long q = __double_as_longlong(quotient(jd, rd, yd));
    // times 2^(zr - z), exact: the quotient is at least 2^-53
    const long long s = q + ((long long)(zr - z) << 52);
    u[k] = a == 0 ? 0.0 : __longlong_as_double(s | (j[k] & (1ll << 63)));
  }
  ux = u[0];
  uy = u[1];
  return true;
}

}  // namespace kss
