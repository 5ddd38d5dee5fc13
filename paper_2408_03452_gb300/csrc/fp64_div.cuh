// FP64 division in integer arithmetic.
#pragma once
#include <cstdint>
#include <cstring>

#ifdef __CUDACC__
#define TPFA_HD __host__ __device__ __forceinline__
#else
#define TPFA_HD inline
#endif

namespace tpfa {

// The quotient digits of div_rn: round-to-nearest of ma 2^52 / mb for integers
// 2^52 <= mb < 2^53, mb <= ma < 2 mb, from y0, the reciprocal of mb 2^-52 with a
// relative error below 2^-21.5.
//
// Long division with two digits of 26 and 27 bits:
//   Y  = y0 2^31 after one Newton step in integers, |Y mb 2^-83 - 1| < 2^-29.4;
//   q1 = ma 2^25 / mb to within 0.72, so |R1| < 0.72 mb for R1 = ma 2^25 - q1 mb;
//   q2 = R1 2^27 / mb, the exact value between q2 - 0.64 and q2 + 0.89 (the 0.25
//        from R1's 23 dropped bits, 0.14 from Y, the rest from rounding).
// The remainder R = ma 2^52 - (q1 2^27 + q2) mb is exact modulo 2^64 and below mb
// in size, so comparing 2R with +-mb leaves the nearest integer.  A tie would
// make (2Q + 1) mb = 2^53 ma with 2Q + 1 odd and above 2^53 > its odd part's
// bound in ma: there is none.
TPFA_HD uint64_t div_digits(uint64_t ma, uint64_t mb, float y0) {
  uint32_t f;
#ifdef __CUDA_ARCH__
  f = __float_as_uint(fminf(fmaxf(y0, 0.5f), 0.99999994f));
#else
  y0 = y0 < 0.5f ? 0.5f : (y0 < 0.99999994f ? y0 : 0.99999994f);
  memcpy(&f, &y0, 4);
#endif
  const uint32_t Y0 = ((f & 0x7fffffu) | 0x800000u) << 7;  // y0 2^31, y0 in [1/2, 1)
  const uint32_t B = (uint32_t)(mb >> 21);                 // mb 2^-52 in units of 2^-31
  const int64_t err = (int64_t)(((uint64_t)1 << 62) - (uint64_t)Y0 * B);
  const int32_t t = (int32_t)(err >> 20);
  const int32_t corr = (int32_t)(((int64_t)(int32_t)Y0 * t) >> 32) >> 10;
  const uint32_t Yu = Y0 + (uint32_t)corr;
  const uint32_t Y = Yu < 0x7fffffffu ? Yu : 0x7fffffffu;

  const uint32_t q1 = ((uint32_t)(((uint64_t)(uint32_t)(ma >> 22) * Y) >> 32) + 8u) >> 4;
  const int64_t R1 = (int64_t)((ma << 25) - (uint64_t)q1 * mb);
  const int32_t r1 = (int32_t)(R1 >> 23);
  const int32_t q2 = ((int32_t)(((int64_t)r1 * (int32_t)Y) >> 32) + 1) >> 1;
  const int64_t R = (int64_t)(((uint64_t)R1 << 27) - (uint64_t)(int64_t)q2 * mb);
  uint64_t Q = ((uint64_t)q1 << 27) + (uint64_t)(int64_t)q2;
  if (2 * R > (int64_t)mb) Q += 1;
  if (2 * R < -(int64_t)mb) Q -= 1;
  return Q;
}

// A numerator taken apart once: positive normal values have their fraction with
// the leading one and their biased exponent, all others an exponent that sends
// every quotient to the operator.
struct Num {
  double v;
  uint64_t m;
  int e;
};

inline Num make_num(double v) {
  Num n;
  uint64_t u;
  memcpy(&u, &v, 8);
  n.v = v;
  n.m = (u & (((uint64_t)1 << 52) - 1)) | ((uint64_t)1 << 52);
  const uint32_t e = (uint32_t)(u >> 52);  // with the sign above
  n.e = e - 1u < 2046u ? (int)e : -100000;
  return n;
}

#ifdef __CUDACC__
// a / b, rounded to nearest as by the operator, for every a and b.  The FP64 pipe
// runs at 1/64 of the FP32 rate and a division takes about ten of its operations
// (155 cycles of an SM per warp); about sixty integer operations do the same in a
// quarter of that, beside it.  Positive normal operands with a normal quotient
// take this way, everything else the operator.
__device__ __forceinline__ double div_rn(const Num& a, double b) {
  const uint64_t ub = (uint64_t)__double_as_longlong(b);
  const uint32_t eb = (uint32_t)(ub >> 52);  // with the sign above
  const uint64_t one = (uint64_t)1 << 52;
  const uint64_t mb = (ub & (one - 1)) | one;
  const bool lt = a.m < mb;
  const int e1 = a.e - (int)eb + (lt ? 1021 : 1022);  // biased exponent of the quotient, less one
  if (eb - 1u >= 2046u || (uint32_t)e1 >= 2046u) return a.v / b;
  const float x = __uint_as_float(0x3f800000u | ((uint32_t)(mb >> 29) & 0x7fffffu));
  float y0;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y0) : "f"(x));
  const uint64_t Q = div_digits(lt ? a.m << 1 : a.m, mb, y0);
  return __longlong_as_double((long long)(((uint64_t)(uint32_t)e1 << 52) + Q));
}
#endif

}  // namespace tpfa
