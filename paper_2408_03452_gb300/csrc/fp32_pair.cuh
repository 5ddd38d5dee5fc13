// Unevaluated sums of two floats: about 48 bits on the FP32 units.
#pragma once
#include <cmath>
#include <cstdint>
#include <cstring>

#ifdef __CUDACC__
#define TPFA_PAIR __host__ __device__ __forceinline__
#else
#define TPFA_PAIR inline
#endif

namespace tpfa {

// h + l; after df_fast |l| is at most half an ulp of h.  (The host versions of the
// operations, compiled without contraction, are there for tests.)
struct Dfl {
  float h, l;
};

TPFA_PAIR float fl_add(float a, float b) {
#ifdef __CUDA_ARCH__
  return __fadd_rn(a, b);
#else
  return a + b;
#endif
}
TPFA_PAIR float fl_sub(float a, float b) { return fl_add(a, -b); }
TPFA_PAIR float fl_mul(float a, float b) {
#ifdef __CUDA_ARCH__
  return __fmul_rn(a, b);
#else
  return a * b;
#endif
}
TPFA_PAIR float fl_fma(float a, float b, float c) {
#ifdef __CUDA_ARCH__
  return __fmaf_rn(a, b, c);
#else
  return std::fma(a, b, c);
#endif
}
TPFA_PAIR uint32_t fl_bits(float a) {
#ifdef __CUDA_ARCH__
  return __float_as_uint(a);
#else
  uint32_t u;
  memcpy(&u, &a, 4);
  return u;
#endif
}
TPFA_PAIR float fl_of_bits(uint32_t u) {
#ifdef __CUDA_ARCH__
  return __uint_as_float(u);
#else
  float a;
  memcpy(&a, &u, 4);
  return a;
#endif
}

TPFA_PAIR Dfl df_fast(float a, float b) {  // |a| >= |b| (Dekker 1971)
  const float s = fl_add(a, b);
  return {s, fl_sub(b, fl_sub(s, a))};
}
// a + b, the rounding error of the high parts by TwoSum (Knuth, TAOCP 4.2.2), without
// the final normalisation: for trees of a few levels, where the correction stays
// small; only one addition is on the critical path
TPFA_PAIR Dfl df_acc(Dfl a, Dfl b) {
  const float s = fl_add(a.h, b.h);
  const float v = fl_sub(s, a.h);
  const float e = fl_add(fl_sub(a.h, fl_sub(s, v)), fl_sub(b.h, v));
  return {s, fl_add(e, fl_add(a.l, b.l))};
}
TPFA_PAIR Dfl df_add(Dfl a, Dfl b) {
  const Dfl t = df_acc(a, b);
  return df_fast(t.h, t.l);
}
TPFA_PAIR bool df_le(Dfl a, Dfl b) { return a.h < b.h || (a.h == b.h && a.l <= b.l); }
TPFA_PAIR Dfl df_mulf(Dfl a, float b) {
  const float p = fl_mul(a.h, b);
  return df_fast(p, fl_fma(a.l, b, fl_fma(a.h, b, -p)));
}

// a / b rounded to FP32, for a, b in [2^-50, 2^50] (which keeps the correction in the
// range of normal numbers); y0 the reciprocal of b.h with a relative error below
// 2^-21.  q0 is within 2^-20 of the quotient, and the residual a - q0 b, with the low
// parts, has a relative error of 2^-22; so q0 + q1 is the quotient to 2^-41 before
// the one rounding of the sum: what an FP64 quotient rounded to FP32 gives, unless the
// quotient lies that close to the middle of two floats.
TPFA_PAIR float df_quot_mid(Dfl a, Dfl b, float y0) {
  const float q0 = fl_mul(a.h, y0);
  const float r = fl_fma(-q0, b.l, fl_fma(-q0, b.h, a.h));
  return fl_add(q0, fl_mul(fl_add(r, a.l), y0));
}

// a.h = m 2^k with 1 <= m < 2 (0 stays 0); in two factors, either of which alone could
// leave the range
TPFA_PAIR Dfl df_split(Dfl a, int* k) {
  const bool tiny = a.h < 1.17549435e-38f;  // subnormal: brought into range first
  const float up = tiny ? 16777216.f : 1.f;
  const float h = fl_mul(a.h, up), l = fl_mul(a.l, up);
  const int e = (int)(fl_bits(h) >> 23) & 255, e1 = (127 - e) / 2, e2 = 127 - e - e1;
  *k = 0;
  if (e == 0) return {0.f, 0.f};
  *k = e - 127 - (tiny ? 24 : 0);
  const float f1 = fl_of_bits((uint32_t)(e1 + 127) << 23), f2 = fl_of_bits((uint32_t)(e2 + 127) << 23);
  return {fl_mul(fl_mul(h, f1), f2), fl_mul(fl_mul(l, f1), f2)};
}
// q 2^k; a result below the normal range is rounded there once more
TPFA_PAIR float df_scale(float q, int k) {
  k = k > 254 ? 254 : (k < -252 ? -252 : k);
  const int k1 = k / 2, k2 = k - k1;
  return fl_mul(fl_mul(q, fl_of_bits((uint32_t)(k1 + 127) << 23)),
                fl_of_bits((uint32_t)(k2 + 127) << 23));
}

#ifdef __CUDACC__
// the same for every a >= 0 and b > 0 that are finite
__device__ __forceinline__ float df_quot(Dfl a, Dfl b) {
  constexpr float kLo = 8.8817842e-16f, kHi = 1.1258999e15f;  // 2^-50, 2^50
  if (fminf(a.h, b.h) >= kLo && fmaxf(a.h, b.h) <= kHi)
    return df_quot_mid(a, b, __fdividef(1.f, b.h));
  int ka, kb;
  const Dfl as = df_split(a, &ka), bs = df_split(b, &kb);
  return df_scale(df_quot_mid(as, bs, __fdividef(1.f, bs.h)), ka - kb);
}
#endif

}  // namespace tpfa
