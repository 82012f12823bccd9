// Correctly rounded FP64 square root and quotient from integer arithmetic.
//
// An FP64 instruction of this GPU takes 67 cycles and holds its scheduler's
// FP64 pipe for 64; a square root or a division is a chain of about ten of
// them.  Where one sits on a serial path (the ID's step: a norm downdate, then
// |R_ii|, then the reflector's quotients) the integer pipes are faster: a
// reciprocal (root) of 23 bits from the special-function unit, one Newton step
// in fixed point, two digits of the result with exact remainders, two unit
// corrections by selection, and the rounding from the remainder (the ID's
// reflector, a root and two quotients side by side: 1950 -> 1380 cycles).  The results are the
// IEEE ones (round to nearest even) and so the bits of `sqrt` and `/`; operands
// or results outside the normal range take those.
#pragma once

#include <stdint.h>
#include <string.h>

#ifndef __CUDACC__
#include <math.h>
#define HSS_FP_FN inline
#else
#define HSS_FP_FN __host__ __device__ __forceinline__
#endif

namespace hss {

HSS_FP_FN uint64_t fp_bits(double x) {
#ifdef __CUDA_ARCH__
  return static_cast<uint64_t>(__double_as_longlong(x));
#else
  uint64_t u;
  memcpy(&u, &x, 8);
  return u;
#endif
}
HSS_FP_FN double fp_from_bits(uint64_t u) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double(static_cast<long long>(u));
#else
  double x;
  memcpy(&x, &u, 8);
  return x;
#endif
}
// 1 / x and 1 / sqrt(x), relative error at most 2^-22
HSS_FP_FN float fp_rcp(float x) {
#ifdef __CUDA_ARCH__
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
#else
  return 1.0f / x;
#endif
}
HSS_FP_FN float fp_rsqrt(float x) {
#ifdef __CUDA_ARCH__
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
#else
  return 1.0f / sqrtf(x);
#endif
}

// a / b.  r0: fp_rcp of the divisor's leading 24 bits (a parameter so that a
// test can move it by its error bound).
HSS_FP_FN double fp_div_from(double a, double b, float r0) {
  const uint64_t ua = fp_bits(a), ub = fp_bits(b), one = 1ull << 52;
  const uint64_t ma = (ua & (one - 1)) | one, mb = (ub & (one - 1)) | one;
  // V = 2^83 / mb to 31 bits: r0 is 2^29 / mb to 22
  const uint32_t v0 = static_cast<uint32_t>(r0 * 0x1.0p54f);
  const uint32_t dh = static_cast<uint32_t>(mb >> 21);
  const int64_t e = static_cast<int64_t>((1ull << 62) - static_cast<uint64_t>(v0) * dh);
  const uint32_t v1 =
      v0 + static_cast<uint32_t>((static_cast<int64_t>(v0) * static_cast<int32_t>(e >> 12)) >> 50);
  // the quotient's first digit, a few units of 2^-31 below ma / mb
  const uint32_t q1 =
      static_cast<uint32_t>(((static_cast<uint64_t>(static_cast<uint32_t>(ma >> 21)) * v1) >> 31) - 8);
  const uint64_t r1 = (ma << 31) - static_cast<uint64_t>(q1) * mb;
  // the second, 22 bits further: the estimate is within one unit of the
  // floor, so one less is at most two below it
  const uint32_t q2 =
      static_cast<uint32_t>((static_cast<uint64_t>(static_cast<uint32_t>(r1 >> 26)) * v1) >> 35) - 1;
  int64_t r = static_cast<int64_t>((r1 << 22) - static_cast<uint64_t>(q2) * mb);
  const int64_t mbs = static_cast<int64_t>(mb);
  uint64_t q = (static_cast<uint64_t>(q1) << 22) + q2;
#pragma unroll
  for (int t = 0; t < 2; ++t) {
    const int64_t less = r - mbs;
    q += less >= 0 ? 1 : 0;
    r = less >= 0 ? less : r;
  }
  int64_t ex = static_cast<int64_t>((ua >> 52) & 0x7ff) - static_cast<int64_t>((ub >> 52) & 0x7ff) + 1023;
  {   // ma < mb: one more bit
    const bool more = q < (1ull << 53);
    const int64_t r2 = r << 1, less = r2 - mbs;
    const uint64_t qm = (q << 1) + (less >= 0 ? 1 : 0);
    ex -= more ? 1 : 0;
    q = more ? qm : q;
    r = more ? (less >= 0 ? less : r2) : r;
  }
  uint64_t mant = q >> 1;
  mant += (q & 1) & ((r != 0 ? 1u : 0u) | (mant & 1));
  return fp_from_bits(((ua ^ ub) & (1ull << 63)) | ((static_cast<uint64_t>(ex) << 52) + (mant - one)));
}

HSS_FP_FN double fp_div(double a, double b) {
  const uint64_t ua = fp_bits(a), ub = fp_bits(b);
  const int ea = static_cast<int>((ua >> 52) & 0x7ff), eb = static_cast<int>((ub >> 52) & 0x7ff);
  const int ex = ea - eb;
  if (ea == 0 || eb == 0 || ea == 0x7ff || eb == 0x7ff || ex < -1020 || ex > 1020) return a / b;
  const uint32_t lead = static_cast<uint32_t>(((ub & ((1ull << 52) - 1)) | (1ull << 52)) >> 29);
  return fp_div_from(a, b, fp_rcp(static_cast<float>(lead)));
}

// sqrt(a) for a normal a > 0; y0: fp_rsqrt of the leading 24 bits
HSS_FP_FN double fp_sqrt_from(double a, float y0) {
  const uint64_t ua = fp_bits(a), one = 1ull << 52;
  int ex = static_cast<int>(ua >> 52) - 1023;
  uint64_t x = (ua & (one - 1)) | one;
  if (ex & 1) {
    x <<= 1;
    --ex;
  }
  // Y = 2^57 / sqrt(x) to 30 bits
  const uint32_t v0 = static_cast<uint32_t>(y0 * 0x1.0p42f);
  const uint32_t t = static_cast<uint32_t>((static_cast<uint64_t>(v0) * v0) >> 31);
  const uint32_t xh = static_cast<uint32_t>(x >> 22);
  const int64_t e = static_cast<int64_t>((1ull << 61) - static_cast<uint64_t>(t) * xh);
  const uint32_t v1 =
      v0 + static_cast<uint32_t>((static_cast<int64_t>(v0) * static_cast<int32_t>(e >> 12)) >> 50);
  // sqrt(x) 2^4, a few units below
  const uint32_t s1 = static_cast<uint32_t>(((static_cast<uint64_t>(xh) * v1) >> 31) - 6);
  const uint64_t r1 = (x << 8) - static_cast<uint64_t>(s1) * s1;
  const uint64_t dl = (static_cast<uint64_t>(static_cast<uint32_t>(r1 >> 4)) * v1) >> 35;
  // floor(sqrt(x) 2^27): the estimate is the floor or one below it (one less,
  // so that an estimate above it would be corrected too)
  uint64_t s = (static_cast<uint64_t>(s1) << 23) + dl - 1;
  int64_t r = static_cast<int64_t>((x << 54) - s * s);
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const int64_t less = r - static_cast<int64_t>(2 * s + 1);
    r = less >= 0 ? less : r;
    s += less >= 0 ? 1 : 0;
  }
  uint64_t mant = s >> 1;
  mant += (s & 1) & ((r != 0 ? 1u : 0u) | (mant & 1));
  return fp_from_bits((static_cast<uint64_t>((ex >> 1) + 1023) << 52) + (mant - one));
}

HSS_FP_FN double fp_sqrt(double a) {
  const uint64_t ua = fp_bits(a);
  const int ea = static_cast<int>(ua >> 52);   // the sign bit makes a negative a too large
  if (ea == 0 || ea >= 0x7ff) return sqrt(a);
  uint64_t x = (ua & ((1ull << 52) - 1)) | (1ull << 52);
  if (((ea - 1023) & 1) != 0) x <<= 1;
  return fp_sqrt_from(a, fp_rsqrt(static_cast<float>(static_cast<uint32_t>(x >> 30))));
}

}  // namespace hss
