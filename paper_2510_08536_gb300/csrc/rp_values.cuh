// Conversions, scaling, reciprocal and square root of matrix values without the FP64 pipe, shared by the value
// update (rp_update.cu) and the sliced layout (rp_sliced.cu).
//
// GB300 converts and multiplies FP64 at two lanes a clock and SM. An entry of
// the update needs its value rounded to FP32 and, for S A S, two FP64 products
// and another rounding: four of these hold the pipe for longer than HBM needs
// for the entry's 40 bytes.
#pragma once

#include "rp_common.cuh"

namespace rp {

// buffer value at slot s (bounds-checked build: slots outside [0, len) read 0)
__device__ __forceinline__ double slot_value(const double* __restrict__ buf, int32_t s, int64_t len) {
  return RP_IN(s, 0, len, kChkPermute) ? __ldg(buf + s) : 0.0;
}

// (float)v, rounded to nearest even, in integer instructions: the exponent is
// rebased, 29 fraction bits are rounded off, and a carry runs on into the
// exponent (up to infinity). Zeros, subnormal results, infinities and NaN take
// the conversion itself.
__device__ __forceinline__ float f32_rn(double v) {
  const uint32_t hi = (uint32_t)__double2hiint(v), lo = (uint32_t)__double2loint(v);
  if (((hi >> 20) & 0x7ffu) - 897u >= 254u) return (float)v;
  uint32_t f = __funnelshift_l(lo, (hi & 0x7fffffffu) - (896u << 20), 3);
  f += (lo & 0x1fffffffu) + (f & 1u) > 0x10000000u ? 1u : 0u;
  return __uint_as_float(f | (hi & 0x80000000u));
}

// The 24 leading bits of |v| as a float of v's exponent (rebased) and sign, and
// the next 23 bits: v = x + y (1 + 2^-23), |y| < 2^-23 |v|. v in FP32's normal range.
__device__ __forceinline__ float2 split_f32(double v) {
  const uint32_t hi = (uint32_t)__double2hiint(v), lo = (uint32_t)__double2loint(v);
  const uint32_t x = __funnelshift_l(lo, (hi & 0x7fffffffu) - (896u << 20), 3);
  const uint32_t sg = hi & 0x80000000u, e = ((x & 0x7f800000u) - (23u << 23)) | sg;  // exponent of the 24th bit
  return make_float2(__uint_as_float(x | sg), __uint_as_float(e | ((lo & 0x1fffffffu) >> 6)) - __uint_as_float(e));
}

// s > 0 as such a pair, or NaN where scaled_value has to take its FP64 form:
// outside [2^-20, 2^20], infinities and NaN.
__device__ __forceinline__ float2 scale_pair(double s) {
  const uint32_t e = (uint32_t)__double2hiint(s) >> 20;
  return e - 1003u <= 39u ? split_f32(s) : make_float2(__int_as_float(0x7fffffff), 0.f);
}

// fl32(v (s_i s_j)), the FP64 products rounded each, by FP32 pairs (error-free
// FMA products and sums; Dekker 1971). With u = 2^-24 a pair is off by 4 u^2
// (its low part below 2 u), so the product of the pairs a and b is off by 22 u^2
// (8 u^2 of the pairs, 4 u^2 the dropped low product, 10 u^2 two additions to
// terms of 5 u) and the one with v by 52 u^2 (4 u^2 the split of v, 10 u^2
// dropped, 16 u^2 two additions to terms of 8 u) < 2^-42; the FP64 form by
// 2^-51. Where hi is the rounded value of hi + lo + t for both t = +-2^-41 |hi|
// it is therefore the FP64 form's result; else (one entry in 2^15, v outside
// [2^-40, 2^40], NaN) ok is false and the caller computes that.
__device__ __forceinline__ float scaled_value(double v, float2 a, float2 b, bool& ok) {
  const float2 vp = split_f32(v);
  const float vh = vp.x, vl = vp.y;
  const float p = __fmul_rn(a.x, b.x);  // (intrinsics: never contracted into the sums below)
  float pe = __fmaf_rn(a.x, b.x, -p);
  pe = __fmaf_rn(a.x, b.y, pe);
  pe = __fmaf_rn(a.y, b.x, pe);
  const float r = __fmul_rn(p, vh);
  float re = __fmaf_rn(p, vh, -r);
  re = __fmaf_rn(p, vl, re);
  re = __fmaf_rn(pe, vh, re);
  const float hi = __fadd_rn(r, re), lo = __fsub_rn(re, __fsub_rn(hi, r));
  const float w = fabsf(hi) * 0x1p-41f;
  ok = (((uint32_t)__double2hiint(v) >> 20) & 0x7ffu) - 983u <= 80u && hi + (lo + w) == hi && hi + (lo - w) == hi;
  return hi;
}

// ---- 1/d and sqrt(d), rounded to nearest even, digit by digit in integers.
//
// The FP64 division and square root of the update's diagonal pass (two
// divisions, a root and their conversions: 25 FP64 instructions a row) held the
// FP64 pipe 85% of 104 us at 128^3 (30 us now). Here an FP32 seed of 22 bits gives the
// quotient (the root) 19 and then 12 (16 and 13) bits further by the exact
// remainder, which stays below 2^63 and is formed modulo 2^64; the last
// remainder decides the rounding. Ties do not occur: an odd multiple of half a
// unit would need a power of two as 2 d q (the root: a square ending in 1/4).

// v, |v| < 2^22, as a float, and back (rounded), through the bias 1.5 2^23
__device__ __forceinline__ float small_float(int v) { return __int_as_float(v + 0x4b400000) - 12582912.0f; }
__device__ __forceinline__ int small_int(float v) { return __float_as_int(v + 12582912.0f) - 0x4b400000; }

__device__ __forceinline__ double recip_rn(double d) {
  const uint32_t hi = (uint32_t)__double2hiint(d), lo = (uint32_t)__double2loint(d);
  const uint32_t e = (hi >> 20) & 0x7ffu;
  if (e - 100u > 1846u || ((hi & 0xfffffu) | lo) == 0u) return 1.0 / d;  // and powers of two
  const uint64_t m = (uint64_t)((hi & 0xfffffu) | 0x100000u) << 32 | lo;  // 2^52 < m < 2^53
  const float f = __uint_as_float(0x3f800000u | (__funnelshift_l(lo, hi, 3) & 0x7fffffu));
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(f));
  const uint32_t q1 = __float_as_uint(y + 1.0f) - 0x3f800000u;  // y 2^23: 2^75 / m to 22 bits
  int64_t r = (int64_t)(0ull - (uint64_t)q1 * m);               // 2^75 - q1 m, below 2^55
  const int q2 = small_int(small_float((int)(r >> 33)) * (y * 0x1p-1f));   // r 2^18 / m
  r = (int64_t)(((uint64_t)r << 18) - (uint64_t)(int64_t)q2 * m);          // below 2 m
  const int q3 = small_int(small_float((int)(r >> 33)) * (y * 0x1p-7f));   // r 2^12 / m
  r = (int64_t)(((uint64_t)r << 12) - (uint64_t)(int64_t)q3 * m);          // below 3/2 m
  int64_t q = ((((int64_t)q1 << 18) + q2) << 12) + q3;                     // 2^105 / m
  const int64_t h = (int64_t)(m >> 1);
  q += r > h ? 1 : r < -h ? -1 : 0;
  return __longlong_as_double((int64_t)((uint64_t)(hi & 0x80000000u) << 32) |
                              (((int64_t)(2045u - e) << 52) + (q - (1ll << 52))));
}

// a / b, a and b > 0, in the same way: 18, 17 and 17 bits (a's mantissa below b's:
// one more) after the exact first step. Exponents 1021 apart at most, so that the
// quotient is a normal number in either case (1022 below, a smaller mantissa makes
// it subnormal); else the division itself.
__device__ __forceinline__ double quot_rn(double a, double b) {
  const uint32_t ah = (uint32_t)__double2hiint(a), al = (uint32_t)__double2loint(a);
  const uint32_t bh = (uint32_t)__double2hiint(b), bl = (uint32_t)__double2loint(b);
  const int ea = (int)(ah >> 20), eb = (int)(bh >> 20);  // with the sign bit
  if ((unsigned)(ea - 1) > 2045u || (unsigned)(eb - 1) > 2045u || (unsigned)(ea - eb + 1021) > 2042u) return a / b;
  const uint64_t ma = (uint64_t)((ah & 0xfffffu) | 0x100000u) << 32 | al;
  const uint64_t mb = (uint64_t)((bh & 0xfffffu) | 0x100000u) << 32 | bl;
  const float f = __uint_as_float(0x3f800000u | (__funnelshift_l(bl, bh, 3) & 0x7fffffu));
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(f));
  // q 2^52 (2^53) for a quotient in [1, 2) ([1/2, 1))
  const int more = ma < mb ? 1 : 0;
  int64_t r = (int64_t)(ma << more), q = 1;
  r -= (int64_t)mb;  // the leading bit of the quotient: 0 <= r < mb
  const float yq = y * 0x1p-1f;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const int t = k == 0 ? 18 : 17;
    const int dgt = small_int(small_float((int)(r >> 33)) * (k == 0 ? yq : yq * 0.5f));  // r 2^t / mb
    r = (int64_t)(((uint64_t)r << t) - (uint64_t)(int64_t)dgt * mb);
    q = (q << t) + dgt;
  }
  // |r| < 3/2 mb: to nearest (ties do not occur: the quotient of two 53-bit integers is no odd
  // multiple of half a 53-bit unit)
  const int64_t h = (int64_t)(mb >> 1);
  q += r > h ? 1 : r < -h ? -1 : 0;
  return __longlong_as_double(((int64_t)(ea - eb - more + 1023) << 52) + (q - (1ll << 52)));
}

__device__ __forceinline__ double sqrt_rn(double d) {
  const uint32_t hi = (uint32_t)__double2hiint(d), lo = (uint32_t)__double2loint(d);
  if ((hi >> 20) - 1u > 2045u) return sqrt(d);  // zeros, subnormals, negative values, infinities, NaN
  const uint32_t e = hi >> 20, odd = (e & 1u) ^ 1u;
  const uint64_t m = ((uint64_t)((hi & 0xfffffu) | 0x100000u) << 32 | lo) << odd;  // 2^52 <= m < 2^54
  const float f = __uint_as_float((0x3f800000u + (odd << 23)) | (__funnelshift_l(lo, hi, 3) & 0x7fffffu));
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(f));
  const float s0 = fminf(fmaxf(f * y, 1.0f), 0x1.fffffep0f);
  const uint32_t s1 = (__float_as_uint(s0) & 0x7fffffu) | 0x800000u;  // the root of m 2^-6
  int64_t r = (int64_t)(m - ((uint64_t)s1 * s1 << 6));
  const int d1 = small_int(small_float((int)(r >> 13)) * (y * 0x1p-1f));  // r 2^9 / s1
  const int64_t t = ((int64_t)s1 << 16) + d1;                              // the root of m 2^26
  r = (int64_t)(((uint64_t)r << 26) - (uint64_t)(((int64_t)s1 << 17) + d1) * (uint64_t)(int64_t)d1);
  const int d2 = small_int(small_float((int)(r >> 23)) * (y * 0x1p-4f));  // r 2^12 / t
  int64_t q = (t << 13) + d2;                                              // the root of m 2^52
  r = (int64_t)(((uint64_t)r << 26) - (uint64_t)((t << 14) + d2) * (uint64_t)(int64_t)d2);
  q += r > q ? 1 : r <= -q ? -1 : 0;
  // (e - odd - 1023) is even
  return __longlong_as_double(((int64_t)(((int)(e - odd) - 1023) / 2 + 1023) << 52) + (q - (1ll << 52)));
}

}  // namespace rp
