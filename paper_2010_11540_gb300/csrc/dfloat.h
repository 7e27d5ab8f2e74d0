// Sums of two floats (F2: h + l, about 47 significant bits) for the parts of
// the maps that need fewer bits than the state itself.  GB300 issues one FP64
// warp instruction per 64 clocks and SM sub-partition but a float instruction
// every clock, so a correction worked out in some twenty float instructions is
// several times cheaper than the two or three float64 instructions it replaces.
// A correction c to a float64 value v is safe here when |c| 2^-46 stays below
// v's own rounding; each caller states why it does.
//
// Error-free steps: the product's error by a fused multiply-add, the sum's by
// Knuth's two-sum or, for |a| >= |b|, Dekker's fast two-sum (T. J. Dekker,
// Numer. Math. 18 (1971) 224).  Plain C++ so that host tests can compile it
// (with contraction off: the device code spells out each rounding).
#pragma once
#include "fixpt.h"
#if !defined(__CUDACC__)
#include <math.h>
#endif

namespace sc {

#if defined(__CUDA_ARCH__)
SC_HD float f_mul(float a, float b) { return __fmul_rn(a, b); }
SC_HD float f_add(float a, float b) { return __fadd_rn(a, b); }
SC_HD float f_sub(float a, float b) { return __fsub_rn(a, b); }
SC_HD float f_fma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
SC_HD uint32_t f_bits(float v) { return __float_as_uint(v); }
SC_HD float bits_f(uint32_t b) { return __uint_as_float(b); }
#else
SC_HD uint32_t f_bits(float v) {
  uint32_t b;
  memcpy(&b, &v, 4);
  return b;
}
SC_HD float bits_f(uint32_t b) {
  float v;
  memcpy(&v, &b, 4);
  return v;
}
SC_HD float f_mul(float a, float b) { return a * b; }
SC_HD float f_add(float a, float b) { return a + b; }
SC_HD float f_sub(float a, float b) { return a - b; }
SC_HD float f_fma(float a, float b, float c) { return fmaf(a, b, c); }
#endif

struct F2 {
  float h, l;
};

// High word of |v|: what range tests compare (a NaN or infinity is 0x7ff00000 or more).
SC_HD uint32_t abs_hi(double v) { return (uint32_t)(f64_bits(v) >> 32) & 0x7fffffffu; }
constexpr uint32_t kHi2p50 = (1023u + 50u) << 20;  // high word of 2^50

// v as h + l, by moving bits (no FP64 conversion): h takes the leading 24
// significant bits, l the 23 below them (truncated: |error| < 2^-46 |v|).
// |v| < 2^127 (callers test); below 2^-95 it counts as 2^-95 in size.
SC_HD F2 f2_split(double v) {
  const uint64_t b = f64_bits(v);
  const uint32_t hi = (uint32_t)(b >> 32), lo = (uint32_t)b;
  uint32_t a = hi & 0x7fffffffu;
  a = a < 0x3a000000u ? 0x3a000000u : a;
  // sign | exponent - 896 | 23 bits; the shift drops the exponent's top two bits, the subtraction wraps
  const uint32_t f = (((a << 3) | (lo >> 29)) - 0xc0000000u) | (hi & 0x80000000u);
  const uint32_t e = (f & 0xff800000u) - (23u << 23);
  const float l = f_sub(bits_f(e | ((lo >> 6) & 0x7fffffu)), bits_f(e));
  return F2{bits_f(f), l};
}

// a + b as a sum and its error, any order of sizes
SC_HD F2 two_sum(float a, float b) {
  const float s = f_add(a, b), t = f_sub(s, a);
  return F2{s, f_add(f_sub(a, f_sub(s, t)), f_sub(b, t))};
}
SC_HD F2 f2_add(F2 a, F2 b) {
  F2 s = two_sum(a.h, b.h);
  s.l = f_add(s.l, f_add(a.l, b.l));
  return s;
}
SC_HD F2 f2_neg(F2 a) { return F2{-a.h, -a.l}; }
SC_HD F2 f2_mul(F2 a, F2 b) {
  const float p = f_mul(a.h, b.h);
  return F2{p, f_fma(a.l, b.h, f_fma(a.h, b.l, f_fma(a.h, b.h, -p)))};
}
SC_HD F2 f2_sqr(F2 a) {
  const float p = f_mul(a.h, a.h);
  return F2{p, f_fma(f_add(a.h, a.h), a.l, f_fma(a.h, a.h, -p))};
}

// h + l as a double, by moving bits: the sum rounded to a float s, the rest
// counted in units of s's last float64 bit (half as large below a power of
// two).  Good to 2^-52 of itself down to 2^-75; below, the low part fades out,
// and |h + l| < 2^-126 gives 0.
SC_HD double f2_to_double(F2 a) {
  const float s = f_add(a.h, a.l);
  const float r = f_sub(a.l, f_sub(s, a.h));
  const uint32_t u = f_bits(s), mag = u & 0x7fffffffu;
  const uint32_t e = mag >> 23;
  // 2^(52 - exponent): biased 127 + 52 - (e - 127), kept representable for tiny s
  const float t = f_mul(bits_f(f_bits(r) ^ (u & 0x80000000u)), bits_f((306u - (e < 52u ? 52u : e)) << 23));
#if defined(__CUDA_ARCH__)
  int k = __float2int_rn(t);
#else
  int k = (int)lrintf(t);
#endif
  if ((mag & 0x7fffffu) == 0u && k < 0) k += k;
  const uint64_t b = ((uint64_t)((mag >> 3) + 0x38000000u) << 32 | (uint64_t)(uint32_t)(mag << 29)) + (uint64_t)(int64_t)k;
  return bits_f64(mag < 0x00800000u ? 0ull : b | (uint64_t)(u & 0x80000000u) << 32);
}

// (1 - u)^(-1/2) - 1 for 0 <= u < 2^-10 by its power series,
//   u/2 + u^2 (3/8 + 5/16 u + 35/128 u^2 + 63/256 u^3),
// absolute error below 2^-54: the factor 1 + w of a drift then has float64
// accuracy.  (Next term 231/1024 u^6 < 2^-62; the bracket's float part is off
// by at most u 2^-25, so u^3 2^-25 < 2^-55.)
constexpr float kDriftMaxU = 0.0009765625f;
SC_HD F2 rsqrt1m_series(F2 u) {
  const float s = f_mul(u.h, f_fma(u.h, f_fma(u.h, 0.24609375f, 0.2734375f), 0.3125f));
  const float vh = f_add(0.375f, s);
  const F2 v{vh, f_add(f_sub(0.375f, vh), s)};
  const F2 z = f2_mul(f2_sqr(u), v);
  const float uh = f_mul(0.5f, u.h), wh = f_add(uh, z.h);
  return F2{wh, f_add(f_fma(0.5f, u.l, f_add(f_sub(uh, wh), z.h)), z.l)};
}

// (1 - u)^(-1/2) - 1 over the wider range |u| < 2^-7 (either sign),
//   u/2 + u^2 (3/8 + u (5/16 + u (35/128 + 63/256 u + 231/1024 u^2 + 429/2048 u^3))),
// absolute error below 2^-53: the leading sum's own 2^-46 of 2^-8, halved by its
// rounding; the innermost float part's u 2^-25 enters times u^4, and the next
// term is 6435/32768 u^8 < 2^-58.
constexpr float kSlopeMaxU = 0.0078125f;
SC_HD F2 rsqrt1m_wide(F2 u) {
  const float s = f_mul(u.h, f_fma(u.h, f_fma(u.h, 0.20947265625f, 0.2255859375f), 0.24609375f));
  const float qh = f_add(0.2734375f, s);
  const F2 q{qh, f_add(f_sub(0.2734375f, qh), s)};
  const F2 t = f2_add(F2{0.3125f, 0.f}, f2_mul(u, q));
  const F2 v = f2_add(F2{0.375f, 0.f}, f2_mul(u, t));
  const F2 z = f2_mul(f2_sqr(u), v);
  return f2_add(F2{f_mul(0.5f, u.h), f_mul(0.5f, u.l)}, z);
}

// 1 - sqrt(1 - v) for |v| < 2^-9 by its power series,
//   v/2 + v^2 (1/8 + v/16 + 5/128 v^2 + 7/256 v^3 + 21/1024 v^4),
// absolute error below 2^-54 (next term 33/2048 v^7 < 2^-68; the bracket's
// float part is off by at most v 2^-28).
constexpr float kSlipMaxV = 0.001953125f;
SC_HD F2 one_minus_sqrt1m(F2 v) {
  const float s =
      f_mul(v.h, f_fma(v.h, f_fma(v.h, f_fma(v.h, 0.0205078125f, 0.02734375f), 0.0390625f), 0.0625f));
  const float bh = f_add(0.125f, s);
  const F2 b{bh, f_add(f_sub(0.125f, bh), s)};
  const F2 z = f2_mul(f2_sqr(v), b);
  const float vh = f_mul(0.5f, v.h), wh = f_add(vh, z.h);
  return F2{wh, f_add(f_fma(0.5f, v.l, f_add(f_sub(vh, wh), z.h)), z.l)};
}

// An F2 in the place of a double (the same eight bytes), and back.
SC_HD double f2_pack(F2 a) { return bits_f64((uint64_t)f_bits(a.l) << 32 | f_bits(a.h)); }
SC_HD F2 f2_unpack(double v) {
  const uint64_t b = f64_bits(v);
  return F2{bits_f((uint32_t)b), bits_f((uint32_t)(b >> 32))};
}

// sg's change over a thick quadrupole (maps.cuh: map_quad),
//   ps Lg - L4 (px0^2 + py0^2) - qi (x1 px1 + y1 py1 + x0 (K x0 - px0) - y0 (K y0 + py0)),
// K = L k1, L4 = L/4, Lg = L/gamma0^2, qi = 1/(4(1-ps)).  A product is good to 3 2^-46 (the
// neglected l l and three roundings), a sum to 2^-46: with three products and five sums in a
// row every term comes out within 14 2^-46 of itself.
SC_HD F2 quad_slip(F2 x0, F2 px0, F2 y0, F2 py0, F2 x1, F2 px1, F2 y1, F2 py1, F2 ps, F2 qi, F2 L4, F2 Lg, F2 K) {
  const F2 ax = f2_add(f2_mul(K, x0), f2_neg(px0)), ay = f2_add(f2_mul(K, y0), py0);
  const F2 t = f2_add(f2_add(f2_mul(x1, px1), f2_mul(y1, py1)), f2_add(f2_mul(x0, ax), f2_neg(f2_mul(y0, ay))));
  const F2 pp = f2_add(f2_sqr(px0), f2_sqr(py0));
  return f2_add(f2_mul(ps, Lg), f2_neg(f2_add(f2_mul(pp, L4), f2_mul(t, qi))));
}

// The sum of the sizes of quad_slip's terms, its differences' two sides counted
// apart: what the 14 2^-46 above are of.
SC_HD float quad_slip_size(F2 x0, F2 px0, F2 y0, F2 py0, F2 x1, F2 px1, F2 y1, F2 py1, F2 ps, F2 qi, F2 L4, F2 Lg, F2 K) {
  const float k = fabsf(K.h);
  const float ax = f_fma(k, fabsf(x0.h), fabsf(px0.h)), ay = f_fma(k, fabsf(y0.h), fabsf(py0.h));
  const float t = f_fma(fabsf(x1.h), fabsf(px1.h),
                        f_fma(fabsf(y1.h), fabsf(py1.h), f_fma(fabsf(x0.h), ax, f_mul(fabsf(y0.h), ay))));
  const float pp = f_fma(px0.h, px0.h, f_mul(py0.h, py0.h));
  return f_fma(fabsf(ps.h), fabsf(Lg.h), f_fma(pp, L4.h, f_mul(t, fabsf(qi.h))));
}

}  // namespace sc
