// Exact split of a grid coordinate xi = (x - xmin) / h into its cell index
// floor(xi), the CIC fixed-point weight rint(frac(xi) * 2^20) (ties to even)
// and, when asked, the fraction frac(xi) as a double -- all from the IEEE-754
// bits of xi with integer instructions (on GB300 every FP64 instruction,
// conversions included, takes one of two FP64 slots per SM clock, while
// integer instructions are plentiful).  The results are the ones the float64
// formulas floor / subtract / multiply / rint give: floor(xi) and xi - floor(xi)
// are exact in float64, and so is the scaling by 2^20 before the rounding.
// Plain C++ so that host tests can compile it.
#pragma once
#include <stdint.h>

#if defined(__CUDACC__)
#define SC_HD __host__ __device__ __forceinline__
#else
#define SC_HD inline
#include <string.h>
#endif

namespace sc {

SC_HD uint64_t f64_bits(double v) {
#if defined(__CUDA_ARCH__)
  return (uint64_t)__double_as_longlong(v);
#else
  uint64_t b;
  memcpy(&b, &v, 8);
  return b;
#endif
}

SC_HD double bits_f64(uint64_t b) {
#if defined(__CUDA_ARCH__)
  return __longlong_as_double((long long)b);
#else
  double v;
  memcpy(&v, &b, 8);
  return v;
#endif
}

SC_HD int clz64(uint64_t v) {
#if defined(__CUDA_ARCH__)
  return __clzll((long long)v);
#else
  return __builtin_clzll(v);
#endif
}

// float -> double by moving bits (IEEE 754 binary32 -> binary64: sign kept,
// exponent rebiased by 1023 - 127, significand extended with zeros), so that
// widening a float32 field value takes integer instructions instead of a
// conversion on the FP64 pipe.  Equal to (double)f for zero, normal, infinite
// and NaN values; a subnormal float (below 2^-126) becomes zero of its sign.
SC_HD double f32_widen(float f) {
#if defined(__CUDA_ARCH__)
  const uint32_t u = (uint32_t)__float_as_uint(f);
#else
  uint32_t u;
  memcpy(&u, &f, 4);
#endif
  const uint32_t mag = u & 0x7fffffffu;
  uint32_t hi = (mag >> 3) + 0x38000000u, lo = mag << 29;
  if (mag < 0x00800000u) hi = lo = 0u;                                  // zero, subnormal
  if (mag >= 0x7f800000u) hi = 0x7ff00000u | ((mag >> 3) & 0x000fffffu);  // infinity, NaN
  return bits_f64(((uint64_t)(hi | (u & 0x80000000u)) << 32) | lo);
}

// 0 <= xi < limit (finite; -0.0 counts as 0): true, with i = floor(xi), the
// fixed-point weight a = rint((xi - i) * 2^20) in [0, 2^20], and, if f is not
// NULL, *f = xi - i.  Otherwise false (outputs unspecified).  limit <= 2^30.
SC_HD bool cic_split(double xi, int limit, int& i, int& a, double* f) {
  uint64_t b = f64_bits(xi);
  if (b == 0x8000000000000000ull) b = 0;  // -0.0
  const int e = (int)(b >> 52);           // biased exponent; the sign bit pushes negatives past 2047
  if (e >= 1023 + 30) return false;       // negative, >= 2^30, infinite or NaN
  if (e < 1023 - 60) {                    // |xi| < 2^-60 (zero, subnormal): weight rounds to 0
    i = 0;
    a = 0;
    if (f) *f = xi == 0.0 ? 0.0 : xi;
    return limit > 0;
  }
  const uint64_t m = (b & ((1ull << 52) - 1)) | (1ull << 52);  // xi = m * 2^-sh
  const int sh = 1075 - e;                                      // 23 .. 112 fraction bits
  uint64_t frac;
  if (sh <= 52) {
    i = (int)(m >> sh);
    frac = m & ((1ull << sh) - 1);
  } else {
    i = 0;
    frac = m;
  }
  if ((unsigned)i >= (unsigned)limit) return false;
  // a = frac * 2^(20 - sh), rounded to nearest, ties to even
  const int s = sh - 20;  // 3 .. 92
  if (s >= 64) {
    a = 0;
  } else {
    uint64_t q = frac >> s;
    const uint64_t r = frac & ((1ull << s) - 1), half = 1ull << (s - 1);
    if (r > half || (r == half && (q & 1ull))) ++q;
    a = (int)q;
  }
  if (f) {
    if (frac == 0) {
      *f = 0.0;
    } else {
      const int h = 63 - clz64(frac);  // leading bit of frac (h <= 52)
      const uint64_t mant = (frac << (52 - h)) & ((1ull << 52) - 1);
      *f = bits_f64(((uint64_t)(h - sh + 1023) << 52) | mant);
    }
  }
  return true;
}

// 0 <= z < limit (finite; -0.0 counts as 0): true with k = floor(z).
SC_HD bool floor_index(double z, int limit, int& k) {
  uint64_t b = f64_bits(z);
  if (b == 0x8000000000000000ull) b = 0;
  const int e = (int)(b >> 52);
  if (e >= 1023 + 30) return false;
  if (e < 1023) {
    k = 0;
  } else {
    const uint64_t m = (b & ((1ull << 52) - 1)) | (1ull << 52);
    k = (int)(m >> (1075 - e));
  }
  return (unsigned)k < (unsigned)limit;
}

SC_HD uint64_t mulhi64(uint64_t a, uint64_t b) {
#if defined(__CUDA_ARCH__)
  return __umul64hi(a, b);
#else
  return (uint64_t)(((unsigned __int128)a * b) >> 64);
#endif
}

// One axis of a grid for fix_split: the coordinate as a 63-bit integer in
// units of 2^-s, s set by the largest |x| of the grid, times inv_h as a 64-bit
// integer gives xi with F fraction bits (F near 55), without an FP64
// instruction.  That is nearer to (x - xmin) inv_h than the two rounded FP64
// operations whose decision counts, and differs from them by at most T units:
// only a coordinate within T of a place where the decision changes (a multiple
// of 2^-21: weights change half-way between multiples of 2^-20, cells at
// integers) is undecided, about one in 2^23.
struct FixAxis {
  uint64_t c;      // inv_h's significand, normalised to 2^63..2^64
  uint64_t neg_x0; // minus (xmin 2^s less what T units of xi are)
  uint64_t t;      // T
  int32_t top;     // exponent field of the largest |x| of the grid; 0: not usable (fix_split is not called)
  int32_t f;       // F
  uint32_t near;   // 2 T in units of 2^-53 (rounded up)
  int32_t limit;   // cells
};

// |(x - xmin) inv_h - its two-rounding value| <= cells 2^-52; the integers
// truncate x (1 unit of D), xmin (1), the product (1) and T's own place (2).
inline FixAxis make_fix_axis(double xmin, double inv_h, int cells) {
  FixAxis a{};
  a.limit = cells;
  if (!(inv_h > 0.0) || cells < 1 || cells > 4096) return a;
  const double xmax = xmin + cells / inv_h;
  const double big = (xmin < 0 ? -xmin : xmin) > (xmax < 0 ? -xmax : xmax) ? (xmin < 0 ? -xmin : xmin) : (xmax < 0 ? -xmax : xmax);
  const int top = (int)(f64_bits(big) >> 52), ei = (int)(f64_bits(inv_h) >> 52);
  if (top < 100 || top > 1946 || ei < 100 || ei > 1946) return a;
  const int s = 1084 - top, f = s + 1022 - ei;  // units of x; fraction bits of xi
  if (f < 43 || f > 62) return a;               // (cells 2^f < 2^63 by construction)
  a.c = ((f64_bits(inv_h) & ((1ull << 52) - 1)) | (1ull << 52)) << 11;
  a.t = (uint64_t)((((unsigned __int128)(cells + 1) << f) >> 52) + 1) + 8;
  // 2 T at most 2^-7 of the spacing of the places: else too many coordinates are undecided
  if ((2 * a.t) >> (f - 28)) return a;
  a.near = (uint32_t)(((unsigned __int128)(2 * a.t) << (85 - f)) >> 32) + 1;
  // floor(xmin 2^s): xmin = m 2^(e - 1075), |xmin| 2^s = m 2^9 >> (top - e)
  const uint64_t b = f64_bits(xmin);
  const int e = (int)((b >> 52) & 0x7ff);
  const uint64_t m = e ? (((b & ((1ull << 52) - 1)) | (1ull << 52)) << 9) : 0;
  const int sh = top - e;
  const uint64_t q = sh > 63 ? 0 : m >> sh;
  const bool rest = sh > 63 ? xmin != 0.0 : (q << sh) != m;
  int64_t x0 = (b >> 63) ? -(int64_t)q - (rest ? 1 : 0) : (int64_t)q;
  const uint64_t off = (uint64_t)((((unsigned __int128)a.t) << 64) / a.c) + 1;  // T units of xi, in units of x
  a.neg_x0 = (uint64_t)(-(x0 - (int64_t)off));
  a.f = f;
  a.top = top;
  return a;
}

// Cell i, weight w (as cic_split's) and z = xi 2^F + T of coordinate x.
// Returns 1: inside, as cic_split of the two-rounding xi says; 0: outside, as
// it says; -1: undecided, ask cic_split.
SC_HD int fix_split(const FixAxis& a, double x, int& i, int& w, uint64_t& z) {
  const uint64_t b = f64_bits(x);
  const uint32_t hi = (uint32_t)(b >> 32), lo = (uint32_t)b;
  const int e = (int)((hi >> 20) & 0x7ffu);
  const int sh = a.top - e;
  // significand << 9 (62 bits), shifted to units of 2^-s
  uint64_t m = (uint64_t)((((hi << 9) | (lo >> 23)) & 0x1fffffffu) | 0x20000000u) << 32 | (uint32_t)(lo << 9);
#if defined(__CUDA_ARCH__)
  asm("shr.b64 %0, %0, %1;" : "+l"(m) : "r"(sh));  // a shift beyond 63 gives 0
#else
  m = (sh < 0 || sh > 63) ? 0 : m >> sh;
#endif
  const uint64_t neg = (uint64_t)((int64_t)b >> 63);
  z = mulhi64((m ^ neg) - neg + a.neg_x0, a.c);
  i = (int)((uint32_t)(z >> 32) >> (a.f - 32));
  w = (int)((((uint32_t)(z >> (a.f - 21)) - ((uint32_t)i << 21)) + 1u) >> 1);
  if (sh < 0) return 0;  // beyond every node, infinite or NaN
  if ((uint32_t)((z << (85 - a.f)) >> 32) < a.near) return -1;
  return (uint32_t)i < (uint32_t)a.limit ? 1 : 0;
}

// The fraction xi - i of a decided coordinate, as a double (its leading bits
// truncated at 2^-F), by shifting its leading bit into place.
SC_HD double fix_fraction(const FixAxis& a, uint64_t z) {
  const uint64_t fr = (z - a.t) << (64 - a.f);  // in units of 2^-64
  if (fr == 0) return 0.0;
  const int n = clz64(fr);
  return bits_f64(((uint64_t)(1021 - n) << 52) + ((fr << n) >> 11));  // the leading bit adds one to the exponent
}

// Whether those fractions are as good as the two-rounding ones, which are off
// by up to cells 2^-53 in mid-grid: four units of 2^-F (x, xmin and the product
// truncated, T's place) no larger.  Not so on grids more than some thirty of
// their widths off centre.
inline bool fix_fraction_serves(const FixAxis& a) {
  return a.top && (((unsigned __int128)a.limit << a.f) >> 55) != 0;
}

// The leading 64 bits of a b from three 32 x 32-bit products, short by at most three units.
SC_HD uint64_t mulhi64_near(uint64_t a, uint64_t b) {
  const uint32_t ah = (uint32_t)(a >> 32), al = (uint32_t)a, bh = (uint32_t)(b >> 32), bl = (uint32_t)b;
#if defined(__CUDA_ARCH__)
  const uint32_t m1 = __umulhi(ah, bl), m2 = __umulhi(al, bh);
#else
  const uint32_t m1 = (uint32_t)(((uint64_t)ah * bl) >> 32), m2 = (uint32_t)(((uint64_t)al * bh) >> 32);
#endif
  return (uint64_t)ah * bh + m1 + m2;
}

// The same decision for the stand-alone deposit, which with integers alone kept
// the issue slots 74% and the FP64 pipe 0% busy: the integer of x is read from
// the bits of x + magic, magic = 1.5 2^k large enough that the sum's last bit
// is worth the same 2^-s for every x of the grid -- one FP64 instruction in
// place of some fourteen integer ones (65% and 68%, deposit.cu).
// 52 bits instead of 63: F is near 44, one coordinate in 2^18 is undecided.
struct SumAxis {
  double magic;
  uint64_t c;       // inv_h's significand, normalised to 2^63..2^64
  uint64_t neg_x0;  // minus (the bits of xmin + magic, less what T units of xi are)
  int32_t f;        // F; 0: not usable
  uint32_t near;    // 2 T in units of 2^-53 (rounded up)
  int32_t limit;    // cells
};

// T: the two roundings' cells 2^-52, one unit each for the sums of x and xmin,
// three for the product, two for T's own place.
inline SumAxis make_sum_axis(double xmin, double inv_h, int cells) {
  SumAxis a{};
  a.limit = cells;
  if (!(inv_h > 0.0) || cells < 1 || cells > 4096) return a;
  const double xmax = xmin + cells / inv_h;
  const double lo = xmin < 0 ? -xmin : xmin, hi = xmax < 0 ? -xmax : xmax, big = lo > hi ? lo : hi;
  const int top = (int)(f64_bits(big) >> 52), ei = (int)(f64_bits(inv_h) >> 52);
  if (top < 100 || top > 1946 || ei < 100 || ei > 1946) return a;
  // |x| < 2^(top - 1022) in the grid: 1.5 2^k + x stays between 2^k and 2^(k+1) for k = top - 1021, its
  // last bit worth 2^(k - 52)
  const int s = 1073 - top, f = s + 1022 - ei;
  if (f < 34 || f > 62) return a;
  const uint64_t t = (uint64_t)((((unsigned __int128)(cells + 1) << f) >> 52) + 1) + 8;
  if ((2 * t) >> (f - 28)) return a;  // 2 T above 2^-7 of the spacing of the places: too many undecided
  a.magic = bits_f64((uint64_t)(top + 2) << 52 | 1ull << 51);
  a.c = ((f64_bits(inv_h) & ((1ull << 52) - 1)) | (1ull << 52)) << 11;
  a.neg_x0 = (uint64_t)((((unsigned __int128)t) << 64) / a.c) + 1 - f64_bits(xmin + a.magic);
  a.near = (uint32_t)(((unsigned __int128)(2 * t) << (85 - f)) >> 32) + 1;
  a.f = f;
  return a;
}

// As fix_split.  (Coordinates below the grid, infinities and NaN wrap to
// integers beyond its end: the bits of the sum grow with it.)
SC_HD int sum_split(const SumAxis& a, double x, int& i, int& w) {
#if defined(__CUDA_ARCH__)
  const double v = __dadd_rn(x, a.magic);
#else
  const double v = x + a.magic;
#endif
  const uint64_t z = mulhi64_near(f64_bits(v) + a.neg_x0, a.c);
  i = (int)((uint32_t)(z >> 32) >> (a.f - 32));
  w = (int)((((uint32_t)(z >> (a.f - 21)) - ((uint32_t)i << 21)) + 1u) >> 1);
  if ((uint32_t)((z << (85 - a.f)) >> 32) < a.near) return -1;
  return (uint32_t)i < (uint32_t)a.limit ? 1 : 0;
}

}  // namespace sc
