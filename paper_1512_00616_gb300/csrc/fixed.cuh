// FP64 dot products of block rows in integer arithmetic.
//
// GB300 issues 1.68 FP64 FMAs per clock and SM but 63 32 x 32 + 64 bit integer multiply-adds, so
// a product of two doubles as four of the latter is nine times cheaper than one DFMA.  A group of
// doubles (a block row; the slice of a vector that belongs to one element) is held as 58-bit
// signed integers q with a common exponent E, the largest biased exponent of the group:
//   x = q 2^(E - 1079),  |q| < 2^57,
// so entries within a factor 16 of the largest keep all 53 bits and the others are rounded at
// 2^-58 of the group's scale (a DFMA chain rounds every partial sum at 2^-53 of itself).
// q is stored as hi 2^29 + lo with |hi| <= 2^28 and -2^28 <= lo < 2^28, and the dot product over
// up to kFixTerms terms is exact in three 64-bit sums (hi hi, hi lo + lo hi, lo lo).
// The one rounding is the conversion of the sum to double.
// Entries more than a factor 16 below the largest hold fewer than 53 bits, so a group that mixes variables is
// scaled first (VarScale: the energy is 1 / M^2 of the density at Mach number M).  Error of a product with the
// folded blocks against 80-bit sums, relative 2-norm over the rows of the variable that is worst (O-grid, p = 2,
// tangent right-hand sides after four products | adjoint ones), M = 0.2, 0.05, 0.01: FP64 chains 2.8e-16, 3.0e-16,
// 2.6e-16 | 3.0e-16, 2.7e-16, 2.9e-16; this 6.7e-17, 7.0e-17, 7.0e-17 | 7.5e-17, 6.5e-17, 7.0e-17.
// Infinities and NaN set E = 2047 and make the result NaN; subnormal numbers count as zero.
#pragma once

namespace pp {

// the cross sum takes two products of up to 2^56 a term: 2 63 2^56 < 2^63
constexpr int kFixTerms = 63;

struct __align__(8) Fix {
  int hi, lo;
};

// 2^e, zero below the normal range and 2^1023 above it
__device__ __forceinline__ double fix_pow2(int e) {
  if (e < -1022) return 0.0;
  return __hiloint2double((e > 1023 ? 2046 : e + 1023) << 20, 0);
}

// s + w 2^e for |w| < 2^63, rounded as one operation also where 2^e is below the normal range
__device__ __forceinline__ double fix_scale(double w, int e, double s) {
  if (e < -1022) {  // w and 2^e exchange a factor 2^128, which is exact
    w *= 0x1p-128;
    e += 128;
  }
  return fma(w, fix_pow2(e), s);
}

__device__ __forceinline__ int fix_exponent(double v) { return (__double2hiint(v) >> 20) & 0x7ff; }

// The signed 53-bit significand of v (biased exponent ex) shifted right by d - 4, rounded: d = emax - ex
// for a group with the largest exponent emax.
__device__ __forceinline__ long long fix_shifted(double v, int d) {
  const long long bits = __double_as_longlong(v);
  const long long m = (bits & 0xfffffffffffffLL) | 0x10000000000000LL;
  const int sh = d - 4;
  const long long q = sh <= 0 ? m << -sh : (sh < 55 ? (m + (1LL << (sh - 1))) >> sh : 0LL);
  return bits < 0 ? -q : q;
}

// q of v against the exponent emax as one integer (0 for zeros and subnormals)
__device__ __forceinline__ long long fix_word(double v, int emax) {
  const int ex = fix_exponent(v);
  return ex == 0 ? 0 : fix_shifted(v, emax - ex);
}

__device__ __forceinline__ Fix fix_split(long long q) {
  const int lo = (int)((q << 35) >> 35);
  return Fix{(int)((q - lo) >> 29), lo};
}

__device__ __forceinline__ Fix fix_shift(double v, int d) { return fix_split(fix_shifted(v, d)); }

// v against the group exponent emax >= fix_exponent(v)
__device__ __forceinline__ Fix fix_encode(double v, int emax) {
  const int ex = fix_exponent(v);
  return ex == 0 || emax == 0x7ff ? Fix{0, 0} : fix_shift(v, emax - ex);
}

__device__ __forceinline__ double fix_decode(Fix x, int e) {
  if (e == 0x7ff) return __longlong_as_double(0x7ff8000000000000LL);
  return (double)(((long long)x.hi << 29) + x.lo) * fix_pow2(e - 1079);
}

struct FixDot {
  long long hh, hl, ll;
  __device__ __forceinline__ void clear() { hh = hl = ll = 0; }
  __device__ __forceinline__ void add(Fix a, Fix b) {
    hh += (long long)a.hi * b.hi;
    hl += (long long)a.hi * b.lo;
    hl += (long long)a.lo * b.hi;
    ll += (long long)a.lo * b.lo;
  }
  // s + (hh 2^58 + hl 2^29 + ll) 2^(e2 - 2158), e2 the sum of the two group exponents; NaN if bad.  The unit of
  // the sum is 2^60 below it, so sums under 2^-960 become zero; Small keeps them (squared norms of small vectors;
  // its branch costs the products 3 %).
  template <bool Small = false>
  __device__ __forceinline__ double result(int e2, bool bad, double s) const {
    const long long mid = hl + (ll >> 29);                 // units of 2^29; what ll loses is 2^-85 of the scale
    const long long top = hh + (mid >> 29);                // units of 2^58
    const unsigned rest = (unsigned)mid & 0x1fffffffu;
    // top 2^29 + rest as a 64-bit integer with at least 62 significant bits, or exactly
    const int n = __clzll(top ^ (top >> 63)) - 1;          // leading bits that may be shifted out
    const int sh = n < 29 ? n : 29;
    const long long w = (top << sh) | (long long)(rest >> (29 - sh));
    const int e = e2 - 2158 + 58 - sh;                     // of w's unit
    if constexpr (Small) {
      const double r = fix_scale((double)w, e, s);
      return bad ? __longlong_as_double(0x7ff8000000000000LL) : r;
    }
    double scale = fix_pow2(e);
    if (bad) scale = __longlong_as_double(0x7ff8000000000000LL);
    return fma((double)w, scale, s);
  }
  __device__ __forceinline__ double result(int ea, int eb) const {
    return result(ea + eb, ea == 0x7ff || eb == 0x7ff, 0.0);
  }
};

}  // namespace pp
