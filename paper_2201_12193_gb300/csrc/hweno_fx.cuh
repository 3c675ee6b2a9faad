// 64-bit block fixed point for the linear part of the FP64 reconstruction.
//
// GB300 issues 2 FP64 operations per clock and SM against 64 32-bit integer
// multiply-adds with a 64-bit sum (measured: DFMA 2.0, IMAD.WIDE 52-64 per
// clock and SM, each at its full rate beside the other).  The dot products of
// the reconstruction (smoothness-indicator rows, polynomial values) therefore
// run in integers: the stencil data of one variable share an exponent and are
// held as 57-bit integers, a coefficient is a 64-bit integer, and one
// multiply-add is three 32 x 32 -> 64 products (the low x low one, below the
// last place kept, is left out): 0.05 clocks per SM against 0.5.  The data are
// deviations from the target cell's average, so their common exponent is that of the
// variation: the rounding is 2^-55 to 2^-57 of the largest deviation (FP64's is 2^-53
// of the largest datum).  Data of which a level q_l takes only a part have an exponent
// per level where their sizes differ (fx_uneven in hweno_device.cuh).  Nonlinear
// parts stay FP64.
#pragma once

#include <cuda_runtime.h>

namespace hwfx {

// x = h 2^32 + l with both halves signed (|l| <= 2^31)
struct Half2 { int h, l; };

// The halves pass through an empty asm: seen as parts of a 64-bit value, the
// compiler multiplies them as 64 x 64 bits (measured: three times the instructions).
__device__ __forceinline__ Half2 halves(long long x) {
  int h = (int)((x + 0x80000000LL) >> 32), l = (int)x;
  asm("" : "+r"(h), "+r"(l));
  return Half2{h, l};
}

// Sum of products a b: the h h products and the mixed ones (2^-32 of them).
struct Acc { long long hh, m; };

__device__ __forceinline__ Acc prod(Half2 a, int bh, int bl) {
  return Acc{(long long)a.h * bh, (long long)a.h * bl + (long long)a.l * bh};
}
__device__ __forceinline__ void mac(Acc& s, Half2 a, int bh, int bl) {
  s.hh += (long long)a.h * bh;
  s.m += (long long)a.h * bl;
  s.m += (long long)a.l * bh;
}
// the sum times 2^-F (33 <= F <= 64)
template <int F>
__device__ __forceinline__ long long scaled(const Acc& s) {
  return (s.hh << (64 - F)) + (s.m >> (F - 32));
}

constexpr int BITS = 57;        // data: |d| < 2^BITS units
constexpr int EMIN = 64;        // smallest block exponent (biased; to_fx asks for 64): the unit is 2^-1015 then,
                                // about the smallest normal double
constexpr int EMAX = 1900;      // largest one: above it the FP64 weights overflow (they are not finite)
constexpr int CBITS = 61;       // weights c_k: |c| < 2^CBITS units
constexpr int CEMIN = 64;
constexpr int CF = 61;          // the weighted sums keep the product times 2^-CF

__device__ __forceinline__ int bexp(double x) { return (__double2hiint(x) >> 20) & 0x7FF; }

// x in units of 2^(e - 1022 - B), truncated; e at least x's biased exponent and
// at least 64 (a zero then shifts out).
template <int B>
__device__ __forceinline__ long long to_fx(double x, int e) {
  const int hi = __double2hiint(x);
  const int k = min(e - ((hi >> 20) & 0x7FF), 63);
  unsigned long long m =
      ((unsigned long long)(unsigned)((hi & 0xFFFFF) | 0x100000) << 32) | (unsigned)__double2loint(x);
  m = (m << (B - 53)) >> k;
  const long long s = (long long)(hi >> 31);
  return ((long long)m ^ s) - s;
}

// A sum of squares, exact: x = h 2^30 + l with |l| <= 2^29, |x| < 2^61; the sum
// below 2^122 and at most 32 terms.  A square is four additions and shifts and
// three multiply-adds; in FP64 it took a conversion to double (15 instructions)
// and one FP64 operation, which holds its pipe for 64 clocks.
struct Squares { long long hh, hl, ll; };

__device__ __forceinline__ void add_square(Squares& s, long long x) {
  int h = (int)((x + (1LL << 29)) >> 30), l = (int)((unsigned)x - ((unsigned)h << 30));
  asm("" : "+r"(h), "+r"(l));
  s.hh += (long long)h * h;
  s.hl += (long long)h * l;
  s.ll += (long long)l * l;
}
// The sum's leading 64 bits; their unit is 2^k.
__device__ __forceinline__ unsigned long long leading(const Squares& s, int& k) {
  const unsigned __int128 t = ((unsigned __int128)(__int128)s.hh << 60) + ((unsigned __int128)(__int128)s.hl << 31) +
                              (unsigned long long)s.ll;
  unsigned long long hi = (unsigned long long)(t >> 64), lo = (unsigned long long)t;
  const bool one = hi == 0;
  if (one) { hi = lo; lo = 0; }
  const int n = __clzll((long long)hi);
  k = (one ? 0 : 64) - n;
  return (hi << (n & 63)) | (n & 63 ? lo >> (64 - n) : 0ull);
}
// The sum times 2^e as a double; results below 2^-1022 become 0, above the range infinity.
__device__ __forceinline__ double sum_of(const Squares& s, int e) {
  int k;
  const unsigned long long m = leading(s, k);
  const int f = k + e + 1085;                        // the biased exponent less 1
  const unsigned long long r = (((m >> 10) + 1) >> 1) + ((unsigned long long)(unsigned)f << 52);
  if (m == 0 || f < 0) return 0.0;
  return __longlong_as_double(f >= 2046 ? 0x7FF0000000000000LL : (long long)r);
}

// x 2^eb as a double (integer work; rounded to 53 bits, halves up); results below 2^-1022 become 0, the
// caller keeps them below the largest.
__device__ __forceinline__ double from_fx(long long x, int eb) {
  const long long s = x >> 63;
  const unsigned long long a = (unsigned long long)((x ^ s) - s);
  const int n = __clzll((long long)a);
  const unsigned long long m = (((a << (n & 63)) >> 10) + 1) >> 1;   // a carry to 2^53 raises the exponent
  const int f = 1085 - n + eb;                       // the biased exponent less 1
  const unsigned long long r = m + ((unsigned long long)(unsigned)f << 52);
  return __longlong_as_double(a && f >= 0 ? (long long)(r | ((unsigned long long)s << 63)) : 0LL);
}

// x 2^eb as a double-float pair hi + lo (truncated to 48 bits); magnitudes below 2^-126 become 0.
__device__ __forceinline__ float2 from_fx_pair(long long x, int eb) {
  const long long s = x >> 63;
  const unsigned long long a = (unsigned long long)((x ^ s) - s);
  const int n = __clzll((long long)a);
  const unsigned long long m = a << (n & 63);
  const int fe = 189 - n + eb;                       // hi's biased FP32 exponent less 1
  if (a == 0 || fe < 0) return make_float2(0.0f, 0.0f);
  const unsigned sg = (unsigned)s & 0x80000000u;
  const float hi = __uint_as_float((((unsigned)fe << 23) + (unsigned)(m >> 40)) | sg);
  // the next 32 bits, rounded to 24, times their unit 2^(8 - n + eb)
  const float unit = __uint_as_float((unsigned)max(fe - 54, 0) << 23);
  const float lo = __fmul_rn(__uint2float_rn((unsigned)(m >> 8)), unit);
  return make_float2(hi, __uint_as_float(__float_as_uint(lo) ^ sg));
}

// The sum of squares times 2^e as a pair; above FP32's range infinity.
__device__ __forceinline__ float2 sum_of_pair(const Squares& s, int e) {
  int k;
  const unsigned long long m = leading(s, k);
  if (k + e > 64) return make_float2(__int_as_float(0x7F800000), 0.0f);
  return from_fx_pair((long long)(m >> 1), k + e + 1);
}

// A float in the units of to_fx<B> at biased (FP64) exponent e.
template <int B>
__device__ __forceinline__ long long to_fx(float x, int e) {
  const int b = __float_as_int(x), f = (b >> 23) & 0xFF;
  const int k = min(e - (f + 896), 63);
  const long long m = (long long)((unsigned long long)(unsigned)(f ? (b & 0x7FFFFF) | 0x800000 : 0) << (B - 24)) >> k;
  const long long s = (long long)(b >> 31);
  return (m ^ s) - s;
}

}  // namespace hwfx
