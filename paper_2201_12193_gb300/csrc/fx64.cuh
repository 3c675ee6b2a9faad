// The compute precision of the FP64 forms: a double whose every operation is
// FP64, as a type of its own because the functions that carry the work have
// versions for it that GB300's scarce FP64 pipe needs (recon1d / recon2d in
// block fixed point, rcp and sqrt in integers).  Plain double keeps the plain
// versions (IEEE's results throughout): the learned indicator's stages use it.  Its network
// decides by a threshold on BF16-rounded features, which are noise-sized
// wherever the data hardly vary, so a last-bit change of the point values
// moves decisions (measured with fx64 there: one to three cells of 1024^2
// change sides per step on blast data).
#pragma once

#include "fx64_roots.h"

namespace hw {

struct fx64 {
  double v;
  fx64() = default;
  __host__ __device__ constexpr fx64(double x) : v(x) {}
  __host__ __device__ explicit constexpr operator double() const { return v; }
};

__device__ __forceinline__ fx64 operator+(fx64 a, fx64 b) { return a.v + b.v; }
__device__ __forceinline__ fx64 operator-(fx64 a, fx64 b) { return a.v - b.v; }
__device__ __forceinline__ fx64 operator*(fx64 a, fx64 b) { return a.v * b.v; }
__device__ __forceinline__ fx64 operator/(fx64 a, fx64 b) { return a.v / b.v; }
__device__ __forceinline__ fx64 operator-(fx64 a) { return -a.v; }
__device__ __forceinline__ fx64& operator+=(fx64& a, fx64 b) { a.v += b.v; return a; }
__device__ __forceinline__ fx64& operator-=(fx64& a, fx64 b) { a.v -= b.v; return a; }
__device__ __forceinline__ fx64& operator*=(fx64& a, fx64 b) { a.v *= b.v; return a; }
__device__ __forceinline__ bool operator<(fx64 a, fx64 b) { return a.v < b.v; }
__device__ __forceinline__ bool operator>(fx64 a, fx64 b) { return a.v > b.v; }
__device__ __forceinline__ bool operator<=(fx64 a, fx64 b) { return a.v <= b.v; }
__device__ __forceinline__ bool operator>=(fx64 a, fx64 b) { return a.v >= b.v; }
__device__ __forceinline__ bool operator==(fx64 a, fx64 b) { return a.v == b.v; }
__device__ __forceinline__ fx64 fma(fx64 a, fx64 b, fx64 c) { return ::fma(a.v, b.v, c.v); }
// Square root and reciprocal in integers (fx64_roots.h), correctly rounded by the
// remainder's sign, where the FP64 steps held the FP64 pipe for five and three operations.
// At 2048^2: Step 3 8.0 -> 5.8 ms per launch, the reconstruction 5.5 -> 5.1 (without the last
// rounding step, 1.2 % of a step less).
__device__ __forceinline__ unsigned long long root_bits(unsigned h, unsigned l) {   // of a positive normal h:l
  const unsigned odd = ~(h >> 20) & 1u;              // the mantissa in [1, 4), the exponent left even
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(__uint_as_float(fxr::seed_bits(h, l) + (odd << 23))));
  unsigned mh = (h & 0xFFFFFu) | 0x100000u;
  mh = odd ? __funnelshift_l(l, mh, 1) : mh;
  unsigned long long s = fxr::sqrt_mantissa(mh, l << odd, fxr::seed_fixed(__float_as_uint(__fadd_rz(y, fxr::ROOT_ONE))));
  s = fxr::sqrt_nearest(mh, l << odd, s);
  return s + ((unsigned long long)((((h >> 20) + 1023u) >> 1) - 1u) << 52);
}
__device__ __forceinline__ unsigned long long rcp_bits(unsigned h, unsigned l) {   // biased exponent 1 .. 2044
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(__uint_as_float(fxr::seed_bits(h, l))));
  const unsigned mh = (h & 0xFFFFFu) | 0x100000u;
  unsigned long long s = fxr::rcp_mantissa(mh, l, fxr::seed_fixed(__float_as_uint(__fadd_rz(y, fxr::RCP_ONE))));
  s = fxr::rcp_nearest(mh, l, s);
  return s + ((unsigned long long)((2044u - ((h >> 20) & 0x7FFu)) | ((h >> 20) & 0x800u)) << 52);
}
// Outside IEEE's common range (its results there cost a branch at every call, 1 to 4 % of a
// step).  Root: zero gives zero; a negative argument, a subnormal one, infinity and NaN
// give NaN.  Reciprocal: zero, a subnormal argument, infinity and NaN give NaN; results
// below 2^-1022 become 0.
__device__ __forceinline__ fx64 sqrt(fx64 a) {
  const unsigned h = (unsigned)__double2hiint(a.v), l = (unsigned)__double2loint(a.v);
  const unsigned long long s = root_bits(h, l);
  if (h - 0x00100000u < 0x7FE00000u) return __longlong_as_double((long long)s);
  return ((h << 1) | l) == 0u ? a.v : __longlong_as_double(0x7FF8000000000000LL);
}
__device__ __forceinline__ fx64 reciprocal(fx64 a) {
  const unsigned h = (unsigned)__double2hiint(a.v), l = (unsigned)__double2loint(a.v);
  const unsigned e = (h >> 20) & 0x7FFu;
  const unsigned long long s = rcp_bits(h, l);
  if (e - 1u < 2044u) return __longlong_as_double((long long)s);
  return e == 0x7FFu || e == 0u ? __longlong_as_double(0x7FF8000000000000LL) : 0.0;
}
// IEEE's root, reciprocal and quotient of plain double, the common range in integers
// (the learned form's stages, 1024^2: 26.2 -> 23.7 ms a step; the same bits).
__device__ __forceinline__ double sqrt_ieee(double x) {
  const unsigned h = (unsigned)__double2hiint(x);
  if (h - 0x00100000u < 0x7FE00000u) return __longlong_as_double((long long)root_bits(h, (unsigned)__double2loint(x)));
  return __dsqrt_rn(x);
}
__device__ __forceinline__ double rcp_ieee(double x) {
  const unsigned h = (unsigned)__double2hiint(x);
  if (((h >> 20) & 0x7FFu) - 1u < 2044u) return __longlong_as_double((long long)rcp_bits(h, (unsigned)__double2loint(x)));
  return __drcp_rn(x);
}
__device__ __forceinline__ double div_ieee(double x, double z) {
  const unsigned h = (unsigned)__double2hiint(x), l = (unsigned)__double2loint(x);
  const unsigned g = (unsigned)__double2hiint(z), k = (unsigned)__double2loint(z);
  const unsigned eh = (h >> 20) & 0x7FFu, eg = (g >> 20) & 0x7FFu, sg = (h ^ g) & 0x80000000u;
  const unsigned e = eh + 1022u - eg;                // the biased exponent less 1, for A >= B
  if (eg - 1u < 2046u && eh - 1u < 2046u && e - 1u < 2044u) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(__uint_as_float(fxr::seed_bits(g, k))));
    unsigned less;
    const unsigned long long q =
        fxr::quotient((h & 0xFFFFFu) | 0x100000u, l, (g & 0xFFFFFu) | 0x100000u, k,
                      fxr::seed_fixed(__float_as_uint(__fadd_rz(y, fxr::RCP_ONE))), less);
    return __longlong_as_double((long long)((q + ((unsigned long long)(e - less) << 52)) | ((unsigned long long)sg << 32)));
  }
  return eg - 1u < 2046u && ((h << 1) | l) == 0u ? __hiloint2double((int)sg, 0) : __ddiv_rn(x, z);
}

// a b in integers: the same bits as a * b where operands and result are normal.  Subnormal
// operands and products below 2^-1022 (before rounding) become 0, infinite operands NaN.
__device__ __forceinline__ fx64 product(fx64 a, fx64 b) {
  return __longlong_as_double((long long)fxr::product((unsigned)__double2hiint(a.v), (unsigned)__double2loint(a.v),
                                                      (unsigned)__double2hiint(b.v), (unsigned)__double2loint(b.v)));
}

// Comparisons and halving by integer work: an FP64 compare takes the FP64 pipe's
// full issue slot.  NaN compares false; -0 counts as negative.
__device__ __forceinline__ bool nonneg(fx64 a) { return (unsigned)__double2hiint(a.v) < 0x7FF00000u; }   // 0 <= a, finite
__device__ __forceinline__ bool nonpos(fx64 a) {
  const unsigned h = (unsigned)__double2hiint(a.v);
  return (h >= 0x80000000u && h <= 0xFFF00000u) || (h | (unsigned)__double2loint(a.v)) == 0u;
}
__device__ __forceinline__ bool below(fx64 a, fx64 b) {   // a < b for b >= 0 or NaN
  const long long x = __double_as_longlong(a.v), y = __double_as_longlong(b.v);
  return x < y && y <= 0x7FF0000000000000LL;
}
__device__ __forceinline__ fx64 half(fx64 a) {   // a / 2; results below 2^-1022 become 0
  const int h = __double2hiint(a.v), e = (h >> 20) & 0x7FF;
  if ((unsigned)(e - 2) < 0x7FDu) return __hiloint2double(h - 0x100000, __double2loint(a.v));
  return e == 0x7FF ? a.v : 0.0;
}

}  // namespace hw
