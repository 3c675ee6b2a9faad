// The compute precision of the FP64 forms: a double whose every operation is
// FP64, as a type of its own because the functions that carry the work have
// versions for it that GB300's scarce FP64 pipe needs (recon1d / recon2d in
// block fixed point, rcp).  Plain double keeps the plain versions (all in FP64,
// IEEE reciprocals): the learned indicator's stages use it.  Its network
// decides by a threshold on BF16-rounded features, which are noise-sized
// wherever the data hardly vary, so a last-bit change of the point values
// moves decisions (measured with fx64 there: one to three cells of 1024^2
// change sides per step on blast data).
#pragma once

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
// Square root: the hardware's approximation y of 1/sqrt(x) (2^-20) and one
// third-order step of Householder's iteration on g = x y, g (1 + r/2 + 3/8 r^2)
// with r = 1 - g y: within 0.75 units in the last place (half of g's rounding and
// the last one), five FP64 operations where the IEEE root takes nine (measured
// rates).  Zero gives zero, a negative argument NaN, infinity NaN.
__device__ __forceinline__ fx64 sqrt(fx64 a) {
  const double x = a.v;
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double g = x * y;
  const double r = ::fma(-g, y, 1.0);
  const double s = ::fma(g, ::fma(r, 0.375, 0.5) * r, g);
  return ((__double2hiint(x) << 1) | __double2loint(x)) == 0 ? x : s;
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
