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
__device__ __forceinline__ fx64 sqrt(fx64 a) { return ::sqrt(a.v); }

}  // namespace hw
