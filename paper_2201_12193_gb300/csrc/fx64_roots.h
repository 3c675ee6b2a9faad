// Reciprocal and square root of a double in 32-bit integer steps, for fx64.
//
// An FP64 instruction holds a scheduler's FP64 pipe for 64 clocks, an integer
// one for 1 or 2, so a Newton correction of three to five FP64 operations (192
// to 320 clocks) costs more than the same correction in some 35 to 50 integer
// instructions.  Both start from the FP32 approximation of the mantissa's
// reciprocal (or reciprocal root), lowered so that it lies below the true
// value (the residual is then never negative), and add the first terms of the
// binomial series of the residual (Householder's iteration):
//   1/m     = y (1 + e + e^2 + ...),              e = 1 - m y   < 2^-19.8
//   sqrt(m) = m y (1 + r/2 + 3/8 r^2 + ...),      r = 1 - m y^2 < 2^-19
// The residual comes from the low words of a product whose high words cancel.
// What the series leaves out is below 2^-58 relative, the truncations of the
// fixed point below 2^-59; the result is rounded to 53 bits once, to within 0.52
// units in the last place, and the sign of the remainder corrects it to the nearest
// (rcp_nearest, sqrt_nearest).  Plain C++: also compiled for the host.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define FXR_HD __host__ __device__ __forceinline__
#else
#define FXR_HD inline
#endif

namespace fxr {

FXR_HD uint64_t wide(uint32_t a, uint32_t b) { return (uint64_t)a * b; }

// The 32-bit halves (through an empty asm on the device: products of halves the
// compiler recognises are multiplied as 64 x 64 bits).
FXR_HD void split(uint64_t x, uint32_t& h, uint32_t& l) {
  h = (uint32_t)(x >> 32);
  l = (uint32_t)x;
#ifdef __CUDA_ARCH__
  asm("" : "+r"(h), "+r"(l));
#endif
}

// The leading 24 bits of the mantissa of a double (high word h, low word l) as the bits of a float in [1, 2).
FXR_HD uint32_t seed_bits(uint32_t h, uint32_t l) { return (((h << 3) | (l >> 29)) & 0x7FFFFFu) | 0x3F800000u; }

// y - D 2^-24 in units of 2^-23 from the bits of 1 - D 2^-24 + y (rounded towards zero), 0.49 < y < 1.0000003
FXR_HD uint32_t seed_fixed(uint32_t bits_1py) { return bits_1py & 0x7FFFFFu; }
constexpr float RCP_ONE = 1.0f - 5.0f / 16777216.0f;    // D = 5: the approximation's 2^-23 and the mantissa's truncation
constexpr float ROOT_ONE = 1.0f - 4.0f / 16777216.0f;   // D = 4: 2^-22.9 and half the truncation

// 2^62 / m (at most a few units too small) for the mantissa M = mh:ml
// (2^52 <= M < 2^53, m = M 2^-52) from y in units of 2^-23.
FXR_HD uint64_t rcp62(uint32_t mh, uint32_t ml, uint32_t y) {
  const uint64_t t = wide(ml, y) + ((uint64_t)(uint32_t)(mh * y) << 32);   // m y, units 2^-75, less 1
  const uint64_t r = 0 - t;                                                // e
  uint32_t rh, rl;
  split(r, rh, rl);
  const uint64_t e = r + (wide(rh, rh) >> 11);                             // e + e^2
  split(e, rh, rl);
  const uint64_t c = wide(y, rh) + (wide(y, rl) >> 32);                    // y (e + e^2), units 2^-66
  return ((uint64_t)(y << 7) << 32) + (c >> 4);
}
// 1/m rounded, in units of 2^-53.
FXR_HD uint64_t rcp_mantissa(uint32_t mh, uint32_t ml, uint32_t y) { return (rcp62(mh, ml, y) + 256) >> 9; }

// sqrt(m) 2^52, rounded, for m = M 2^-52 in [1, 4) (M = mh:ml below 2^54) from y in units of 2^-23.
FXR_HD uint64_t sqrt_mantissa(uint32_t mh, uint32_t ml, uint32_t y) {
  uint32_t h, l;
  split(wide(y, y), h, l);                                                 // y^2, units 2^-46
  const uint64_t s = (wide(ml, l) >> 32) + wide(ml, h) + wide(mh, l) + ((uint64_t)(uint32_t)(mh * h) << 32);
  const uint64_t r = 0 - s;                                                // r, units 2^-66
  const uint32_t q = (uint32_t)(r >> 24);
  const uint64_t c = r + (wide(q, 3 * q) >> 20);                           // r/2 + 3/8 r^2, units 2^-67
  const uint64_t g = wide(mh << 10, y << 9) + (wide(ml, y) >> 13);         // m y, units 2^-62
  uint32_t gh, gl, ch, cl;
  split(g, gh, gl);
  split(c, ch, cl);
  const uint64_t d = wide(gh, ch) + ((wide(gh, cl) + wide(gl, ch)) >> 32); // m y c, units 2^-65
  return (g + (d >> 3) + 512) >> 10;
}

// rcp_mantissa's q is at most the correctly rounded one and at least that less 1
// (every truncation above lowers it): the sign of 2^105 - q M - M/2 tells which.
FXR_HD uint64_t rcp_nearest(uint32_t mh, uint32_t ml, uint64_t q) {
  uint32_t qh, ql;
  split(q, qh, ql);
  const uint64_t p = wide(ql, ml) + ((uint64_t)(uint32_t)(qh * ml + ql * mh) << 32);
  const int64_t r2 = (int64_t)((0 - p) << 1);
  return q + (r2 > (int64_t)(((uint64_t)mh << 32) | ml) ? 1u : 0u);
}
// The same for the root: one up if M 2^52 exceeds q (q + 1).
FXR_HD uint64_t sqrt_nearest(uint32_t mh, uint32_t ml, uint64_t q) {
  uint32_t qh, ql;
  split(q, qh, ql);
  const uint64_t p = wide(ql, ql) + ((uint64_t)(uint32_t)(2u * qh * ql) << 32);
  const int64_t d = (int64_t)(((uint64_t)(ml << 20) << 32) - p);
  return q + (d > (int64_t)q ? 1u : 0u);
}

// A / B for mantissas, rounded to nearest (a quotient of two doubles is never a
// tie), in units of 2^-52, of 2^-53 (less = 1) if A < B; y as for 1/B.
FXR_HD uint64_t quotient(uint32_t ah, uint32_t al, uint32_t bh, uint32_t bl, uint32_t y, uint32_t& less) {
  uint32_t qh, ql, h, l;
  split(rcp62(bh, bl, y), qh, ql);
  const uint64_t a = ((uint64_t)ah << 32) | al, b = ((uint64_t)bh << 32) | bl;
  split(a << 11, h, l);
  const uint64_t lo = wide(h, ql) + (wide(l, ql) >> 32);                   // A / B, units 2^-61
  uint32_t xh, xl;
  split(lo, xh, xl);
  const uint64_t t = wide(h, qh) + xh + ((wide(l, qh) + xl) >> 32);
  less = a < b ? 1u : 0u;
  const uint64_t q = (t + (256u >> less)) >> (9u - less);
  split(q, qh, ql);
  const uint64_t p = wide(ql, bl) + ((uint64_t)(uint32_t)(qh * bl + ql * bh) << 32);
  const int64_t r2 = (int64_t)((((uint64_t)(al << (20u + less)) << 32) - p) << 1);
  return q + (r2 > (int64_t)b ? 1u : 0u);
}

// a b for the doubles ah:al and bh:bl, rounded to nearest even as the FP64
// product is, bit for bit, where operands and result are normal.  Subnormal
// operands and results become 0, an infinite operand gives NaN.
FXR_HD uint64_t product(uint32_t ah, uint32_t al, uint32_t bh, uint32_t bl) {
  const uint32_t ea = (ah >> 20) & 0x7FFu, eb = (bh >> 20) & 0x7FFu, sg = (ah ^ bh) & 0x80000000u;
  const uint32_t mh = (ah & 0xFFFFFu) | 0x100000u, nh = (bh & 0xFFFFFu) | 0x100000u;
  uint32_t w0, w1, w2, w3, x;                        // the 106-bit product w3:w2:w1:w0
  split(wide(al, bl), x, w0);
  split(wide(mh, bl) + (wide(al, nh) + x), x, w1);
  split(wide(mh, nh) + x, w3, w2);                   // w3:w2 in [2^40, 2^42)
  const uint32_t n = w3 >> 9, k = 20u + n;           // the mantissa is the product times 2^-(32 + k)
  uint32_t h = (w3 << (32u - k)) | (w2 >> k), l = (w2 << (32u - k)) | (w1 >> k);
  const uint32_t rest = (w1 << (32u - k)) | (w0 != 0u ? 1u : 0u);
  const uint64_t q = (((uint64_t)h << 32) | l) + (rest + (l & 1u) > 0x80000000u ? 1u : 0u);
  const int e = (int)(ea + eb + n) - 1024;           // biased exponent less 1: a carry of the rounding raises it
  split(q, h, l);
  uint32_t rh = (h + ((uint32_t)e << 20)) | sg;
  const uint32_t lo = ea < eb ? ea : eb, hi = ea < eb ? eb : ea;
  if (lo == 0u || (uint32_t)e >= 2046u || hi == 0x7FFu) {
    l = 0u;
    rh = hi == 0x7FFu ? 0x7FF80000u : sg | (lo != 0u && e >= 2046 ? 0x7FF00000u : 0u);
  }
  return ((uint64_t)rh << 32) | l;
}

}  // namespace fxr
