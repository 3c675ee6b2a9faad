"""Host check of the integer reciprocal, square root, quotient and product of the FP64 forms.

The hardware's starting values may be off by its stated error either way; the
results have to be within 0.52 units in the last place for every start allowed,
and exact where the true value is representable.  A product has the bits of the
FP64 one; below the normal range it is zero.  The forms plain double takes have
IEEE's bits.
"""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(__file__), "..", "paper_2201_12193_gb300", "csrc")

SOURCE = r"""
#include "fx64_roots.h"
#include <cmath>
#include <cstdio>
#include <cstring>
#include <random>
static uint32_t bits(float f) { uint32_t b; memcpy(&b, &f, 4); return b; }
static float flt(uint32_t b) { float f; memcpy(&f, &b, 4); return f; }
static uint32_t seed(float y, float one) {          // the sum rounded towards zero
  const double s = (double)y + one;
  float f = (float)s;
  if (f > s) f = nextafterf(f, -1.0f);
  return fxr::seed_fixed(bits(f));
}
// units of the last place from n / 2^52 to sqrt(m / 2^52), m < 2^54
static double root_error(uint64_t n, uint64_t m) {
  const __int128 d = (__int128)m * ((__int128)1 << 52) - (__int128)n * n;
  return std::fabs((double)d / (2.0 * (double)n));
}
int main() {
  std::mt19937_64 g(7);
  double er = 0, es = 0;
  for (long k = 0; k < 600000; ++k) {
    uint64_t M = (1ull << 52) | (g() >> 12);
    if (k < 300) M = (1ull << 52) + k / 3;                                   // just above 1
    else if (k < 600) M = (1ull << 53) - 1 - (k - 300) / 3;                  // just below 2
    else if (k % 4 == 1) M &= ~((1ull << (g() % 53)) - 1);                   // few bits
    else if (k % 4 == 2) M |= (1ull << (g() % 52)) - 1;
    const double p = k % 3 - 1;                                              // the start's error: least, none, most
    const uint32_t h = M >> 32, l = (uint32_t)M, sb = fxr::seed_bits(h, l);
    const float m = flt(sb);
    const uint64_t q = fxr::rcp_mantissa(h, l, seed((float)((1.0 / m) * (1 + p * std::ldexp(1.0, -23))), fxr::RCP_ONE));
    // q / 2^53 against 2^52 / M: (2^105 - q M) / M
    const __int128 d = ((__int128)1 << 105) - (__int128)q * M;
    er = std::fmax(er, std::fabs((double)d / (double)M));
    if ((M & (M - 1)) == 0 && q != 1ull << 53) { printf("2^k\n"); return 1; }
    for (int odd = 0; odd < 2; ++odd) {
      const uint64_t N = M << odd;
      const float z = flt(sb + ((uint32_t)odd << 23));
      const float y = (float)((1.0 / std::sqrt((double)z)) * (1 + p * std::exp2(-22.9)));
      es = std::fmax(es, root_error(fxr::sqrt_mantissa(N >> 32, (uint32_t)N, seed(y, fxr::ROOT_ONE)), N));
    }
    const uint64_t a = (1u << 26) + g() % (1u << 26);                        // a square: a^2, a < 2^27
    const uint64_t S = a * a;                                                // m = S / 2^52 in [1, 4)
    const float sf = flt(bits((float)1.0f) + (uint32_t)((S >> 53) << 23) | (uint32_t)((S << (S >> 53 ? 11 : 12)) >> 41));
    const uint64_t r = fxr::sqrt_mantissa(S >> 32, (uint32_t)S, seed((float)(1.0 / std::sqrt((double)sf)), fxr::ROOT_ONE));
    if (r != a << 26) { printf("square %llu\n", (unsigned long long)a); return 1; }
  }
  printf("%.4f %.4f\n", er, es);
  return er <= 0.52 && es <= 0.52 ? 0 : 1;
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")
def test_reciprocal_and_root_within_half_a_unit(tmp_path):
    src = tmp_path / "roots.cpp"
    src.write_text(SOURCE)
    subprocess.check_call(["g++", "-O2", "-I", CSRC, "-o", str(tmp_path / "roots"), str(src)])
    out = subprocess.run([str(tmp_path / "roots")], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout


PRODUCT = r"""
#include "fx64_roots.h"
#include <cmath>
#include <cstdio>
#include <cstring>
#include <random>
int main() {
  std::mt19937_64 g(11);
  auto draw = [&](long k) {                            // few bits, many bits, powers of two, all exponents, zeros
    uint64_t m = g() >> 12, e = k % 3 ? 1015 + g() % 16 : g() % 2047;
    if (k % 5 == 1) m &= ~((1ull << (g() % 52)) - 1);
    if (k % 5 == 2) m |= (1ull << (g() % 52)) - 1;
    if (k % 11 == 0) m = 0;
    if (k % 13 == 0) m &= ~((1ull << 27) - 1);         // products of these meet exact ties
    if (e == 0) m = 0;
    return (g() & 1) << 63 | e << 52 | m;
  };
  for (long k = 0; k < 2000000; ++k) {
    const uint64_t x = draw(k), y = draw((long)(g() % 100000));
    double a, b;
    memcpy(&a, &x, 8);
    memcpy(&b, &y, 8);
    const double c = a * b;
    uint64_t want;
    memcpy(&want, &c, 8);
    const uint64_t got = fxr::product(x >> 32, (uint32_t)x, y >> 32, (uint32_t)y);
    if (std::fabs(c) <= 2.2250738585072014e-308 && (got << 1) == 0) continue;
    if (got != want) { printf("%a %a: %llx %llx\n", a, b, (unsigned long long)got, (unsigned long long)want); return 1; }
  }
  const uint64_t inf = 0x7FFull << 52, one = 1023ull << 52;
  const uint64_t n = fxr::product(inf >> 32, 0, one >> 32, 0);
  return (n >> 52 & 0x7FF) == 0x7FF && (n << 12) != 0 ? 0 : 2;
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")
def test_product_has_the_fp64_bits(tmp_path):
    src = tmp_path / "product.cpp"
    src.write_text(PRODUCT)
    subprocess.check_call(["g++", "-O2", "-I", CSRC, "-o", str(tmp_path / "product"), str(src)])
    out = subprocess.run([str(tmp_path / "product")], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout


NEAREST = r"""
#include "fx64_roots.h"
#include <cmath>
#include <cstdio>
#include <cstring>
#include <random>
static uint32_t bits(float f) { uint32_t b; memcpy(&b, &f, 4); return b; }
static float flt(uint32_t b) { float f; memcpy(&f, &b, 4); return f; }
static uint32_t seed(float y, float one) {          // the sum rounded towards zero
  const double s = (double)y + one;
  float f = (float)s;
  if (f > s) f = nextafterf(f, -1.0f);
  return fxr::seed_fixed(bits(f));
}
int main() {
  std::mt19937_64 g(3);
  auto draw = [&](long k) {
    uint64_t M = (1ull << 52) | (g() >> 12);
    if (k % 4 == 1) M &= ~((1ull << (g() % 53)) - 1);
    if (k % 4 == 2) M |= (1ull << (g() % 52)) - 1;
    return M;
  };
  for (long k = 0; k < 600000; ++k) {
    const uint64_t M = k < 300 ? (1ull << 52) + k / 3 : k < 600 ? (1ull << 53) - 1 - (k - 300) / 3 : draw(k);
    uint64_t A = k % 5 ? draw(k / 7) : M + k % 3 - 1;                        // equal and neighbouring mantissas too
    if (A < 1ull << 52 || A >= 1ull << 53) A = M;
    const double p = k % 3 - 1;
    const uint32_t h = M >> 32, l = (uint32_t)M, sb = fxr::seed_bits(h, l);
    const uint32_t y = seed((float)((1.0 / flt(sb)) * (1 + p * std::ldexp(1.0, -23))), fxr::RCP_ONE);
    const double m = std::ldexp((double)M, -52);
    if (std::ldexp((double)fxr::rcp_nearest(h, l, fxr::rcp_mantissa(h, l, y)), -53) != 1.0 / m) { printf("1/%a\n", m); return 1; }
    uint32_t less;
    const uint64_t q = fxr::quotient(A >> 32, (uint32_t)A, h, l, y, less);
    if (std::ldexp((double)q, -52 - (int)less) != (double)A / (double)M) { printf("%llx / %llx\n", (unsigned long long)A, (unsigned long long)M); return 1; }
    for (int odd = 0; odd < 2; ++odd) {
      const uint64_t N = M << odd;
      const float z = flt(sb + ((uint32_t)odd << 23));
      const uint32_t w = seed((float)((1.0 / std::sqrt((double)z)) * (1 + p * std::exp2(-22.9))), fxr::ROOT_ONE);
      const uint64_t r = fxr::sqrt_nearest(N >> 32, (uint32_t)N, fxr::sqrt_mantissa(N >> 32, (uint32_t)N, w));
      if (std::ldexp((double)r, -52) != std::sqrt(std::ldexp((double)N, -52))) { printf("sqrt %llx\n", (unsigned long long)N); return 1; }
    }
  }
  return 0;
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")
def test_corrected_forms_have_the_ieee_bits(tmp_path):
    src = tmp_path / "nearest.cpp"
    src.write_text(NEAREST)
    subprocess.check_call(["g++", "-O2", "-ffp-contract=off", "-I", CSRC, "-o", str(tmp_path / "nearest"), str(src)])
    out = subprocess.run([str(tmp_path / "nearest")], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout
