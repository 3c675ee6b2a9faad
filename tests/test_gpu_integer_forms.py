"""The device forms of the integer root, reciprocal, quotient and product against
the hardware's FP64 operations, bit for bit: all exponents, both signs, the edges
of the integer range, zeros, subnormals, infinities and NaN.  Plain double's forms
are IEEE's throughout; those of fx64 where operand and result are normal, with
what fx64.cuh states elsewhere."""
import ctypes
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

CSRC = os.path.join(os.path.dirname(__file__), "..", "paper_2201_12193_gb300", "csrc")

SOURCE = r"""
#include <cuda_runtime.h>
#include "fx64.cuh"
using namespace hw;
__global__ void forms(const double* a, const double* b, double* got, double* want, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double x = a[i], y = b[i];
  const double g[7] = {sqrt_ieee(x), rcp_ieee(x), div_ieee(x, y), sqrt(fx64(x)).v, reciprocal(fx64(x)).v,
                       product(fx64(x), fx64(y)).v, half(fx64(x)).v};
  const double w[7] = {__dsqrt_rn(x), __drcp_rn(x), __ddiv_rn(x, y), __dsqrt_rn(x), __drcp_rn(x), __dmul_rn(x, y),
                       __dmul_rn(x, 0.5)};
  for (int k = 0; k < 7; ++k) { got[k * n + i] = g[k]; want[k * n + i] = w[k]; }
}
extern "C" int run_forms(const double* a, const double* b, double* got, double* want, int n) {
  forms<<<(n + 127) / 128, 128>>>(a, b, got, want, n);
  return (int)cudaDeviceSynchronize();
}
"""
LEAST = 2.0 ** -1022
NAMES = ["sqrt_ieee", "rcp_ieee", "div_ieee", "fx64 sqrt", "fx64 reciprocal", "fx64 product", "fx64 half"]


@pytest.fixture(scope="module")
def forms(tmp_path_factory):
    import torch
    from paper_2201_12193_gb300 import build
    d = tmp_path_factory.mktemp("forms")
    (d / "forms.cu").write_text(SOURCE)
    subprocess.check_call([build.nvcc(), *build.ARCH, "-O3", "-std=c++17", "-Xcompiler", "-fPIC", "-shared", "-I" + CSRC,
                           "-o", str(d / "forms.so"), str(d / "forms.cu")])
    lib = ctypes.CDLL(str(d / "forms.so"))
    lib.run_forms.argtypes = [ctypes.c_void_p] * 4 + [ctypes.c_int]

    def run(a, b):
        x, y = torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda()
        got = torch.empty(7, len(a), dtype=torch.float64, device="cuda")
        want = torch.empty_like(got)
        torch.cuda.synchronize()
        assert lib.run_forms(x.data_ptr(), y.data_ptr(), got.data_ptr(), want.data_ptr(), len(a)) == 0
        return got.cpu().numpy(), want.cpu().numpy()
    return run


def _draw(kind, n, seed):
    g = np.random.default_rng(seed)
    m = g.integers(0, 1 << 52, n, dtype=np.uint64)
    few = g.integers(0, 53, n).astype(np.uint64)
    m = np.where(g.random(n) < 0.3, m >> few << few, m)
    m = np.where(g.random(n) < 0.1, np.uint64((1 << 52) - 1) - m % np.uint64(64), m)
    sign = g.integers(0, 2, n).astype(np.uint64) << np.uint64(63)
    if kind == "near one":
        e = g.integers(1015, 1032, n)
    elif kind == "all exponents":
        e = g.integers(1, 2047, n)
    elif kind == "edges":
        e = g.choice([0, 1, 2, 3, 52, 53, 1022, 1023, 1024, 2043, 2044, 2045, 2046], n)
    else:
        e = g.choice([0, 2047], n)
        m = np.where(g.random(n) < 0.5, 0, m)
    return (sign | e.astype(np.uint64) << np.uint64(52) | m.astype(np.uint64)).view(np.float64)


def _stated(form, a, b, want):
    """fx64's results: `want` in the normal range, elsewhere as fx64.cuh has them."""
    def exps(x):
        return (x.view(np.uint64) >> np.uint64(52) & np.uint64(2047)).astype(int)
    ea, eb, zero = exps(a), exps(b), np.zeros_like(a)
    if form == 3:
        return np.where(a == 0, a, np.where((ea > 0) & (ea < 2047) & (a > 0), want, np.nan))
    if form == 4:
        return np.where((ea == 0) | (ea == 2047), np.nan, np.where(ea > 2044, zero, want))
    if form == 5:
        signed = np.copysign(zero, np.copysign(1.0, a) * np.copysign(1.0, b))
        with np.errstate(all="ignore"):
            low = (ea == 0) | (eb == 0) | (np.abs(a * b) < LEAST)
        for i in np.flatnonzero(~low & (np.abs(want) == LEAST)):     # below it before rounding
            low[i] = abs(Fraction(a[i]) * Fraction(b[i])) < Fraction(LEAST)
        return np.where((ea == 2047) | (eb == 2047), np.nan, np.where(low, signed, want))
    if form == 6:
        return np.where(ea < 2, zero, want)
    return want


@pytest.mark.parametrize("form", range(7), ids=NAMES)
@pytest.mark.parametrize("other", ["near one", "all exponents", "edges", "special"])
@pytest.mark.parametrize("kind", ["near one", "all exponents", "edges", "special"])
def test_bits_of_the_hardware_operations(forms, form, kind, other):
    n = 200000
    a, b = _draw(kind, n, 1), _draw(other, n, 2)
    if form in (0, 3):
        a = np.where(np.arange(n) % 16 == 0, a, np.abs(a))
    got, want = (x[form] for x in forms(a, b))
    want = _stated(form, a, b, want)
    bad = (got.view(np.uint64) != want.view(np.uint64)) & ~(np.isnan(got) & np.isnan(want))
    k = np.flatnonzero(bad)[:3]
    assert not bad.any(), [(a[i].hex(), b[i].hex(), got[i].hex(), want[i].hex()) for i in k]
