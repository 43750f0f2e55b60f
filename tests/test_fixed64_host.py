"""The 64-bit fixed-point arithmetic of the FP64 2D wave solve (csrc/fixed64.cuh), compiled for the
host and checked against exact integer and rational arithmetic (CPU only)."""

import ctypes as C
import os
import shutil
import subprocess
import sys
from fractions import Fraction

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2507_23613_gb300", "csrc")
sys.path.insert(0, os.path.dirname(os.path.abspath(__file__)))
from test_fpair_host import _cuda_include  # noqa: E402

SHIM = r"""
#include <cstring>
#include <cstdint>
#include <cuda_runtime.h>
#include "fixed64.cuh"
using namespace mfwh;
extern "C" {
int64_t mac(int64_t d, int64_t x, uint64_t a) {
  return fx_mac(d, x, FxCoef{(uint32_t)a, (uint32_t)(a >> 32), a >> 1});
}
void products(const int64_t* w, const int64_t* x, int n, int64_t* s) {
  FxSum S{0, 0};
  for (int i = 0; i < n; ++i) {
    int hi, lo;
    fx_digits(w[i], hi, lo);
    const int2 v = fx_level_digits(x[i]);
    fx_madd(S, hi, v);
    S.s2 += (int64_t)lo * v.x;   // (in FP32 in the kernel)
  }
  s[0] = S.s1; s[1] = S.s2;
}
int64_t from_double(double v, int e) {
  uint64_t b;
  std::memcpy(&b, &v, 8);
  return fx_from_bits(b, e);
}
int64_t rescale(int64_t x, int k) { return fx_rescale(x, k); }
}
"""


@pytest.fixture(scope="module")
def fx(tmp_path_factory):
    inc = _cuda_include()
    if shutil.which("g++") is None or inc is None:
        pytest.skip("no host C++ compiler or CUDA headers")
    d = tmp_path_factory.mktemp("fixed64")
    src, so = d / "fixed64_host.cpp", d / "libfixed64_host.so"
    src.write_text(SHIM)
    subprocess.run(["g++", "-std=c++17", "-O2", "-shared", "-fPIC", "-I", inc, "-I", CSRC,
                    str(src), "-o", str(so)], check=True, capture_output=True)
    lib = C.CDLL(str(so))
    lib.mac.argtypes, lib.mac.restype = [C.c_int64, C.c_int64, C.c_uint64], C.c_int64
    lib.from_double.argtypes, lib.from_double.restype = [C.c_double, C.c_int], C.c_int64
    lib.rescale.argtypes, lib.rescale.restype = [C.c_int64, C.c_int], C.c_int64
    return lib


def draw(rng, bits):
    """A signed integer of at most `bits` bits, with runs of zeros and ones among them."""
    v = int(rng.integers(0, 2**62)) >> (62 - int(rng.integers(1, bits + 1)))
    if rng.random() < 0.2:
        v = (1 << int(rng.integers(0, bits))) - int(rng.integers(0, 2))
    return -v if rng.random() < 0.5 else v


def nearest(f):
    return (f + Fraction(1, 2)).__floor__()   # halves up


def test_multiply_add_rounds_to_the_nearest_quantum(fx):
    rng = np.random.default_rng(1)
    edges = [0, 1, -1, 2**31, -2**31, 2**32, -2**32, 2**62 - 1, -2**62, 2**63 - 1, -2**63]
    for i in range(40000):
        x = edges[i % 11] if i < 2000 else draw(rng, 62)
        a = int(rng.integers(0, 2**63, dtype=np.uint64)) * 2
        if i % 3 == 0:
            a = int(rng.uniform(2.0**-10, 1.0) * 2.0**53) << 11   # a double's 53 bits
        d = draw(rng, 60)
        assert fx.mac(d, x, a) == d + nearest(Fraction(a * x, 2**64)), (d, x, a)


def test_digit_sums_are_the_products_but_for_the_lowest(fx):
    """With weights up to 2^60 and levels up to 2^59, eight terms: the sums hold every product but
    low digit times low digit (each at most 2^62), of the level less 2^31."""
    rng = np.random.default_rng(2)
    s = (C.c_int64 * 2)()
    for i in range(4000):
        big = i % 5 == 0
        w = [(2**60 - 128 if rng.random() < .5 else 128 - 2**60) if big else draw(rng, 60) for _ in range(8)]
        x = [(2**59 - 1 if rng.random() < .5 else -2**59) if big else draw(rng, 59)
             for _ in range(8)]
        fx.products((C.c_int64 * 8)(*w), (C.c_int64 * 8)(*x), 8, s)
        got = s[0] * 2**64 + s[1] * 2**32
        want = sum(a * (b - 2**31) for a, b in zip(w, x))
        assert abs(got - want) <= 8 * 2**62


def test_conversion_and_rescaling_round_to_nearest(fx):
    rng = np.random.default_rng(3)
    for _ in range(20000):
        e = int(rng.integers(-900, 900))
        v = float(np.ldexp(rng.uniform(-1.0, 1.0), e + int(rng.integers(-70, 62))))
        assert abs(Fraction(v) / Fraction(2) ** e - fx.from_double(v, e)) <= Fraction(1, 2)
        x, k = draw(rng, 59), int(rng.integers(-70, 3))
        assert abs(Fraction(x) * Fraction(2) ** k - fx.rescale(x, k)) <= Fraction(1, 2)
    for v in (0.0, -0.0, 5e-324):
        assert fx.from_double(v, 0) == 0
