"""The level sums of the FP64 2D wave solve (csrc/fixed64.cuh) on values that no bound covers: points
beyond a tile's valid ring.  Compiled with the undefined-behaviour sanitizer, they must wrap around
(CPU only)."""

import os
import shutil
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2507_23613_gb300", "csrc")
sys.path.insert(0, os.path.dirname(os.path.abspath(__file__)))
from test_fpair_host import _cuda_include  # noqa: E402

MAIN = r"""
#include <cstdint>
#include <cstdio>
#include <cuda_runtime.h>
#include "fixed64.cuh"
using namespace mfwh;
int main() {
  const int64_t v[] = {0, 1, -1, 2147483647, -2147483648ll, INT64_MAX, INT64_MIN, INT64_MAX - 5,
                       INT64_MIN + 7, 1ll << 62, -(1ll << 62), 0x123456789abcdefll};
  const FxCoef A{0xFFFFFFFEu, 0xFFFFFFFFu, 0x7FFFFFFFFFFFFFFFull};
  int64_t sum = 0;
  for (int64_t a : v)
    for (int64_t b : v) {
      if (fx_sub(fx_add(a, b), b) != a || fx_add(fx_sub(a, b), b) != a) return 1;
      if (fx_add(fx_mul15(a), a) != (int64_t)((uint64_t)a << 4)) return 2;
      sum = fx_add(sum, fx_mac(a, b, A));
      for (int k = -70; k <= 2; ++k) sum = fx_add(sum, fx_rescale(a, k));
      int hi, lo;
      fx_digits(a, hi, lo);
      sum = fx_add(sum, (int64_t)hi + lo + fx_level_digits(a).x);
    }
  std::printf("%lld\n", (long long)sum);
  return 0;
}
"""


def test_sums_beyond_the_bounds_wrap_around(tmp_path):
    inc = _cuda_include()
    if shutil.which("g++") is None or inc is None:
        pytest.skip("no host C++ compiler or CUDA headers")
    src, exe = tmp_path / "wrap.cpp", tmp_path / "wrap"
    src.write_text(MAIN)
    r = subprocess.run(["g++", "-std=c++17", "-O1", "-fsanitize=undefined",
                        "-fno-sanitize-recover=all", "-I", inc, "-I", CSRC, str(src), "-o",
                        str(exe)], capture_output=True, text=True)
    if r.returncode != 0 and "ubsan" in r.stderr:
        pytest.skip("no undefined-behaviour sanitizer")
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr


def test_the_step_uses_them():
    """No plain sum or difference of levels in the step kernel's stencil."""
    with open(os.path.join(CSRC, "wave_fx_kernels.cuh")) as fh:
        text = fh.read()
    step = text[text.index("auto step_points = "):text.index("const bool plain = __all_sync")]
    for name in ("w[k][c] +", "w[k][c] -", "+ dnew", "- fs[", "15 * d", "- up.", "- left", "right -",
                 "dxx + dyy", "- dv["):
        assert name not in step, name
