"""The FP32 sums of the one-launch solvers (csrc/sums.cuh), compiled for the host,
against exact rational arithmetic.  The solvers of one launch per step sum exact
products in FP64: at best half an ulp of FP64 of the largest partial sum, which
is at most the sum of the magnitudes, for every addition.  The three-float sum
must be within four of those (2^-51 of the sum of the magnitudes, with the
conversion of its three parts to FP64) however many terms there are; two floats
are not, and serve for the projector coefficients, whose terms are FP32."""
import os
import shutil
import subprocess
from fractions import Fraction

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

MAIN = r"""
#include <cmath>
#include <cstdio>
#include <vector>
#define __device__
#define __forceinline__ inline
struct float2 { float x, y; };
inline float2 make_float2(float x, float y) { return {x, y}; }
inline float __fadd_rn(float a, float b) { return a + b; }
inline float __fsub_rn(float a, float b) { return a - b; }
inline float __fmul_rn(float a, float b) { return a * b; }
template <class T> T __shfl_xor_sync(unsigned, T a, int) { return a; }
template <class T> T __shfl_sync(unsigned, T a, int) { return a; }
using std::fmaf;
#include "sums.cuh"
using namespace gw;
int main(int argc, char** argv) {
  FILE* f = std::fopen(argv[1], "rb");
  int n;
  if (!f || std::fread(&n, 4, 1, f) != 1) return 1;
  std::vector<float> a(n), b(n);
  if (std::fread(a.data(), 4, n, f) != (size_t)n || std::fread(b.data(), 4, n, f) != (size_t)n) return 1;
  F3 dot{0, 0, 0}, lanes[32] = {};
  float2 sum[32] = {};
  for (int i = 0; i < n; ++i) {
    acc_fma(dot, a[i], b[i]);
    acc_in(sum[i % 32], a[i]);
    acc_fma(lanes[i % 32], a[i], b[i]);
  }
  for (int o = 16; o > 0; o >>= 1)
    for (int l = 0; l < o; ++l) {
      lanes[l] = acc_add(lanes[l], lanes[l + o]);
      sum[l] = acc_add(sum[l], sum[l + o]);
    }
  std::printf("%a %a %a %a\n", acc_dbl(dot), acc_dbl(lanes[0]), (double)sum[0].x + (double)sum[0].y,
              (double)acc_val(sum[0]));
}
"""


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("sums")
    (d / "m.cpp").write_text(MAIN)
    subprocess.run([cxx, "-std=c++17", "-O2", "-ffp-contract=off", "-I" + os.path.join(ROOT, "paper_1408_3036_gb300", "csrc"),
                    str(d / "m.cpp"), "-o", str(d / "m")], check=True)
    return d


@pytest.mark.parametrize("n", [1, 7, 333, 20000])
@pytest.mark.parametrize("kind", ["positive", "mixed", "cancelling"])
def test_three_floats_are_as_exact_as_fp64(exe, n, kind):
    rng = np.random.default_rng(n)
    a = (rng.standard_normal(n) * 10.0 ** rng.uniform(-4, 0, n)).astype(np.float32)
    b = rng.standard_normal(n).astype(np.float32)
    if kind == "positive":
        a, b = np.abs(a), np.abs(b)
    elif kind == "cancelling":                  # every term but the first few has its negative
        h = n // 2
        a[n - h:], b[n - h:] = -a[:h], b[:h]
    (exe / "in").write_bytes(np.int32(n).tobytes() + a.tobytes() + b.tobytes())
    out = subprocess.run([str(exe / "m"), str(exe / "in")], check=True, capture_output=True, text=True).stdout.split()
    dot, tree, tot, val = (Fraction(float.fromhex(x)) for x in out)
    fa, fb = [Fraction(float(x)) for x in a], [Fraction(float(x)) for x in b]
    ref, mag = sum(x * y for x, y in zip(fa, fb)), sum(abs(x * y) for x, y in zip(fa, fb))
    assert abs(dot - ref) <= mag / 2 ** 51 and abs(tree - ref) <= mag / 2 ** 51
    # projector coefficients: two floats over a lane's FP32 partial sums, then over the lanes.  The errors of
    # n / 32 additions are summed in FP32 themselves, the rest is renormalised to 2^-47
    ref, mag, eps = sum(fa), sum(map(abs, fa)), Fraction(n // 32 + 8, 2 ** 48)
    assert abs(tot - ref) <= mag * eps
    assert abs(val - ref) <= abs(ref) / 2 ** 24 + mag * eps          # one rounding to FP32
