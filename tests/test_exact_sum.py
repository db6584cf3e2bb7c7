"""The warm start's sum of four FP32 values at a time is as exact as FP64 allows (CPU)."""
import os
import shutil
import subprocess
from fractions import Fraction

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2406_13651_gb300", "csrc")

PROGRAM = r"""
#include "exact_sum.cuh"
#include <cstdio>
int main() {
  float v[4];
  while (std::fread(v, sizeof v, 1, stdin) == 1) {
    double acc = 0.0;
    clamp::add_four(acc, v[0], v[1], v[2], v[3]);
    std::fwrite(&acc, sizeof acc, 1, stdout);
  }
  return 0;
}
"""


def _sums(tmp_path, fours):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no g++")
    src, exe = tmp_path / "sum.cpp", str(tmp_path / "sum")
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-O2", "-ffp-contract=off", "-I" + CSRC, "-o", exe, str(src)], check=True)
    out = subprocess.run([exe], input=fours.astype(np.float32).tobytes(), capture_output=True, check=True, timeout=60)
    return np.frombuffer(out.stdout, np.float64)


def test_within_fp64_rounding(tmp_path):
    """Three FP64 additions of 2^-53 each, whatever the values' exponents (a tail rounded in FP32 is off by up to
    2^-48 of the sum)."""
    rng = np.random.default_rng(4)
    fours = rng.uniform(1.0, 2.0, (20000, 4)) * 2.0 ** -rng.integers(0, 40, (20000, 4))
    fours[10000:] *= rng.choice([-1.0, 1.0], (10000, 4))
    fours = fours.astype(np.float32)
    worst = 0.0
    for v, s in zip(fours, _sums(tmp_path, fours)):
        exact = sum(Fraction(float(x)) for x in v)
        scale = max(abs(Fraction(float(x))) for x in v)
        worst = max(worst, float(abs(Fraction(float(s)) - exact) / scale))
    assert worst <= 3 * 4 * 2.0 ** -53, worst   # the sum is at most four times the largest value


def test_not_finite_and_beyond_fp32(tmp_path):
    big = 2.0 ** 127
    got = _sums(tmp_path, np.array([[big, big, 1, 0], [np.inf, 1, 1, 1], [np.nan, 1, 1, 1], [np.inf, -np.inf, 0, 0]]))
    assert got[0] == 2 * big + 1 and got[1] == np.inf and np.isnan(got[2]) and np.isnan(got[3])
