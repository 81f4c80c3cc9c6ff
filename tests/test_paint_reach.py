"""paint_safe_log2 (csrc/intconv.cuh), compiled for the host: positions below 2^k in magnitude lie within 2^37 cells
of the corner on every axis, k is the largest such exponent, and a corner that is too far away or not a number
gives no exponent at all. Decided against exact fractions; the call itself, made for every painted catalog, takes no search."""
import math
import os
import random
import shutil
import subprocess
from fractions import Fraction

import pytest

CSRC = os.path.join(os.path.dirname(__file__), "..", "paper_1704_02357_gb300", "csrc")

PROGRAM = r"""
#include <chrono>
#include <cstdio>
#include "intconv.cuh"
int main() {
  double c[3], inv;
  while (std::scanf("%la %la %la %la", &c[0], &c[1], &c[2], &inv) == 4) std::printf("%d\n", pspec::paint_safe_log2(c, inv));
  long long s = 0;
  const auto t0 = std::chrono::steady_clock::now();
  for (int i = 0; i < 100000; i++) {
    c[0] = i;
    c[1] = c[2] = -i;
    s += pspec::paint_safe_log2(c, 0.256);
  }
  std::printf("%lld %f\n", s, std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count() / 100000 * 1e6);
}
"""


def test_safe_exponent(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no C++ compiler")
    (tmp_path / "t.cpp").write_text(PROGRAM)
    exe = str(tmp_path / "t")
    subprocess.run([cxx, "-O2", "-std=c++17", "-I", CSRC, str(tmp_path / "t.cpp"), "-o", exe], check=True)
    rng = random.Random(4)
    cases = []
    for _ in range(4000):
        inv = rng.uniform(0.5, 1) * 2.0 ** rng.choice([-3, 0, 8, rng.randint(-300, 300), rng.randint(-900, 900)])
        far = 2.0 ** 37 / inv
        f = rng.choice([0.0, 1e-9, 0.3, 1 - 2 ** -50, 1.0, 1 + 2 ** -50, 3.0])
        cases.append(([rng.uniform(-1, 1) * f * far, -f * far, 0.0], inv))
    # away from the origin by more than 2^37 cells, by next to nothing less, and what is no number
    bad = [([math.nan, 0.0, 0.0], 1.0), ([0.0, math.nan, 1.0], 1.0), ([0.0, 0.0, math.inf], 1.0), ([0.0, -math.inf, 0.0], 1.0),
           ([0.0, 0.0, 0.0], math.nan), ([2.0 ** 37, 0.0, 0.0], 1.0), ([1.0, 2.0, 3.0], math.inf)]
    lines = ["%s %s" % (" ".join(float(v).hex() for v in c), float(inv).hex()) for c, inv in cases + bad]
    out = subprocess.run([exe], input="\n".join(lines), capture_output=True, text=True, check=True).stdout.split()
    got = [int(v) for v in out[:len(lines)]]
    assert got[len(cases):] == [-5000] * len(bad)
    eps = Fraction(1, 2 ** 50)  # reach is a quotient and a difference in FP64
    for (c, inv), k in zip(cases, got):
        # distances in units of 2^37 cells
        inv, c = Fraction(inv) / 2 ** 37, max(abs(Fraction(v)) for v in c)
        if k == -5000:
            assert (c + Fraction(2) ** -900) * inv > 1 - eps
            continue
        assert -900 <= k <= 900
        assert (c + Fraction(2) ** k) * inv < 1 + eps
        if k < 900:
            assert (c + Fraction(2) ** (k + 1)) * inv > 1 - eps
    assert float(out[-1]) < 1.0  # microseconds a call
