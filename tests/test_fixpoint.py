"""The fixed-point arithmetic of the FP64 transforms (csrc/fixpoint.cuh) and the integer forms the
paint uses (csrc/intconv.cuh), compiled for the host.

Conversions are compared with exact integer arithmetic; products by a unit factor with exact integers
(per real factor the term below one unit that they leave out, and one rounding: at most 1.5 units, 2.5
for a complex product); the scale with the bound it has to keep."""
import math
import os
import random
import shutil
import subprocess
from fractions import Fraction

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1704_02357_gb300", "csrc")

SRC = r"""
#include <cstdio>
#include <vector>
#include "fixpoint.cuh"
using namespace pspec;
int main() {
  char op; 
  while (std::scanf(" %c", &op) == 1) {
    if (op == 'i') { double v; int c; std::scanf("%la %d", &v, &c); std::printf("%lld\n", fx_from_double(v, c)); }
    if (op == 'o') { long long q; int c; std::scanf("%lld %d", &q, &c); std::printf("%a\n", fx_to_double(q, c)); }
    if (op == 'f') { double v; std::scanf("%la", &v); FloatPair p = float_pair(v); std::printf("%a %a %u %d\n", p.lo, p.hi, p.thr, (int)float_pair_ok(v)); }
    if (op == 'd') { double v; int k; std::scanf("%la %d", &v, &k); std::printf("%lld\n", d2ll_rn_scaled(v, k)); }
    if (op == 'h') { long long q; std::scanf("%lld", &q); std::printf("%lld\n", fx_half(q)); }
    if (op == 'm') {
      lc a; int c, d, e, f; std::scanf("%lld %lld %d %d %d %d", &a.x, &a.y, &c, &d, &e, &f);
      lc r = fx_mul(a, c, d, e, f); std::printf("%lld %lld %lld\n", r.x, r.y, fx_mul_const(a.x, c, d));
    }
    if (op == 's') {
      int n, extra, lg; std::scanf("%d %d %d", &n, &lg, &extra); FxBound b{0u, 0.f};
      for (int i = 0; i < n; i++) { double v; std::scanf("%la", &v); fx_bound_add(b, v); }
      FxScale s = fx_scale(b, lg, extra); std::printf("%d %d\n", s.S, (int)s.bad);
    }
  }
}
"""


@pytest.fixture(scope="module")
def ask(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("fx")
    (d / "t.cpp").write_text(SRC)
    exe = str(d / "t")
    subprocess.run([cxx, "-O2", "-std=c++17", "-x", "c++", "-I", CSRC, str(d / "t.cpp"), "-o", exe], check=True)

    def run(lines):
        out = subprocess.run([exe], input="\n".join(lines), capture_output=True, text=True, check=True).stdout
        return [ln.split() for ln in out.splitlines()]
    return run


def test_conversions_round_to_nearest(ask):
    rng = random.Random(1)
    ins = [(0.0, 1084), (-0.0, 900), (5e-324, 1084), (math.ldexp(1, 61), 1084), (-math.ldexp(1, 61), 1084)]
    for _ in range(20000):
        S = rng.randint(-900, 900)
        ins.append((math.ldexp(rng.uniform(-1, 1), 62 - S - rng.randint(0, 80)), 1084 - S))
    for (v, c), r in zip(ins, ask([f"i {v.hex()} {c}" for v, c in ins])):
        x = Fraction(v) * Fraction(2) ** (1084 - c)
        assert abs(Fraction(int(r[0])) - x) <= Fraction(1, 2), (v, c, r)
    outs = [(0, 1085), (1, 1085), (-1, 1085), (2 ** 62, 1085), (-2 ** 63 + 1, 1085), (2 ** 63 - 1, 1085), (2 ** 53 + 1, 1085)]
    for _ in range(20000):
        q = rng.getrandbits(rng.randint(1, 63)) * rng.choice([1, -1])
        outs.append((q, 1085 - rng.randint(-900, 900)))
    for (q, c), r in zip(outs, ask([f"o {q} {c}" for q, c in outs])):
        got, want = float.fromhex(r[0]), Fraction(q) * Fraction(2) ** (c - 1085)
        ulp = Fraction(math.ulp(got)) if got else Fraction(0)
        assert abs(Fraction(got) - want) <= ulp / 2, (q, c, r)
    halves = list(range(-9, 10)) + [2 ** 62 + 1, -2 ** 62 - 1]
    for q, r in zip(halves, ask([f"h {q}" for q in halves])):
        assert int(r[0]) == round(Fraction(q, 2)), q  # ties to even


def test_products_by_unit_factors(ask):
    rng = random.Random(2)
    cases = []
    for i in range(20000):
        th = rng.choice([0.0, math.pi / 2, math.pi, rng.uniform(0, 7)])
        mod, ph = 2.0 ** 62 * rng.choice([1.0, rng.random(), 2.0 ** -rng.randint(1, 60)]), rng.uniform(0, 7)
        a = (int(mod * math.cos(ph) * (1 - 1e-9)), int(mod * math.sin(ph) * (1 - 1e-9)))
        w = []
        for comp in (math.cos(th), math.sin(th)):
            q = int(Fraction(comp) * 2 ** 62)
            h = (q + 2 ** 31) >> 32
            w += [h, max(q - (h << 32), -2 ** 31 + 1)]
        cases.append((a, w))
    got = ask([f"m {a[0]} {a[1]} {w[0]} {w[1]} {w[2]} {w[3]}" for a, w in cases])
    for (a, w), r in zip(cases, got):
        c, s = Fraction(w[0] * 2 ** 32 + w[1], 2 ** 62), Fraction(w[2] * 2 ** 32 + w[3], 2 ** 62)
        assert abs(int(r[0]) - (a[0] * c - a[1] * s)) <= Fraction(5, 2), (a, w, r)
        assert abs(int(r[1]) - (a[0] * s + a[1] * c)) <= Fraction(5, 2), (a, w, r)
        assert abs(int(r[2]) - a[0] * c) <= Fraction(3, 2), (a, w, r)


@pytest.mark.parametrize("exponent", [-1000, -200, -99, -40, 0, 40, 99, 200, 990])
def test_scale_keeps_the_sum_below_2_62(ask, exponent):
    rng = random.Random(exponent)
    for extra in (0, 1, 2):
        vals = [math.ldexp(rng.uniform(-1, 1) * 2.0 ** -rng.randint(0, 20), exponent) for _ in range(128)]
        S, bad = (int(x) for x in ask([f"s 128 6 {extra} " + " ".join(v.hex() for v in vals)])[0])
        total = sum(abs(Fraction(v)) for v in vals) * Fraction(2) ** (S + extra)
        if exponent == -1000:
            assert S < -2000 and not bad  # counts as zero
            continue
        assert not bad and total <= 2 ** 62
        if abs(exponent) < 90:
            assert total > 2 ** 62 / Fraction(9, 4)  # the largest scale, up to the sum's own slack
    for v in ("inf", "nan"):
        assert ask([f"s 2 1 0 {v} 0x1p+0"])[0][1] == "1"


def test_scaled_rounding_and_float_pairs(ask):
    rng = random.Random(4)
    vals = [(0.0, 24), (-0.0, 24), (5e-324, 24), (0.5 * 2.0 ** -24, 24), (1.5 * 2.0 ** -24, 24), (2.0 ** 37, 24)]
    vals += [(math.ldexp(rng.uniform(-1, 1), rng.randint(-40, 38)), 24) for _ in range(20000)]
    for (v, k), r in zip(vals, ask([f"d {v.hex()} {k}" for v, k in vals])):
        assert int(r[0]) == round(Fraction(v) * 2 ** k), (v, r)  # ties to even
    import struct
    f32 = lambda x: struct.unpack("f", struct.pack("f", x))[0]
    nxt = lambda x, up: struct.unpack("f", struct.pack("I", struct.unpack("I", struct.pack("f", x))[0] + (1 if up else -1)))[0]
    vs = [0.25, -0.25, 1.0 - 2.0 ** -30, -(1.0 - 2.0 ** -30), 1.0 + 2.0 ** -25, 1.0 + 2.0 ** -24, 1.0 + 3 * 2.0 ** -24,
          1.0 - 2.0 ** -25, -0.05]
    vs += [rng.uniform(-1, 1) * 2.0 ** rng.randint(-100, 100) for _ in range(20000)]
    for v, r in zip(vs, ask([f"f {v.hex()}" for v in vs])):
        lo, hi, thr, ok = float.fromhex(r[0]), float.fromhex(r[1]), int(r[2]), r[3] == "1"
        assert ok and lo == f32(v), (v, r)
        if lo == v:
            assert hi == lo and thr == 0
            continue
        assert hi == nxt(lo, abs(v) > abs(lo)) and min(lo, hi) < v < max(lo, hi), (v, r)
        assert thr == Fraction(abs(v - lo)) / Fraction(abs(hi - lo)) * 2 ** 32, (v, r)
    for v in (0.0, 1e-39, 3e38, float("inf"), float("nan")):
        assert ask([f"f {v.hex()}"])[0][3] == "0", v
