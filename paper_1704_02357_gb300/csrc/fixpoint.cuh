// Complex numbers in 62-bit fixed point, for the transforms of FP64 contexts: conversions from and
// to FP64, the product with a unit factor, and the scale of a sequence. Integer instructions only;
// the functions compile for the device and for the host (a CPU test checks them).
//
// Why: GB300 runs 2 FP64 operations per clock and SM (measured: 2.0 multiply-adds, 1.7 adds) but 64
// 64-bit integer additions and 24 widening 32 x 32 + 64 bit multiply-adds. A 512-point column of
// an FP64 radix tree costs 28 FP64 operations per point, 15 clocks; in fixed point the additions
// are exact 64-bit integer additions and a complex product is 12 widening multiply-adds.
//
// Scale: a sequence of L values is held in units of 2^-S with S the largest integer for which the
// sum of |re| + |im| over the sequence stays below 2^62 units. Every intermediate value of a DFT has
// at most that modulus, so no sum or rotated component (sqrt 2 times the modulus at most) leaves
// 64 bits, and the partial products below stay below 2^63. For noise-like data of standard
// deviation s per component the unit is ~2^-52 s, and a 512-point transform ends with an error of
// 0.4 unit per sqrt(512) s: 1.0e-16 rms of the result (measured on the host against 128-bit
// transforms), half that of the FP64 radix tree, which rounds at every addition (2.1e-16).
#pragma once
#include "intconv.cuh"

namespace pspec {

struct alignas(16) lc {
  long long x, y;
};

// round(v 2^S) for |v| 2^S < 2^62; c1 = 1084 - S. Zero and values below half a unit give 0.
PSPEC_HD long long fx_from_double(double v, int c1) {
  const unsigned long long b = ic_bits(v);
  const int e = (int)((b >> 52) & 0x7ff);
  const unsigned long long m = ((b & 0xfffffffffffffull) | 0x10000000000000ull) << 10;  // v = m 2^(e - 1085)
  int sh = c1 - e;  // >= 0
  sh = sh > 63 ? 63 : sh;
  const long long q = (long long)(((m >> sh) + 1ull) >> 1);
  return (long long)b < 0 ? -q : q;
}

// q 2^-S rounded to FP64 (ties away from zero); c2 = 1085 - S. |q| < 2^63. The scale keeps every
// result a normal number (fx_scale).
PSPEC_HD double fx_to_double(long long q, int c2) {
  const unsigned long long a = q < 0 ? 0ull - (unsigned long long)q : (unsigned long long)q;
  const int n = ic_clz64(a | 1ull);
  const unsigned long long u = a << n;  // bit 63 set unless q = 0
  const unsigned long long r = (u >> 11) + ((u >> 10) & 1ull);  // 53 bits, the leading one adds 1 to the exponent
  const unsigned long long b = a ? ((unsigned long long)(unsigned)(c2 - n) << 52) + r : 0ull;
  return ic_double(b | ((unsigned long long)q & 0x8000000000000000ull));
}

// A unit factor or constant K, |K| <= 1, as {K_h, K_l}: K = K_h 2^-30 + K_l 2^-62.
// a K with a < 2^62 in modulus: a = a_h 2^32 + a_l (a_l signed), the term a_l K_l (below one unit) left out.
struct FxSplit {
  int h, l;
};
PSPEC_HD FxSplit fx_split(long long a) {
  FxSplit s;
  s.l = (int)(unsigned)(unsigned long long)a;
  s.h = (int)(a >> 32) + (int)((unsigned)s.l >> 31);
  return s;
}
PSPEC_HD long long fx_shift2(long long m) { return (long long)((unsigned long long)m << 2); }
PSPEC_HD long long fx_mul_const(long long a, int kh, int kl) {
  const FxSplit s = fx_split(a);
  const long long m = (long long)s.h * kh;
  const long long c = (long long)s.l * kh + ((long long)s.h * kl + (1ll << 29));
  return fx_shift2(m) + (c >> 30);
}
// a (c + i s)
PSPEC_HD lc fx_mul(lc a, int ch, int cl, int sh, int sl) {
  const FxSplit x = fx_split(a.x), y = fx_split(a.y);
  const long long rm = (long long)x.h * ch + (long long)y.h * -sh;
  const long long im = (long long)x.h * sh + (long long)y.h * ch;
  const long long rc = (long long)x.l * ch + ((long long)x.h * cl + ((long long)y.l * -sh + ((long long)y.h * -sl + (1ll << 29))));
  const long long ic = (long long)x.l * sh + ((long long)x.h * sl + ((long long)y.l * ch + ((long long)y.h * cl + (1ll << 29))));
  lc r;
  r.x = fx_shift2(rm) + (rc >> 30);
  r.y = fx_shift2(im) + (ic >> 30);
  return r;
}
// t / 2, ties to even (no bias that later stages would add up)
PSPEC_HD long long fx_half(long long t) { return (t + ((t >> 1) & 1)) >> 1; }

// ------------------------------------------------------------------ scale of a sequence
// Partial of one thread over its values: the largest upper word of |re|, |im|, and the sum of
// |re| + |im| as floats (the 20 upper mantissa bits; meaningful for values between 2^-126 and 2^128).
struct FxBound {
  unsigned mx;
  float sum;
};
PSPEC_HD unsigned fx_hi(double v) { return (unsigned)(ic_bits(v) >> 32) & 0x7fffffffu; }
PSPEC_HD void fx_bound_add(FxBound& b, double v) {
  const unsigned h = fx_hi(v);
  b.mx = h > b.mx ? h : b.mx;
  const int d = (int)h - (896 << 20);  // exponent bias 1023 -> 127
  b.sum += ic_float((unsigned)(d > 0 ? d : 0) << 3);
}
// S of the sequence whose partials add up to b; `len` values (complex), times 2^extra of headroom for what is
// done to them before and after the transform. Sets bad when a value is infinite, NaN or too large for
// the results to stay finite: the results are then NaN. Sequences whose values are all below 2^-895 count as 0.
struct FxScale {
  int S;
  bool bad;
};
PSPEC_HD FxScale fx_scale(FxBound b, int log2_len, int extra) {
  FxScale s;
  const int e = (int)(b.mx >> 20);  // largest exponent, |v| < 2^(e - 1022)
  s.bad = e > 2046 - 20;
  if (e > 1023 - 100 && e < 1023 + 100) {
    // the truncated mantissas and the float sum are low by less than 2^-10
    const float f = b.sum * 1.001953125f;
    s.S = 62 - (int)((ic_bits(f) >> 23) - 126u) - extra;  // f < 2^(exponent - 126)
  } else if (e < 128) {
    s.S = -4096;  // every value rounds to 0
  } else {
    s.S = 62 - (e - 1022) - 1 - log2_len - extra;
  }
  return s;
}

}  // namespace pspec
