// Exact-add FP32 transform stages.
//
// The rounding error of an FP32 radix tree sits in its additions: every add level rounds its
// result (about 0.42 u rms of the output, u = 2^-24), nine levels per 512-point pass. In the
// harmonic transforms of the estimator (Sec. 2.1 eq. Fell) that noise is what limits how
// closely a multipole of a few percent of P_0 can be recovered against a shot noise of ~80 P_0.
//
// Here a stage keeps every value as a pair h + l of floats:
//   * h is a multiple of a power-of-two quantum q chosen per thread and stage from the thread's
//     inputs, so that every value of the stage's butterflies stays below 2^11 q: h has at most
//     12 significant bits above q. Sums and differences of such multiples are exact in FP32.
//   * Constants and twiddles are split the same way, K = K12 + Kr with K12 a multiple of 2^-12
//     (|K| <= 1) and Kr the remainder (held to 24 bits of its own). h * K12 then has at most 23
//     significant bits and is exact in FP32, and so are sums of such products; h * Kr and
//     l * K go to l, rounded at ~2^-24 q.
//   * A product lies on the finer quantum q/4096, so before a value is multiplied again it is
//     put back on q (re-split): g = (h + M) - M with M = 1.5 * 2^23 q rounds to q exactly and
//     h - g is exact.
// Values cross the shared-memory exchanges and leave the transform as h + l rounded to one
// float, so a pass rounds each value once per exchange and once at the end, instead of once per
// add level. Every operation whose exactness the scheme relies on uses the _rn intrinsics or an
// FMA whose result is exact, and the compiler never contracts the intrinsics into a multiply-add.
#pragma once
#include "fx_engine.cuh"

namespace pspec {

// Packed FP32 pairs: one instruction adds, multiplies or multiply-adds both halves, each rounded as
// the scalar instruction rounds it. The FMA pipe takes a pair no faster than two scalars (measured: 53
// packed against 117 scalar results per clock and SM), but it takes one issue slot instead of two, and
// these stages were bound by issue (85% of the slots in the z pass with the pipe 67% busy). Values
// are complex numbers, so the pairs are (re, im): additions, splits and products by real constants are
// packed; rotations by i and twiddle products, which mix the halves, stay scalar.
__device__ __forceinline__ float2 add2(float2 a, float2 b) {
  float2 r;
  asm("{.reg .b64 a, b, c; mov.b64 a, {%2, %3}; mov.b64 b, {%4, %5}; add.rn.f32x2 c, a, b; mov.b64 {%0, %1}, c;}"
      : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return r;
}
__device__ __forceinline__ float2 sub2(float2 a, float2 b) {
  float2 r;
  asm("{.reg .b64 a, b, c; mov.b64 a, {%2, %3}; mov.b64 b, {%4, %5}; sub.rn.f32x2 c, a, b; mov.b64 {%0, %1}, c;}"
      : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return r;
}
__device__ __forceinline__ float2 mul2(float2 a, float k) {
  float2 r;
  asm("{.reg .b64 a, b, c; mov.b64 a, {%2, %3}; mov.b64 b, {%4, %4}; mul.rn.f32x2 c, a, b; mov.b64 {%0, %1}, c;}"
      : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(k));
  return r;
}
__device__ __forceinline__ float2 fma2(float2 a, float k, float2 d) {
  float2 r;
  asm("{.reg .b64 a, b, c, d; mov.b64 a, {%2, %3}; mov.b64 b, {%4, %4}; mov.b64 d, {%5, %6}; fma.rn.f32x2 c, a, b, d; "
      "mov.b64 {%0, %1}, c;}"
      : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(k), "f"(d.x), "f"(d.y));
  return r;
}

// A complex value h + l; h = (re, im) on the quantum q.
struct xc {
  float2 h, l;
};

__device__ __forceinline__ float xadd_(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float xsub_(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float xmul_(float a, float b) { return __fmul_rn(a, b); }

// M = 1.5 * 2^23 * q for the smallest power-of-two q with `bound` <= 2^11 q.
__device__ __forceinline__ float xmagic(float bound) {
  int eb = (__float_as_int(bound) >> 23) & 0xff;  // bound < 2^(eb - 126)
  eb = eb > 240 ? 240 : eb;
  return __int_as_float(((eb + 13) << 23) | 0x400000);  // q = 2^(eb - 137), M = 1.5 * 2^(eb - 114)
}
__device__ __forceinline__ float2 xgrid(float2 p, float M) {
  const float2 m = make_float2(M, M);
  return sub2(add2(p, m), m);
}
__device__ __forceinline__ xc xsplit(float2 v, float M) {
  const float2 g = xgrid(v, M);
  return {g, sub2(v, g)};
}
// back onto the quantum q before another multiplication
__device__ __forceinline__ xc xresplit(xc a, float M) {
  const float2 g = xgrid(a.h, M);
  return {g, add2(a.l, sub2(a.h, g))};
}
__device__ __forceinline__ float2 xround(xc a) { return add2(a.h, a.l); }

__device__ __forceinline__ xc operator+(xc a, xc b) { return {add2(a.h, b.h), add2(a.l, b.l)}; }
__device__ __forceinline__ xc operator-(xc a, xc b) { return {sub2(a.h, b.h), sub2(a.l, b.l)}; }
// a + i sgn b
__device__ __forceinline__ float2 xadd_i(float2 a, float2 b, int sgn) {
  return sgn > 0 ? make_float2(xsub_(a.x, b.y), xadd_(a.y, b.x)) : make_float2(xadd_(a.x, b.y), xsub_(a.y, b.x));
}
__device__ __forceinline__ xc xadd_i(xc a, xc b, int sgn) { return {xadd_i(a.h, b.h, sgn), xadd_i(a.l, b.l, sgn)}; }
__device__ __forceinline__ float2 xconj(float2 a) { return make_float2(a.x, -a.y); }
__device__ __forceinline__ xc xconj(xc a) { return {xconj(a.h), xconj(a.l)}; }

// A constant |K| <= 1 as K12 (a multiple of 2^-12) + Kr, with kf = K rounded to FP32.
struct K12 {
  float k12, kr, kf;
  __device__ __forceinline__ constexpr K12(double k)
      : k12((float)((double)(long long)(k * 4096.0 + (k >= 0 ? 0.5 : -0.5)) / 4096.0)),
        kr((float)(k - (double)(long long)(k * 4096.0 + (k >= 0 ? 0.5 : -0.5)) / 4096.0)),
        kf((float)k) {}
};
// a * K; a.h on the quantum q (at most 12 significant bits): a.h * K12 is exact.
__device__ __forceinline__ xc xcm(xc a, const K12& k) { return {mul2(a.h, k.k12), fma2(a.l, k.kf, mul2(a.h, k.kr))}; }

// a * w for a twiddle in the 12-bit form {c12, s12, cr, sr} (tables built on the host); a on the
// quantum q. The h parts are exact: each product has at most 23 significant bits and the FMA's
// exact result is representable.
__device__ __forceinline__ xc xtw(xc a, float4 w) {
  const float cf = xadd_(w.x, w.z), sf = xadd_(w.y, w.w);
  xc r;
  r.h.x = fmaf(a.h.x, w.x, -xmul_(a.h.y, w.y));
  r.h.y = fmaf(a.h.x, w.y, xmul_(a.h.y, w.x));
  r.l.x = fmaf(a.l.x, cf, fmaf(-a.l.y, sf, fmaf(a.h.x, w.z, -xmul_(a.h.y, w.w))));
  r.l.y = fmaf(a.l.x, sf, fmaf(a.l.y, cf, fmaf(a.h.x, w.w, xmul_(a.h.y, w.z))));
  return r;
}
__device__ __forceinline__ xc xtw(float2 a, float4 w, float M) { return xtw(xsplit(a, M), w); }

// ------------------------------------------------------------------ butterflies
// The radix-R DFTs of common.cuh (same decompositions and constants) on exact-add values. The
// inputs may lie on the finer quantum (twiddled): a value is re-split before each internal
// multiplication.
template <int R> struct XDft;

template <> struct XDft<2> {
  static __device__ __forceinline__ void run(xc* v, int, float) {
    const xc a = v[0], b = v[1];
    v[0] = a + b;
    v[1] = a - b;
  }
};

template <> struct XDft<4> {
  static __device__ __forceinline__ void run(xc* v, int dir, float) {
    const xc t0 = v[0] + v[2], t1 = v[0] - v[2];
    const xc t2 = v[1] + v[3], t3 = v[1] - v[3];
    v[0] = t0 + t2;
    v[2] = t0 - t2;
    v[1] = xadd_i(t1, t3, dir);
    v[3] = xadd_i(t1, t3, -dir);
  }
};

// z * (sr cr + i si ci) with sr, si = +-1
__device__ __forceinline__ xc xrot(xc z, const K12& cr, const K12& ci, int sr, int si, float M) {
  z = xresplit(z, M);
  const xc a = xcm(z, cr), b = xcm(z, ci);  // cr z, ci z
  // sr a + i si b
  auto mix = [&](float2 p, float2 q) {
    const float2 u = sr > 0 ? p : make_float2(-p.x, -p.y);
    return si > 0 ? make_float2(xsub_(u.x, q.y), xadd_(u.y, q.x)) : make_float2(xadd_(u.x, q.y), xsub_(u.y, q.x));
  };
  return {mix(a.h, b.h), mix(a.l, b.l)};
}
// z * (sgn + dir i) / sqrt2 (sgn = +-1)
__device__ __forceinline__ xc xdiag(xc z, int sgn, int dir, const K12& h, float M) {
  auto mix = [&](float2 p) {  // sgn p + i dir p
    const float2 u = sgn > 0 ? p : make_float2(-p.x, -p.y);
    return dir > 0 ? make_float2(xsub_(u.x, p.y), xadd_(u.y, p.x)) : make_float2(xadd_(u.x, p.y), xsub_(u.y, p.x));
  };
  const xc r = {mix(z.h), mix(z.l)};
  return xcm(xresplit(r, M), h);
}

template <> struct XDft<8> {
  static __device__ __forceinline__ void run(xc* v, int dir, float M) {
    const K12 h(0.70710678118654752440);
    xc e[4] = {v[0], v[2], v[4], v[6]};
    xc o[4] = {v[1], v[3], v[5], v[7]};
    XDft<4>::run(e, dir, M);
    XDft<4>::run(o, dir, M);
    const xc o1 = xdiag(o[1], 1, dir, h, M);
    const xc o3 = xdiag(o[3], -1, dir, h, M);
    v[0] = e[0] + o[0];
    v[4] = e[0] - o[0];
    v[1] = e[1] + o1;
    v[5] = e[1] - o1;
    v[2] = xadd_i(e[2], o[2], dir);
    v[6] = xadd_i(e[2], o[2], -dir);
    v[3] = e[3] + o3;
    v[7] = e[3] - o3;
  }
};

template <> struct XDft<16> {
  static __device__ __forceinline__ void run(xc* v, int dir, float M) {
    const K12 h(0.70710678118654752440), c1(0.92387953251128675613), s1(0.38268343236508977173);
    xc a[4][4];
#pragma unroll
    for (int n2 = 0; n2 < 4; n2++) {
      xc t[4] = {v[n2], v[n2 + 4], v[n2 + 8], v[n2 + 12]};
      XDft<4>::run(t, dir, M);
#pragma unroll
      for (int k1 = 0; k1 < 4; k1++) a[n2][k1] = t[k1];
    }
    const int d = dir;
    a[1][1] = xrot(a[1][1], c1, s1, 1, d, M);    // m = 1
    a[1][2] = xdiag(a[1][2], 1, d, h, M);        // m = 2
    a[1][3] = xrot(a[1][3], s1, c1, 1, d, M);    // m = 3
    a[2][1] = xdiag(a[2][1], 1, d, h, M);        // m = 2
    a[2][3] = xdiag(a[2][3], -1, d, h, M);       // m = 6
    a[3][1] = xrot(a[3][1], s1, c1, 1, d, M);    // m = 3
    a[3][2] = xdiag(a[3][2], -1, d, h, M);       // m = 6
    a[3][3] = xrot(a[3][3], c1, s1, -1, -d, M);  // m = 9
#pragma unroll
    for (int k1 = 0; k1 < 4; k1++) {
      xc t[4] = {a[0][k1], a[1][k1], a[2][k1], a[3][k1]};
      if (k1 == 2) {  // m = 4: a[2][2] times i d
        const xc t0 = xadd_i(t[0], t[2], d), t1 = xadd_i(t[0], t[2], -d);
        const xc t2 = t[1] + t[3], t3 = t[1] - t[3];
        t[0] = t0 + t2;
        t[2] = t0 - t2;
        t[1] = xadd_i(t1, t3, d);
        t[3] = xadd_i(t1, t3, -d);
      } else {
        XDft<4>::run(t, dir, M);
      }
#pragma unroll
      for (int k2 = 0; k2 < 4; k2++) v[k1 + 4 * k2] = t[k2];
    }
  }
};

template <> struct XDft<3> {
  static __device__ __forceinline__ void run(xc* v, int dir, float M) {
    const K12 s3(0.86602540378443864676);
    const xc t = v[1] + v[2];
    const xc u = xresplit(v[1] - v[2], M);
    const xc m = v[0] - xc{mul2(t.h, 0.5f), mul2(t.l, 0.5f)};
    const xc su = xcm(u, s3);  // sin(2 pi/3) u
    v[0] = v[0] + t;
    v[1] = xadd_i(m, su, dir);
    v[2] = xadd_i(m, su, -dir);
  }
};

// ------------------------------------------------------------------ stages
// One Stockham stage as stage_ct (fft_engine.cuh) on float2 values held per thread, computed in
// exact-add arithmetic. The quantum is chosen from the thread's E inputs: every intermediate of
// a butterfly is a sum of its inputs times factors of modulus <= 1, so each component stays below
// sqrt(2) times the sum of the inputs' |re| + |im|; the bound passed is twice that sum.
template <int E, int L, int R, int NS, int OFF, bool LAST, int LAYOUT, int NSEQ, int DIR>
__device__ __forceinline__ void stage_xp(float2 (&v)[E], float2* sm, int t, int seq, const float4* __restrict__ tw) {
  constexpr int Q = E / R;
  constexpr int Tc = L / E;
  tw += OFF - NS;  // entry r of k at r NS + k
  constexpr bool kShared = (Q > 1) && (NS > 1) && !LAST && (NS <= Tc);
  float4 ws[kShared ? R : 1];
  if constexpr (kShared) {
    const int k = t & (NS - 1);
#pragma unroll
    for (int r = 1; r < R; r++) {
      ws[r] = ldg_u(tw + r * NS + k);
      if (DIR > 0) ws[r] = uconj(ws[r]);
    }
  }
  float bound = 0.f;
#pragma unroll
  for (int e = 0; e < E; e++) bound += fabsf(v[e].x) + fabsf(v[e].y);
  const float M = xmagic(2.f * bound);  // twice: a rotated component reaches sqrt2 |x|
#pragma unroll
  for (int q = 0; q < Q; q++) {
    const int j = t + Tc * q;
    const int k = LAST ? j : (j & (NS - 1));
    xc u[R];
#pragma unroll
    for (int r = 0; r < R; r++) {
      if (NS > 1 && r > 0) {
        float4 w;
        if constexpr (kShared) {
          w = ws[r];
        } else {
          w = ldg_u(tw + r * NS + k);
          if (DIR > 0) w = uconj(w);
        }
        u[r] = xtw(v[q + r * Q], w, M);  // the 12-bit twiddle table
      } else {
        u[r] = xsplit(v[q + r * Q], M);
      }
    }
    XDft<R>::run(u, DIR, M);
    if constexpr (LAST) {
#pragma unroll
      for (int r = 0; r < R; r++) v[q + r * Q] = xround(u[r]);
    } else {
      const int base = (j - k) * R + k;
#pragma unroll
      for (int r = 0; r < R; r++) sm[sidx<LAYOUT, L, NSEQ, 8, Tc>(seq, base, r * NS)] = xround(u[r]);
    }
  }
}

// fft_ct in exact-add arithmetic (same plan, layouts and synchronisation).
template <int E, int L, int LAYOUT, int NSEQ, int DIR, bool WARP = false>
__device__ __forceinline__ void fft_xp(float2 (&v)[E], float2* sm, int t, int seq, const float4* __restrict__ tw) {
  constexpr CtPlan P = ct_plan(L, E);
  constexpr int Tc = L / E;
  static_assert(!WARP || (LAYOUT == kPaddedRows && Tc <= 32 && 32 % Tc == 0), "warp-synchronous rows only");
  static_for<0, P.nst>([&](auto s_) {
    constexpr int s = decltype(s_)::value;
    constexpr bool last = (s == P.nst - 1);
    stage_xp<E, L, P.rad[s], P.ns[s], tw_base(L, E) + tw_stage_off(L, E, s), last, LAYOUT, NSEQ, DIR>(v, sm, t, seq, tw);
    if constexpr (!last) {
      fft_sync<WARP>();
#pragma unroll
      for (int e = 0; e < E; e++) v[e] = sm[sidx<LAYOUT, L, NSEQ, 8, Tc>(seq, t, Tc * e)];
      fft_sync<WARP>();
    }
  });
}

// The transform the kernels call: exact-add stages when XP, fixed point for FP64 values, else the
// plain engine.
template <bool XP, typename C, int E, int L, int LAYOUT, int NSEQ, int DIR, bool WARP = false>
__device__ __forceinline__ void fft_any(C (&v)[E], C* sm, int t, int seq, const ux_of<C>* __restrict__ tw) {
  if constexpr (XP)
    fft_xp<E, L, LAYOUT, NSEQ, DIR, WARP>(v, sm, t, seq, tw);
  else if constexpr (std::is_same<C, double2>::value)
    fft_fx<E, L, LAYOUT, NSEQ, DIR, WARP>(v, sm, t, seq, tw);
  else
    fft_ct<C, E, L, LAYOUT, NSEQ, DIR, WARP>(v, sm, t, seq, tw);
}

// r2c unpack (k_r2c_z) in exact-add arithmetic: 2X[k] = (Z[k] + Z*[L-k]) - i w^k (Z[k] - Z*[L-k]),
// halved once at the end (exact); w in the 12-bit form.
__device__ __forceinline__ float2 r2c_unpack_xp(float2 zk, float2 zm, float4 w) {
  const float bound = fabsf(zk.x) + fabsf(zk.y) + fabsf(zm.x) + fabsf(zm.y);
  const float M = xmagic(4.f * bound);
  const xc a = xsplit(zk, M), b = xsplit(xconj(zm), M);
  const xc s = a + b, d = a - b;
  const xc o = xtw(xc{make_float2(d.h.y, -d.h.x), make_float2(d.l.y, -d.l.x)}, w);  // -i d w
  return mul2(xround(s + o), 0.5f);
}

// c2r pack (k_c2r_z) in exact-add arithmetic: with A = X[k] and B = conj(X[L-k]) (0 for k = 0),
// 2Z = (A + B) + i (A - B) conj(w^k), halved once at the end; wc = conj(w^k) in the 12-bit form.
__device__ __forceinline__ float2 c2r_pack_xp(float2 xk, float2 xm, float4 wc) {
  const float bound = fabsf(xk.x) + fabsf(xk.y) + fabsf(xm.x) + fabsf(xm.y);
  const float M = xmagic(4.f * bound);
  const xc a = xsplit(xk, M), b = xsplit(xconj(xm), M);
  const xc ev = a + b, od = xtw(a - b, wc);
  return mul2(xround(xadd_i(ev, od, 1)), 0.5f);  // (2E + i 2O') / 2
}

}  // namespace pspec
