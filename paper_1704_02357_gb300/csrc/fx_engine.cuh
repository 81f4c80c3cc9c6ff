// The transform stages of FP64 contexts in 62-bit fixed point (fixpoint.cuh): each transform
// takes its FP64 values to integers on a scale of its own (one per row or column), runs the stages of
// fft_engine.cuh on them and returns FP64 values. Plans, layouts and exchanges are those of the FP32
// and FP64 radix trees; an element takes the same four registers.
//
// What it replaces: the FP64 trees were bound by GB300's FP64 pipe (15.3 clocks per point and SM in
// a 512-point y pass, 3.38 ms per 512^3 spectrum, against 0.3 ms of HBM traffic).
#pragma once
#include "fft_engine.cuh"
#include "fixpoint.cuh"

namespace pspec {

// Twiddle table entries {c_h, c_l, s_h, s_l} of FP64 contexts (fx_mul), in place of UnitOf<double>.
template <> struct UnitOf<long long> { using type = int4; };
template <> struct BaseOf<lc> { using type = long long; };

__device__ __forceinline__ lc umul(lc a, int4 w) { return fx_mul(a, w.x, w.y, w.z, w.w); }
__device__ __forceinline__ lc cadd(lc a, lc b) { return lc{a.x + b.x, a.y + b.y}; }
__device__ __forceinline__ lc csub(lc a, lc b) { return lc{a.x - b.x, a.y - b.y}; }
__device__ __forceinline__ lc cmul_i(lc a, int sgn) { return sgn > 0 ? lc{-a.y, a.x} : lc{a.y, -a.x}; }

// constants in units of 2^-62, split as fx_mul_const takes them
constexpr int fx_const_h(long long q) { return (int)((q + (1ll << 31)) >> 32); }
constexpr int fx_const_l(long long q) { return (int)(q - ((long long)fx_const_h(q) << 32)); }
constexpr long long kFxSqrtHalf = 3260954456333195553ll;  // sqrt(1/2) 2^62
constexpr long long kFxSin60 = 3993837246235628775ll;     // sin(2 pi/3) 2^62

template <> struct Dft<lc, 8> {
  static __device__ __forceinline__ void run(lc* v, int dir) {
    auto h = [](long long x) { return fx_mul_const(x, fx_const_h(kFxSqrtHalf), fx_const_l(kFxSqrtHalf)); };
    lc e[4] = {v[0], v[2], v[4], v[6]};
    lc o[4] = {v[1], v[3], v[5], v[7]};
    Dft<lc, 4>::run(e, dir);
    Dft<lc, 4>::run(o, dir);
    const lc o1 = dir > 0 ? lc{h(o[1].x - o[1].y), h(o[1].y + o[1].x)} : lc{h(o[1].x + o[1].y), h(o[1].y - o[1].x)};
    const lc o2 = cmul_i(o[2], dir);
    const lc o3 = dir > 0 ? lc{h(-o[3].x - o[3].y), h(o[3].x - o[3].y)} : lc{h(o[3].y - o[3].x), h(-o[3].x - o[3].y)};
    v[0] = cadd(e[0], o[0]);
    v[4] = csub(e[0], o[0]);
    v[1] = cadd(e[1], o1);
    v[5] = csub(e[1], o1);
    v[2] = cadd(e[2], o2);
    v[6] = csub(e[2], o2);
    v[3] = cadd(e[3], o3);
    v[7] = csub(e[3], o3);
  }
};

template <> struct Dft<lc, 3> {
  static __device__ __forceinline__ void run(lc* v, int dir) {
    auto s3 = [](long long x) { return fx_mul_const(x, fx_const_h(kFxSin60), fx_const_l(kFxSin60)); };
    const lc t = cadd(v[1], v[2]), u = csub(v[1], v[2]);
    const lc m = lc{v[0].x - fx_half(t.x), v[0].y - fx_half(t.y)};
    const long long sx = s3(u.x), sy = s3(u.y);
    const lc isu = dir > 0 ? lc{-sy, sx} : lc{sy, -sx};
    v[0] = cadd(v[0], t);
    v[1] = cadd(m, isu);
    v[2] = csub(m, isu);
  }
};

constexpr int log2_ceil(int n) { return n <= 1 ? 0 : 1 + log2_ceil((n + 1) / 2); }

__device__ __forceinline__ FxBound fx_join(FxBound a, FxBound b) {
  return FxBound{a.mx > b.mx ? a.mx : b.mx, a.sum + b.sum};
}
__device__ __forceinline__ FxBound fx_shfl_xor(FxBound a, int o) {
  return FxBound{__shfl_xor_sync(0xffffffffu, a.mx, o), __shfl_xor_sync(0xffffffffu, a.sum, o)};
}

// Bound of the whole sequence from its threads' partials. Columns (kInterleaved): threads c, c + NSEQ, ... of
// a block of Tc * NSEQ threads. Rows (kPaddedRows): Tc consecutive threads; WARP when they lie in
// one warp. The exchange buffer `sm` is used where a sequence spans several warps; it is free
// again on return. All threads of a sequence get the same bits (the additions of a tree commute).
template <int Tc, int LAYOUT, int NSEQ, bool WARP>
__device__ __forceinline__ FxBound fx_sequence_bound(FxBound b, void* sm, int t, int seq) {
  if constexpr (LAYOUT == kInterleaved) {
    constexpr int NW = (Tc * NSEQ + 31) / 32;
    if constexpr (Tc * NSEQ >= 32) {
#pragma unroll
      for (int o = NSEQ; o < 32; o <<= 1) b = fx_join(b, fx_shfl_xor(b, o));
      if constexpr (NW > 1) {
        FxBound* p = static_cast<FxBound*>(sm);  // [warp][sequence]
        constexpr int PW = NSEQ < 32 ? NSEQ : 32;
        static_assert(NSEQ <= 32, "a warp holds every sequence");
        const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
        if (l < PW) p[w * PW + l] = b;
        __syncthreads();
        b = p[seq];
#pragma unroll
        for (int i = 1; i < NW; i++) b = fx_join(b, p[i * PW + seq]);
        __syncthreads();
      }
    } else {
      // a block of less than a warp (its lanes are the sequences' threads)
      constexpr unsigned mask = Tc * NSEQ >= 32 ? 0xffffffffu : (1u << (Tc * NSEQ)) - 1u;
#pragma unroll
      for (int o = NSEQ; o < Tc * NSEQ; o <<= 1)
        b = fx_join(b, FxBound{__shfl_xor_sync(mask, b.mx, o), __shfl_xor_sync(mask, b.sum, o)});
    }
  } else {
#pragma unroll
    for (int o = 1; o < (Tc < 32 ? Tc : 32); o <<= 1) b = fx_join(b, fx_shfl_xor(b, o));
    if constexpr (Tc > 32) {
      static_assert(!WARP, "a row of more than one warp");
      constexpr int PR = Tc / 32;  // warps per row
      FxBound* p = static_cast<FxBound*>(sm);
      if ((t & 31) == 0) p[seq * PR + t / 32] = b;
      __syncthreads();
      b = p[seq * PR];
#pragma unroll
      for (int i = 1; i < PR; i++) b = fx_join(b, p[seq * PR + i]);
      __syncthreads();
    }
  }
  return b;
}

__device__ __forceinline__ lc fx_in(double2 v, int c1) { return lc{fx_from_double(v.x, c1), fx_from_double(v.y, c1)}; }
__device__ __forceinline__ double2 fx_out(lc v, int c2, bool bad) {
  if (bad) return make_double2(__longlong_as_double(0x7ff8000000000000ll), __longlong_as_double(0x7ff8000000000000ll));
  return make_double2(fx_to_double(v.x, c2), fx_to_double(v.y, c2));
}

// The same by two FP64 additions in place of some 25 integer instructions: hi and lo words pasted into the
// mantissas of 2^84 and 2^52 (times 2^-S), their offsets taken off, one rounding (ties to even). The
// integer pipe bounds the column passes (64% busy) while the FP64 pipe idles, so they convert the real
// parts this way and the imaginary parts in integers.
struct FxPaste {
  int hi, lo;     // upper words of 2^(84-S), 2^(52-S)
  double off;     // (2^84 + 2^63 + 2^52) 2^-S
};
__device__ __forceinline__ FxPaste fx_paste(int S) {
  FxPaste p;
  p.hi = (1023 + 84 - S) << 20;
  p.lo = (1023 + 52 - S) << 20;
  p.off = __hiloint2double(((1023 + 84 - S) << 20), 0) + __hiloint2double((1023 + 63 - S) << 20, 0) +
          __hiloint2double((1023 + 52 - S) << 20, 0);
  return p;
}
__device__ __forceinline__ bool fx_paste_ok(int S) { return S > -800 && S < 900; }
__device__ __forceinline__ double fx_pasted(long long q, const FxPaste& p) {
  const int hi = (int)(q >> 32) ^ 0x80000000, lo = (int)q;
  return (__hiloint2double(p.hi, hi) - p.off) + __hiloint2double(p.lo, lo);
}

// The scale of the sequence of E values per thread, with 2^extra of headroom.
template <int E, int L, int LAYOUT, int NSEQ, bool WARP>
__device__ __forceinline__ FxScale fx_sequence_scale(const double2 (&v)[E], void* sm, int t, int seq, int extra) {
  FxBound b{0u, 0.f};
#pragma unroll
  for (int e = 0; e < E; e++) {
    fx_bound_add(b, v[e].x);
    fx_bound_add(b, v[e].y);
  }
  return fx_scale(fx_sequence_bound<L / E, LAYOUT, NSEQ, WARP>(b, sm, t, seq), log2_ceil(L), extra);
}

// fft_ct of FP64 values through fixed point; `tw` holds int4 entries. PASTE: passes that leave the FP64
// pipe idle otherwise.
template <int E, int L, int LAYOUT, int NSEQ, int DIR, bool WARP = false, bool PASTE = false>
__device__ __forceinline__ void fft_fx(double2 (&v)[E], double2* sm, int t, int seq, const double2* __restrict__ tw) {
  const FxScale sc = fx_sequence_scale<E, L, LAYOUT, NSEQ, WARP>(v, sm, t, seq, 0);
  lc u[E];
#pragma unroll
  for (int e = 0; e < E; e++) u[e] = fx_in(v[e], 1084 - sc.S);
  fft_ct<lc, E, L, LAYOUT, NSEQ, DIR, WARP>(u, reinterpret_cast<lc*>(sm), t, seq, reinterpret_cast<const int4*>(tw));
  if (PASTE && fx_paste_ok(sc.S) && !sc.bad) {
    const FxPaste p = fx_paste(sc.S);
#pragma unroll
    for (int e = 0; e < E; e++) v[e] = make_double2(fx_pasted(u[e].x, p), fx_to_double(u[e].y, 1085 - sc.S));
  } else {
#pragma unroll
    for (int e = 0; e < E; e++) v[e] = fx_out(u[e], 1085 - sc.S, sc.bad);
  }
}

// A row of 2L reals as L packed pairs -> its L modes: the transform, then
// 2X[k] = (Z[k] + Z*[L-k]) - i w^k (Z[k] - Z*[L-k]), both on one scale (|2X| and the sums stay below twice
// the sum of |re| + |im|) and rounded to FP64 once. Mirrors go through the exchange buffer.
template <int E, int L, bool WARP>
__device__ __forceinline__ void fx_row_r2c(double2 (&v)[E], double2* smd, int t, int seq, const double2* __restrict__ twh,
                                           const double2* __restrict__ twr) {
  constexpr int Tc = L / E;
  const FxScale sc = fx_sequence_scale<E, L, kPaddedRows, 1, WARP>(v, smd, t, seq, 1);
  lc* sm = reinterpret_cast<lc*>(smd);
  lc u[E];
#pragma unroll
  for (int e = 0; e < E; e++) u[e] = fx_in(v[e], 1084 - sc.S);
  fft_ct<lc, E, L, kPaddedRows, 1, -1, WARP>(u, sm, t, seq, reinterpret_cast<const int4*>(twh));
#pragma unroll
  for (int e = 0; e < E; e++) sm[sidx<kPaddedRows, L, 1, 16, Tc>(seq, t, Tc * e)] = u[e];
  fft_sync<WARP>();
#pragma unroll
  for (int e = 0; e < E; e++) {
    const int k = t + Tc * e;
    const lc m = sm[sidx<kPaddedRows, L, 1, 16, Tc>(seq, k ? L - k : 0, 0)];
    const lc s = lc{u[e].x + m.x, u[e].y - m.y}, d = lc{u[e].x - m.x, u[e].y + m.y};
    const lc o = umul(lc{d.y, -d.x}, ldg_u(reinterpret_cast<const int4*>(twr) + k));
    v[e] = fx_out(cadd(s, o), 1085 - sc.S - 1, sc.bad);
  }
}

// The inverse: L stored modes X[k] (v) and their mirrors X[L-k] (m; 0 for k = 0) -> L packed pairs
// of reals, unscaled. 2Z = (A + B) + i (A - B) w^-k with A = X[k], B = X*[L-k]; the sum of |2Z| is at most
// four times that of |X|.
template <int E, int L, bool WARP>
__device__ __forceinline__ void fx_row_c2r(double2 (&v)[E], const double2 (&m)[E], double2* smd, int t, int seq,
                                           const double2* __restrict__ twh, const double2* __restrict__ twr) {
  constexpr int Tc = L / E;
  const FxScale sc = fx_sequence_scale<E, L, kPaddedRows, 1, WARP>(v, smd, t, seq, 2);
  lc u[E];
#pragma unroll
  for (int e = 0; e < E; e++) {
    const lc a = fx_in(v[e], 1084 - sc.S), b = fx_in(m[e], 1084 - sc.S);
    const lc s = lc{a.x + b.x, a.y - b.y}, d = lc{a.x - b.x, a.y + b.y};
    const lc o = umul(d, uconj(ldg_u(reinterpret_cast<const int4*>(twr) + t + Tc * e)));
    u[e] = lc{s.x - o.y, s.y + o.x};
  }
  fft_ct<lc, E, L, kPaddedRows, 1, +1, WARP>(u, reinterpret_cast<lc*>(smd), t, seq, reinterpret_cast<const int4*>(twh));
#pragma unroll
  for (int e = 0; e < E; e++) v[e] = fx_out(u[e], 1085 - sc.S - 1, sc.bad);
}

}  // namespace pspec
