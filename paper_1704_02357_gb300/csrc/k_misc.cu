// Catalog sums, mass assignment, finalisation and wedges of the SH-FFT estimator.
//   a1 catalog sums: Sec. 2.1 eq. FKP-density (alpha, I) and the shot-noise term.
//   a2 painting:     Sec. 2.3 (CIC / TSC kernels, interlaced second mesh at u - 1/2).
//   a6 finalise:     Sec. 2.1 eq. Pell-ours (4 pi / (I N_b) for l >= 2; noise for l = 0).
//   a7 wedges:       Sec. 2.2 eqs. wedge-est and Lbar.
#include <cmath>
#include <type_traits>
#include "launch.h"
#include "intconv.cuh"

namespace pspec {

constexpr int kSumThreads = 256;
// Positions further than this many cells from the corner are invalid (reported with the
// non-finite ones): beyond it the periodic reduction of the grid coordinate loses meaning.
constexpr int kMaxCellsLog2 = 38;  // |u| < 2^38 cells for a valid particle

// Grid coordinate of a position along one axis, u = (x - corner) N/L in FP64; the paint takes it to
// an integer in units of 2^-24 cell (grid_int, the power of two goes to the exponent). A particle is valid
// when every |u| is below 2^kMaxCellsLog2 cells (NaN and infinities fail), tested on the exponent
// bits. The test and the conversions (intconv.cuh) use integer instructions: GB300's FP64 pipe is
// narrow, and FP64 compares and conversions between FP64 or FP32 and 64-bit integers all run on it. (One FMA,
// x K - corner K with K = N/L, gives the same u but for rare last-bit ties; measured over 30
// axis-permutation draws of the 512^3 survey catalogs, the FP32 results then came out with higher
// median errors, so the two-operation form is kept.)
struct GridMap {
  double c[3], inv;
  __device__ __forceinline__ explicit GridMap(const PaintArgs& a) : inv(a.inv_cell) {
    c[0] = a.corner[0];
    c[1] = a.corner[1];
    c[2] = a.corner[2];
  }
  __device__ __forceinline__ double u(double x, int d) const { return (x - c[d]) * inv; }
};
__device__ __forceinline__ bool grid_ok(double u) { return exp_below(u, kMaxCellsLog2); }
__device__ __forceinline__ long long grid_int(double u) { return d2ll_rn_scaled(u, 24); }

__device__ __forceinline__ void load_pos(const PaintArgs& a, int64_t p, double& x, double& y, double& z) {
  if (a.pos_f32) {
    const float* q = static_cast<const float*>(a.pos) + 3 * p;
    x = q[0];
    y = q[1];
    z = q[2];
  } else {
    const double* q = static_cast<const double*>(a.pos) + 3 * p;
    x = q[0];
    y = q[1];
    z = q[2];
  }
}

__device__ __forceinline__ double block_sum(double v, double* red) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  __syncthreads();
  if (l == 0) red[w] = v;
  __syncthreads();
  double r = 0.0;
  if (threadIdx.x == 0)
    for (int i = 0; i < (int)(blockDim.x >> 5); i++) r += red[i];
  return r;
}

__device__ __forceinline__ double fkp_w(const PaintArgs& a, double nb) {
  if (!a.nbar) return a.wf_default;
  if (!(a.P0 > 0.0)) return 1.0;
  const double x = 1.0 + nb * a.P0;
  const unsigned e = (unsigned)(__double2hiint(x) >> 20);  // sign and exponent
  return e - 923u < 200u ? rcp_newton(x) : 1.0 / x;         // 2^-100 <= x < 2^100: the rule
}
__device__ __forceinline__ bool finite_bits(double x) { return (__double2hiint(x) & 0x7ff00000) != 0x7ff00000; }

// The FP32 mesh value of one particle: v rounded down or up to a neighbouring float, chosen
// by a hash of (particle, catalog) with the probabilities that make its expectation v. All
// particles of a catalog with constant weights share one v; rounded to nearest, its error
// would scale that catalog's whole field, survey window included, and at the lowest k the
// randoms' window exceeds the data-minus-randoms field by two orders of magnitude. Dithered,
// the rounding errors are independent across particles and only add white noise ~1e-7 of the
// shot noise. The hash is the 32-bit finaliser of MurmurHash3 (Appleby) applied to the
// particle index mixed with a per-catalog salt.
using Dither = FloatPair;  // lo, hi: the two floats around v (equal when v is a float); thr: P(hi) 2^32
__device__ __forceinline__ Dither dither_of(double v) {
  if (float_pair_ok(v)) return float_pair(v);  // integer instructions, no FP64 division
  Dither d;
  d.lo = (float)v;
  const double r = v - (double)d.lo;
  d.hi = r == 0.0 ? d.lo : nextafterf(d.lo, r > 0.0 ? INFINITY : -INFINITY);
  const double p = r == 0.0 ? 0.0 : r / ((double)d.hi - (double)d.lo);  // in [0, 1/2]
  d.thr = (uint32_t)(p * 4294967296.0);
  return d;
}
__device__ __forceinline__ uint32_t mix32(uint32_t h) {
  h ^= h >> 16;
  h *= 0x85ebca6bu;
  h ^= h >> 13;
  h *= 0xc2b2ae35u;
  h ^= h >> 16;
  return h;
}
__device__ __forceinline__ float dither_pick(const Dither& d, int64_t p, int is_randoms) {
  const uint32_t key = (uint32_t)p ^ ((uint32_t)(p >> 32) * 0x9e3779b9u) ^ (is_randoms ? 0x5bd1e995u : 0u);
  return mix32(key) < d.thr ? d.hi : d.lo;
}
// Catalog fields from the device descriptor of the current mock, when the arguments carry one.
__device__ __forceinline__ PaintArgs resolve(const PaintArgs& in) {
  PaintArgs a = in;
  if (a.dc) {
    const DevCat d = a.dc[*a.cur];
    a.pos = d.pos;
    a.weight = d.weight;
    a.nbar = d.nbar;
    a.count = d.count;
    a.pos_f32 = d.pos_f32;
  }
  return a;
}

// ------------------------------------------------------------------ a1: weighted catalogs
// Per-block partials: [0] sum w_c, [1] sum v^2 (v = w_c w_fkp), [2] sum nbar w_c w_fkp^2,
// [3] sum |v| (bounds every mesh value, for the fixed-point scale of the exact paint).
// Invalid particles are left out here and counted by the paint kernel.
// A particle whose coordinates are all below 2^safe_log2 is valid without FP64 arithmetic; a
// catalog without weights and n̄ is then only counted.
__global__ void __launch_bounds__(kSumThreads) k_catalog_partials(PaintArgs a_in, double* out) {
  __shared__ double red[kSumThreads / 32];
  const PaintArgs a = resolve(a_in);
  const GridMap gm(a);
  const bool uniform = (a.weight == nullptr) && (a.nbar == nullptr);
  const int lim32 = a.safe_log2 > 126 ? 253 : a.safe_log2 + 127, lim64 = a.safe_log2 + 1023;
  double s0 = 0.0, s1 = 0.0, s2 = 0.0, s3 = 0.0;
  const bool nb_ok = finite_bits(a.nbar_default);  // a default n̄ that is not a number leaves every particle out
  int n = 0;
  auto valid = [&](int64_t p) {
    if (a.pos_f32) {
      const unsigned* q = static_cast<const unsigned*>(a.pos) + 3 * p;
      const int e0 = (q[0] >> 23) & 0xff, e1 = (q[1] >> 23) & 0xff, e2 = (q[2] >> 23) & 0xff;
      if (max(e0, max(e1, e2)) < lim32) return true;
    } else {
      const double* q = static_cast<const double*>(a.pos) + 3 * p;
      const int e0 = (__double2hiint(q[0]) >> 20) & 0x7ff, e1 = (__double2hiint(q[1]) >> 20) & 0x7ff,
                e2 = (__double2hiint(q[2]) >> 20) & 0x7ff;
      if (max(e0, max(e1, e2)) < lim64) return true;
    }
    double x, y, z;
    load_pos(a, p, x, y, z);
    return grid_ok(gm.u(x, 0)) && grid_ok(gm.u(y, 1)) && grid_ok(gm.u(z, 2));
  };
#pragma unroll 2
  for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < a.count;
       p += (int64_t)gridDim.x * blockDim.x) {
    if (uniform) {
      n += nb_ok && valid(p) ? 1 : 0;
      continue;
    }
    const double wc = a.weight ? a.weight[p] : 1.0;
    const double nb = a.nbar ? a.nbar[p] : a.nbar_default;
    if (!(valid(p) && finite_bits(wc) && finite_bits(nb))) continue;
    const double wf = fkp_w(a, nb);
    const double v = wc * wf;
    s0 += wc;
    s1 += v * v;
    s2 += nb * v * wf;
    s3 += fabs(v);
  }
  if (uniform) {
    const double m = block_sum((double)n, red);
    if (threadIdx.x == 0) {
      const double wf = a.wf_default;
      double* o = out + (int64_t)blockIdx.x * kSumVals;
      o[0] = m;
      o[1] = nb_ok ? m * (wf * wf) : 0.0;
      o[2] = nb_ok ? m * (a.nbar_default * wf * wf) : 0.0;
      o[3] = nb_ok ? m * fabs(wf) : 0.0;
    }
    return;
  }
  const double r0 = block_sum(s0, red);
  const double r1 = block_sum(s1, red);
  const double r2 = block_sum(s2, red);
  const double r3 = block_sum(s3, red);
  if (threadIdx.x == 0) {
    double* o = out + (int64_t)blockIdx.x * kSumVals;
    o[0] = r0;
    o[1] = r1;
    o[2] = r2;
    o[3] = r3;
  }
}

// Neumaier-compensated FP64 accumulator (the block partials are few). The magnitudes are compared
// as integers: FP64 compares run on the narrow FP64 pipe.
struct Neu {
  double s = 0.0, c = 0.0;
  __device__ __forceinline__ void add(double x) {
    const double t = s + x;
    const bool s_larger = (__double_as_longlong(s) & 0x7fffffffffffffffll) >= (__double_as_longlong(x) & 0x7fffffffffffffffll);
    c += ((s_larger ? s : x) - t) + (s_larger ? x : s);
    s = t;
  }
  __device__ __forceinline__ double val() const { return s + c; }
};

// Compensated sum of one column of the block partials by one warp (every lane of it): each lane
// adds every 32nd partial, then the lanes' (sum, compensation) pairs are added in a tree. An FP64
// warp instruction holds GB300's FP64 pipe for 64 cycles however few lanes are active, so one
// thread walking the 304 partials of a catalog column by column took 190 us for a mock's sums and
// 448 us for two weighted catalogs; with one warp per column it is a chain of ~15 additions.
__device__ __forceinline__ Neu column_sum(const double* __restrict__ part, int nb, int col) {
  Neu a;
  const int lane = threadIdx.x & 31;
#pragma unroll 4
  for (int b = lane; b < nb; b += 32) a.add(part[b * kSumVals + col]);
  for (int o = 16; o > 0; o >>= 1) {
    const double s2 = __shfl_down_sync(0xffffffffu, a.s, o), c2 = __shfl_down_sync(0xffffffffu, a.c, o);
    a.add(s2);
    a.c += c2;
  }
  return a;  // lane 0
}
// Columns 0..3 of the data (warps 0..3) and randoms (warps 4..7) partials; nbd or nbr = 0 leaves
// zeros. All threads of a 256-thread block.
__device__ __forceinline__ void all_column_sums(const double* pd, int nbd, const double* pr, int nbr, double (&sum)[8]) {
  const int w = threadIdx.x >> 5;
  const Neu a = w < 4 ? column_sum(pd, nbd, w) : column_sum(pr, nbr, w - 4);
  if ((threadIdx.x & 31) == 0) sum[w] = a.val();
  __syncthreads();
}
constexpr int kFinalThreads = 256;

// The fixed-point scale 2^S of the exact paint for meshes whose values are all bounded by
// `bound` in magnitude: every cell sum then stays below 2^61 in units of 2^-S.
__device__ double fix_scale(double bound) {
  int e = 0;
  frexp(bound, &e);  // bound < 2^e
  int S = bound > 0.0 ? 61 - e : 61;
  S = S > 100 ? 100 : (S < -100 ? -100 : S);
  return ldexp(1.0, S);
}

// One block adds the block partials in a fixed order: deterministic alpha, I, S. `fix`
// (nullable) receives the exact paint's fixed-point scale for data (+v) and randoms
// (-alpha v) painted together.
__global__ void __launch_bounds__(kFinalThreads) k_catalog_final(const double* pd, int nbd, const double* pr, int nbr,
                                                                 double* d, double* fix) {
  __shared__ double sum[8];
  all_column_sums(pd, nbd, pr, nbr, sum);
  if (threadIdx.x != 0) return;
  const double wd = sum[0], sd = sum[1], ad = sum[3], wr = sum[4], sr = sum[5], ir = sum[6], ar = sum[7];
  const double alpha = wd / wr;
  d[D_WD] = wd;
  d[D_WR] = wr;
  d[D_ALPHA] = alpha;
  d[D_I] = alpha * ir;
  d[D_S] = sd + alpha * alpha * sr;
  d[D_NONFINITE] = 0.0;
  d[D_WRAPPED] = 0.0;
  d[D_SD] = sd;
  d[D_SR] = sr;
  d[D_IR] = ir;
  if (fix) *fix = fix_scale(ad + fabs(alpha) * ar);
}

// Unit completeness weights and one n̄: W = counts, v = w_fkp for every particle.
__global__ void k_derive_uniform(int64_t nd, int64_t nr, double wf, double nbar, double* d) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  const double Wd = (double)nd, Wr = (double)nr;
  const double alpha = Wd / Wr;
  const double sd = Wd * wf * wf, sr = Wr * wf * wf, ir = Wr * nbar * wf * wf;
  d[D_WD] = Wd;
  d[D_WR] = Wr;
  d[D_ALPHA] = alpha;
  d[D_I] = alpha * ir;
  d[D_S] = sd + alpha * alpha * sr;
  d[D_NONFINITE] = 0.0;
  d[D_WRAPPED] = 0.0;
  d[D_SD] = sd;
  d[D_SR] = sr;
  d[D_IR] = ir;
  d[D_FIX] = fix_scale(fabs(wf) * (Wd + alpha * Wr));
}

void launch_catalog_partials(const PaintArgs& a, double* partials, int nblocks, cudaStream_t s) {
  k_catalog_partials<<<nblocks, kSumThreads, 0, s>>>(a, partials);
}

void launch_catalog_final(const double* part_d, int nb_d, const double* part_r, int nb_r, double* derived,
                          cudaStream_t s, double* fix) {
  k_catalog_final<<<1, kFinalThreads, 0, s>>>(part_d, nb_d, part_r, nb_r, derived, fix);
}

void launch_derive_uniform(int64_t n_d, int64_t n_r, double wf, double nbar, double* derived, cudaStream_t s) {
  k_derive_uniform<<<1, 32, 0, s>>>(n_d, n_r, wf, nbar, derived);
}

// ------------------------------------------------------------------ a2: painting
__device__ __forceinline__ int wrap(int64_t i, int N) {
  if (i >= 0 && i < N) return (int)i;
  const int r = (int)(i % N);
  return r < 0 ? r + N : r;
}

// One axis of the assignment kernel. FP32 meshes use a 24-bit fixed-point grid coordinate
// U = round(u 2^24) (u computed in FP64), so the cell index is U >> 24 and the fraction is
// exact in FP32; FP64 meshes keep u in FP64. Fills the node indices (wrapped into [0, N))
// and the weights.
template <typename T, int WIN> struct Axis;

template <int WIN> struct Axis<float, WIN> {
  static __device__ __forceinline__ void nodes(int64_t U, int N, int* idx, float* w) {
    if (WIN == PSPEC_WINDOW_CIC) {
      const int64_t c = U >> 24;
      const float d = (float)(U - c * 16777216ll) * 5.9604644775390625e-8f;  // 2^-24
      w[0] = 1.f - d;
      w[1] = d;
      idx[0] = wrap(c, N);
      idx[1] = wrap(c + 1, N);
    } else {
      const int64_t c = (U + (1ll << 23)) >> 24;  // floor(u + 1/2)
      const float d = (float)(U - c * 16777216ll) * 5.9604644775390625e-8f;  // in [-1/2, 1/2)
      w[0] = 0.5f * (0.5f - d) * (0.5f - d);
      w[1] = 0.75f - d * d;
      w[2] = 0.5f * (0.5f + d) * (0.5f + d);
      idx[0] = wrap(c - 1, N);
      idx[1] = wrap(c, N);
      idx[2] = wrap(c + 1, N);
    }
  }
};

template <int WIN> struct Axis<double, WIN> {
  static __device__ __forceinline__ void nodes(double u, int N, int* idx, double* w) {
    if (WIN == PSPEC_WINDOW_CIC) {
      const double f = floor(u);
      const double d = u - f;
      const int64_t c = (int64_t)f;
      w[0] = 1.0 - d;
      w[1] = d;
      idx[0] = wrap(c, N);
      idx[1] = wrap(c + 1, N);
    } else {
      const double f = floor(u + 0.5);
      const double d = u - f;
      const int64_t c = (int64_t)f;
      w[0] = 0.5 * (0.5 - d) * (0.5 - d);
      w[1] = 0.75 - d * d;
      w[2] = 0.5 * (0.5 + d) * (0.5 + d);
      idx[0] = wrap(c - 1, N);
      idx[1] = wrap(c, N);
      idx[2] = wrap(c + 1, N);
    }
  }
};

template <typename T, int WIN>
__device__ __forceinline__ void scatter(T* __restrict__ m, int N, const int (&ix)[3], const int (&iy)[3],
                                        const int (&iz)[3], const T (&wx)[3], const T (&wy)[3], const T (&wz)[3],
                                        T v) {
  constexpr int K = WIN == PSPEC_WINDOW_CIC ? 2 : 3;
#pragma unroll
  for (int a = 0; a < K; a++) {
    const T va = v * wx[a];
#pragma unroll
    for (int b = 0; b < K; b++) {
      const T vb = va * wy[b];
      T* row = m + ((int64_t)ix[a] * N + iy[b]) * N;
#pragma unroll
      for (int c = 0; c < K; c++) atomicAdd(row + iz[c], vb * wz[c]);
    }
  }
}

template <typename T, int WIN, bool INTER>
__global__ void __launch_bounds__(256) k_paint(PaintArgs a_in, int is_randoms, double* __restrict__ derived,
                                               T* __restrict__ m1, T* __restrict__ m2, int N) {
  const PaintArgs a = resolve(a_in);
  const double sign = is_randoms == 1 ? -derived[D_ALPHA] : 1.0;
  const bool uniform = (a.weight == nullptr) && (a.nbar == nullptr);
  const double v_uniform = sign * a.wf_default;
  const Dither d_uniform = dither_of(v_uniform);
  const GridMap gm(a);
  const int64_t lim24 = (int64_t)N << 24;
  unsigned bad = 0, out = 0;
  for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < a.count;
       p += (int64_t)gridDim.x * blockDim.x) {
    double x, y, z;
    load_pos(a, p, x, y, z);
    double wc = 1.0, nb = a.nbar_default;
    if (!uniform) {
      wc = a.weight ? a.weight[p] : 1.0;
      nb = a.nbar ? a.nbar[p] : a.nbar_default;
    }
    const double ux = gm.u(x, 0), uy = gm.u(y, 1), uz = gm.u(z, 2);
    if (!(grid_ok(ux) && grid_ok(uy) && grid_ok(uz) && (uniform || (finite_bits(wc) && finite_bits(nb))))) {
      bad++;
      continue;
    }
    T v;
    if constexpr (sizeof(T) == 4)
      v = dither_pick(uniform ? d_uniform : dither_of(sign * wc * fkp_w(a, nb)), p, is_randoms);
    else
      v = sign * wc * fkp_w(a, nb);
    int ix[3], iy[3], iz[3];
    T wx[3], wy[3], wz[3];
    if constexpr (sizeof(T) == 4) {
      const int64_t Ux = grid_int(ux), Uy = grid_int(uy), Uz = grid_int(uz);
      if (Ux < 0 || Ux >= lim24 || Uy < 0 || Uy >= lim24 || Uz < 0 || Uz >= lim24) out++;
      Axis<float, WIN>::nodes(Ux, N, ix, wx);
      Axis<float, WIN>::nodes(Uy, N, iy, wy);
      Axis<float, WIN>::nodes(Uz, N, iz, wz);
      scatter<T, WIN>(m1, N, ix, iy, iz, wx, wy, wz, v);
      if (INTER) {
        const int64_t h = 1ll << 23;  // half a cell
        Axis<float, WIN>::nodes(Ux - h, N, ix, wx);
        Axis<float, WIN>::nodes(Uy - h, N, iy, wy);
        Axis<float, WIN>::nodes(Uz - h, N, iz, wz);
        scatter<T, WIN>(m2, N, ix, iy, iz, wx, wy, wz, v);
      }
    } else {
      const double lim = (double)N;
      if (ux < 0.0 || ux >= lim || uy < 0.0 || uy >= lim || uz < 0.0 || uz >= lim) out++;
      Axis<double, WIN>::nodes(ux, N, ix, wx);
      Axis<double, WIN>::nodes(uy, N, iy, wy);
      Axis<double, WIN>::nodes(uz, N, iz, wz);
      scatter<T, WIN>(m1, N, ix, iy, iz, wx, wy, wz, v);
      if (INTER) {
        Axis<double, WIN>::nodes(ux - 0.5, N, ix, wx);
        Axis<double, WIN>::nodes(uy - 0.5, N, iy, wy);
        Axis<double, WIN>::nodes(uz - 0.5, N, iz, wz);
        scatter<T, WIN>(m2, N, ix, iy, iz, wx, wy, wz, v);
      }
    }
  }
  // rare events: one atomic per warp that saw any
  const unsigned nb_w = __reduce_add_sync(0xffffffffu, bad);
  const unsigned no_w = __reduce_add_sync(0xffffffffu, out);
  if ((threadIdx.x & 31) == 0) {
    if (nb_w) atomicAdd(&derived[D_NONFINITE], (double)nb_w);
    if (no_w) atomicAdd(&derived[D_WRAPPED], (double)no_w);
  }
}

template <typename T>
void launch_paint(const PaintArgs& a, int window, int interlaced, int is_randoms, double* derived, T* mesh1, T* mesh2,
                  int N, int nblocks, cudaStream_t s) {
  if (!a.dc && a.count <= 0) return;
  const int64_t need = a.dc ? nblocks : (a.count + 255) / 256;
  const int nb = (int)(need < nblocks ? need : nblocks);
  if (window == PSPEC_WINDOW_CIC) {
    if (interlaced)
      k_paint<T, PSPEC_WINDOW_CIC, true><<<nb, 256, 0, s>>>(a, is_randoms, derived, mesh1, mesh2, N);
    else
      k_paint<T, PSPEC_WINDOW_CIC, false><<<nb, 256, 0, s>>>(a, is_randoms, derived, mesh1, mesh2, N);
  } else {
    if (interlaced)
      k_paint<T, PSPEC_WINDOW_TSC, true><<<nb, 256, 0, s>>>(a, is_randoms, derived, mesh1, mesh2, N);
    else
      k_paint<T, PSPEC_WINDOW_TSC, false><<<nb, 256, 0, s>>>(a, is_randoms, derived, mesh1, mesh2, N);
  }
}
template void launch_paint<float>(const PaintArgs&, int, int, int, double*, float*, float*, int, int, cudaStream_t);
template void launch_paint<double>(const PaintArgs&, int, int, int, double*, double*, double*, int, int,
                                   cudaStream_t);

// ------------------------------------------------------------------ a2: tile-binned painting
// FP32 meshes, accumulated exactly. One block per 16^3-cell tile owns its cells: it sums every
// contribution that lands in them as a 64-bit fixed-point integer (units 2^-S, S from the
// catalogs' sum of |v| so that no sum can overflow) and stores each cell once, rounded to FP32.
// Integer sums do not depend on the order of the additions, so the meshes are the exact sums of
// the particles' FP32 contributions, rounded once, identical from run to run. With FP32 atomics
// instead, each run adds in another order, and the rounding of the many small randoms
// contributions left an order-dependent error on the survey window's largest-scale modes large
// enough to move a 3%-of-P_0 quadrupole in the first k bin by ~1e-5.
//
// A particle whose footprint (both interlaced meshes) crosses a tile face is listed for every
// tile it touches: per axis the footprint spans at most 4 cells, so at most 2 tiles per axis.
// Record: per axis the grid coordinate relative to the origin of the particle's first tile,
// in 2^-24 cells (29 bits), with bit 31 set when the footprint reaches the next tile; in the
// tile-sorted copy bit 29 says the record sits in that next tile (coordinate 16 cells less).
constexpr int kPT = 16;  // tile side (cells)
constexpr int kPT3 = kPT * kPT * kPT;
constexpr unsigned kNoTile = 0xffffffffu;
constexpr unsigned kCoordMask = (1u << 29) - 1u;
constexpr unsigned kSpan2 = 1u << 31;
constexpr unsigned kNextTile = 1u << 29;

// Lowest and highest footprint cell along one axis (unwrapped), both meshes.
template <int WIN, bool INTER>
__device__ __forceinline__ void footprint(int64_t U, int64_t& lo, int64_t& hi) {
  if (WIN == PSPEC_WINDOW_CIC) {
    const int64_t c1 = U >> 24;
    lo = INTER ? ((U - (1ll << 23)) >> 24) : c1;
    hi = c1 + 1;
  } else {
    const int64_t c1 = (U + (1ll << 23)) >> 24;  // floor(u + 1/2)
    const int64_t c2 = U >> 24;                   // centre of the mesh painted at u - 1/2
    lo = (INTER ? (c1 < c2 ? c1 : c2) : c1) - 1;
    hi = (INTER ? (c1 > c2 ? c1 : c2) : c1) + 1;
  }
}

// Catalogs of one prep launch (blockIdx.y): their records follow one another.
struct PrepArgs {
  PaintArgs a[2];
  int kind[2];
};
// Meshes of up to this many tiles (256^3) count and place records per block in shared memory first: few
// tiles mean many records each, and the global counter of a tile then takes one atomic add per block
// instead of one per record (0.4 million galaxies on 128^3, whose densest tiles hold thousands:
// prep 95 -> 17 us, scatter 94 -> 18 us). Whole paint of 9 million survey particles, CIC, with global counters and this
// way: 128^3 3.80 and 1.02 ms, 192^3 1.91 and 0.82, 256^3 1.06 and 0.86; uniform ones at 256^3 0.88 and 0.92 (TSC 1.90 and
// 1.63); 55 000 at 256^3 0.091 and 0.095. At 512^3 placing per block was slower.
constexpr int kSharedTiles = 4096;

template <int WIN, bool INTER, bool SHARED>
__global__ void __launch_bounds__(512) k_ptile_prep(const __grid_constant__ PrepArgs pa, double* __restrict__ derived,
                                                    TileArgs ta, int N) {
  extern __shared__ __align__(16) unsigned hist[];  // SHARED: records per tile of this block
  const PaintArgs a = resolve(pa.a[blockIdx.y]);
  const int is_randoms = pa.kind[blockIdx.y];
  const int64_t offset = blockIdx.y ? pa.a[0].count : 0;
  const double sign = is_randoms == 1 ? -derived[D_ALPHA] : 1.0;
  const bool uniform = (a.weight == nullptr) && (a.nbar == nullptr);
  const double v_uniform = sign * a.wf_default;
  const Dither d_uniform = dither_of(v_uniform);
  const GridMap gm(a);
  const int64_t lim24 = (int64_t)N << 24;
  const int nts = N / kPT, ntiles = nts * nts * nts;
  unsigned* cnt = SHARED ? hist : ta.cnt;
  if (SHARED) {
    if ((int64_t)blockIdx.x * blockDim.x >= a.count) return;  // uniform over the block
    for (int i = threadIdx.x; i < ntiles; i += blockDim.x) hist[i] = 0u;
    __syncthreads();
  }
  unsigned bad = 0, out = 0;
  for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < a.count;
       p += (int64_t)gridDim.x * blockDim.x) {
    double x, y, z;
    load_pos(a, p, x, y, z);
    double wc = 1.0, nb = a.nbar_default;
    if (!uniform) {
      wc = a.weight ? a.weight[p] : 1.0;
      nb = a.nbar ? a.nbar[p] : a.nbar_default;
    }
    const double uu[3] = {gm.u(x, 0), gm.u(y, 1), gm.u(z, 2)};
    if (!(grid_ok(uu[0]) && grid_ok(uu[1]) && grid_ok(uu[2]) && (uniform || (finite_bits(wc) && finite_bits(nb))))) {
      bad++;
      ta.tile_of[offset + p] = kNoTile;
      continue;
    }
    const int64_t Ud[3] = {grid_int(uu[0]), grid_int(uu[1]), grid_int(uu[2])};
    if (Ud[0] < 0 || Ud[0] >= lim24 || Ud[1] < 0 || Ud[1] >= lim24 || Ud[2] < 0 || Ud[2] >= lim24) out++;
    const float v = dither_pick(uniform ? d_uniform : dither_of(sign * wc * fkp_w(a, nb)), p, is_randoms);
    unsigned packed[3];
    int tb[3], span[3];
    for (int d = 0; d < 3; d++) {
      const int64_t U = Ud[d];
      int64_t lo, hi;
      footprint<WIN, INTER>(U, lo, hi);
      const int low = wrap(lo, N);  // the footprint's first cell, wrapped; U shifted by the same period
      tb[d] = low / kPT;
      const int64_t rel = U - (lo - low + (int64_t)tb[d] * kPT) * 16777216ll;  // in [0, 19 cells)
      span[d] = (low - tb[d] * kPT) + (int)(hi - lo) >= kPT ? 2 : 1;
      packed[d] = (unsigned)rel | (span[d] == 2 ? kSpan2 : 0u);
    }
    const unsigned tile = (unsigned)((tb[0] * nts + tb[1]) * nts + tb[2]);
    ta.rec[offset + p] = make_uint4(packed[0], packed[1], packed[2], __float_as_uint(v));
    ta.tile_of[offset + p] = tile;
    for (int dx = 0; dx < span[0]; dx++)
      for (int dy = 0; dy < span[1]; dy++)
        for (int dz = 0; dz < span[2]; dz++) {
          const int t = ((((tb[0] + dx) % nts) * nts + (tb[1] + dy) % nts) * nts) + (tb[2] + dz) % nts;
          atomicAdd(&cnt[t], 1u);
        }
  }
  if (SHARED) {
    __syncthreads();
    for (int i = threadIdx.x; i < ntiles; i += blockDim.x)
      if (hist[i]) atomicAdd(&ta.cnt[i], hist[i]);
  }
  const unsigned nb_w = __reduce_add_sync(0xffffffffu, bad);
  const unsigned no_w = __reduce_add_sync(0xffffffffu, out);
  if ((threadIdx.x & 31) == 0) {
    if (nb_w) atomicAdd(&derived[D_NONFINITE], (double)nb_w);
    if (no_w) atomicAdd(&derived[D_WRAPPED], (double)no_w);
  }
}

// Places in the tile-sorted copy: off[] and cursor[]. Each block takes 1024 tiles, one a thread, adds
// their counts up in an exclusive prefix sum and reserves the block's range with one atomic add on
// the counter behind the counts (cleared with them). The ranges of the blocks lie in any order: a
// tile only needs a range of its own. (One block scanning all tiles, each thread a run of them
// twice over, took 85 us at 512^3 and 177 us at 768^3.)
__global__ void __launch_bounds__(1024) k_ptile_scan(TileArgs ta, int ntiles) {
  __shared__ unsigned wsum[32], base;
  const int i = blockIdx.x * 1024 + threadIdx.x, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const unsigned n = i < ntiles ? ta.cnt[i] : 0u;
  unsigned inc = n;
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned v = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += v;
  }
  if (lane == 31) wsum[w] = inc;
  __syncthreads();
  if (w == 0) {
    unsigned v = wsum[lane];
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned u = __shfl_up_sync(0xffffffffu, v, o);
      if (lane >= o) v += u;
    }
    wsum[lane] = v;
    if (lane == 31) base = atomicAdd(&ta.cnt[ntiles], v);
  }
  __syncthreads();
  if (i >= ntiles) return;
  const unsigned at = base + (w ? wsum[w - 1] : 0u) + inc - n;
  ta.off[i] = at;
  ta.cursor[i] = at;
  ta.cursor[ntiles + i] = at + n;
}

// Each record goes to every tile its footprint touches (the order within a tile is free: the
// tile's sums are exact): a record that touches one tile only to the front of that tile's range, the
// copies of the others to its back, so that the tile paint runs the front without tests.
__global__ void __launch_bounds__(256) k_ptile_scatter(TileArgs ta, int64_t total, const DevCat* dc, const int* cur,
                                                       int N) {
  if (dc) total = dc[*cur].count;
  const int nts = N / kPT, ntiles = nts * nts * nts;
  for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < total; p += (int64_t)gridDim.x * blockDim.x) {
    const unsigned t = ta.tile_of[p];
    if (t == kNoTile) continue;
    const uint4 r = ta.rec[p];
    if (!((r.x | r.y | r.z) & kSpan2)) {
      ta.sorted[atomicAdd(&ta.cursor[t], 1u)] = r;
      continue;
    }
    const int tb[3] = {(int)(t / (nts * nts)), (int)((t / nts) % nts), (int)(t % nts)};
    const int sx = (r.x & kSpan2) ? 2 : 1, sy = (r.y & kSpan2) ? 2 : 1, sz = (r.z & kSpan2) ? 2 : 1;
    for (int dx = 0; dx < sx; dx++)
      for (int dy = 0; dy < sy; dy++)
        for (int dz = 0; dz < sz; dz++) {
          const int tt = ((((tb[0] + dx) % nts) * nts + (tb[1] + dy) % nts) * nts) + (tb[2] + dz) % nts;
          const unsigned pos = atomicSub(&ta.cursor[ntiles + tt], 1u) - 1u;
          ta.sorted[pos] = make_uint4((r.x & kCoordMask) | (dx ? kNextTile : 0u),
                                      (r.y & kCoordMask) | (dy ? kNextTile : 0u),
                                      (r.z & kCoordMask) | (dz ? kNextTile : 0u), r.w);
        }
  }
}

// The same for meshes of few tiles: each block first counts its records per tile in shared memory,
// reserves the block's share of every tile's range, front and back, with one atomic add each, and
// then places its records with shared cursors.
__global__ void __launch_bounds__(512) k_ptile_scatter_shared(TileArgs ta, int64_t total, const DevCat* dc, const int* cur,
                                                              int N) {
  extern __shared__ __align__(16) unsigned at[];  // [2][ntiles]: counts, then the next place
  if (dc) total = dc[*cur].count;
  const int nts = N / kPT, ntiles = nts * nts * nts;
  const int64_t p0 = (int64_t)blockIdx.x * blockDim.x, step = (int64_t)gridDim.x * blockDim.x;
  if (p0 >= total) return;  // uniform over the block
  for (int i = threadIdx.x; i < 2 * ntiles; i += blockDim.x) at[i] = 0u;
  __syncthreads();
  // f(entry of `at`, copy) for each tile the record touches
  auto each = [&](unsigned t, unsigned sx, unsigned sy, unsigned sz, auto&& f) {
    if (!((sx | sy | sz) & kSpan2)) {
      f((int)t, 0u, 0u, 0u);
      return;
    }
    const int tb[3] = {(int)(t / (nts * nts)), (int)((t / nts) % nts), (int)(t % nts)};
    const unsigned ex = sx >> 31, ey = sy >> 31, ez = sz >> 31;
    for (unsigned dx = 0; dx <= ex; dx++)
      for (unsigned dy = 0; dy <= ey; dy++)
        for (unsigned dz = 0; dz <= ez; dz++)
          f(ntiles + ((((tb[0] + (int)dx) % nts) * nts + (tb[1] + (int)dy) % nts) * nts) + (tb[2] + (int)dz) % nts, dx, dy, dz);
  };
  for (int64_t p = p0 + threadIdx.x; p < total; p += step) {
    const unsigned t = ta.tile_of[p];
    if (t == kNoTile) continue;
    const uint4 r = ta.rec[p];
    each(t, r.x, r.y, r.z, [&](int i, unsigned, unsigned, unsigned) { atomicAdd(&at[i], 1u); });
  }
  __syncthreads();
  for (int i = threadIdx.x; i < ntiles; i += blockDim.x) {
    const unsigned nf = at[i], nb = at[ntiles + i];
    if (nf) at[i] = atomicAdd(&ta.cursor[i], nf);
    if (nb) at[ntiles + i] = atomicSub(&ta.cursor[ntiles + i], nb) - nb;
  }
  __syncthreads();
  for (int64_t p = p0 + threadIdx.x; p < total; p += step) {
    const unsigned t = ta.tile_of[p];
    if (t == kNoTile) continue;
    const uint4 r = ta.rec[p];
    each(t, r.x, r.y, r.z, [&](int i, unsigned dx, unsigned dy, unsigned dz) {
      ta.sorted[atomicAdd(&at[i], 1u)] = make_uint4((r.x & kCoordMask) | (dx ? kNextTile : 0u), (r.y & kCoordMask) | (dy ? kNextTile : 0u),
                                                    (r.z & kCoordMask) | (dz ? kNextTile : 0u), r.w);
    });
  }
}

// Tile-local node indices (may fall outside [0, kPT): not this tile's) and weights along one
// axis from the tile-local grid coordinate V (2^24 per cell).
template <int WIN>
__device__ __forceinline__ void tile_nodes(int V, int* idx, float* w) {
  if (WIN == PSPEC_WINDOW_CIC) {
    const int c = V >> 24;
    const float d = (float)(V - c * 16777216) * 5.9604644775390625e-8f;
    w[0] = 1.f - d;
    w[1] = d;
    idx[0] = c;
    idx[1] = c + 1;
  } else {
    const int c = (V + (1 << 23)) >> 24;
    const float d = (float)(V - c * 16777216) * 5.9604644775390625e-8f;
    w[0] = 0.5f * (0.5f - d) * (0.5f - d);
    w[1] = __fmaf_rn(-d, d, 0.75f);  // one rounding, whatever the compiler contracts elsewhere
    w[2] = 0.5f * (0.5f + d) * (0.5f + d);
    idx[0] = c - 1;
    idx[1] = c;
    idx[2] = c + 1;
  }
}

__device__ __forceinline__ bool in_tile(int i) { return (unsigned)i < (unsigned)kPT; }

// Adds the 64-bit integer q into the cell's sum held as two 32-bit words (lo at acc[c], hi at
// acc[c + hi_off]) with 32-bit shared atomics: lo wraps modulo 2^32, and each add that wraps it
// (the returned old value shows it) carries 1 into hi, so hi:lo is the exact sum modulo 2^64 in
// any order. The hi add is skipped when it adds 0 (small q, or a small negative q that carried).
__device__ __forceinline__ void add64(unsigned* acc, int c, int hi_off, long long q) {
  const unsigned long long u = (unsigned long long)q;
  const unsigned lo = (unsigned)u, hi = (unsigned)(u >> 32);
  const unsigned old = atomicAdd(acc + c, lo);
  const unsigned h = hi + (old + lo < old ? 1u : 0u);
  if (h) atomicAdd(acc + c + hi_off, h);
}

// |X| rounded to an integer (nearest, ties to even) for 0 <= X < 2^62, as f2ll_rn_int. Nearly every
// contribution has an exponent past its 24 bits (X >= 2^23) and only shifts.
__device__ __forceinline__ unsigned long long f2ull_mag(float X) {
  const unsigned b = __float_as_uint(X);
  const int sh = (int)(b >> 23) - 150;
  if (sh >= 0) return (unsigned long long)((b & 0x7fffffu) | 0x800000u) << sh;
  return __float2uint_rn(X);
}

// The contributions v wx wy wz (FP32, rounded as the direct paint rounds them) in units of 2^-S;
// vs = |v| 2^S (a power of two: the products round alike), neg its sign. FULL: every cell lies in
// the tile.
template <int WIN, bool FULL>
__device__ __forceinline__ void tile_scatter(unsigned* acc, int hi_off, const int (&ix)[3], const int (&iy)[3],
                                             const int (&iz)[3], const float (&wx)[3], const float (&wy)[3],
                                             const float (&wz)[3], float vs, bool neg) {
  constexpr int K = WIN == PSPEC_WINDOW_CIC ? 2 : 3;
#pragma unroll
  for (int a = 0; a < K; a++) {
    if (!FULL && !in_tile(ix[a])) continue;
    const float va = vs * wx[a];
#pragma unroll
    for (int b = 0; b < K; b++) {
      if (!FULL && !in_tile(iy[b])) continue;
      const float vb = va * wy[b];
      const int row = (ix[a] * kPT + iy[b]) * kPT;
#pragma unroll
      for (int c = 0; c < K; c++) {
        if (!FULL && !in_tile(iz[c])) continue;
        const unsigned long long q = f2ull_mag(vb * wz[c]);
        add64(acc, row + iz[c], hi_off, (long long)(neg ? 0ull - q : q));
      }
    }
  }
}

// Both meshes' contributions of one record.
template <int WIN, bool INTER, bool FULL>
__device__ __forceinline__ void tile_record(unsigned* acc, const uint4 r, float scale) {
  constexpr int HI = (INTER ? 2 : 1) * kPT3;
  const float v = __uint_as_float(r.w), vs = fabsf(v) * scale;
  const bool neg = (r.w >> 31) != 0u;
  int V[3] = {(int)(r.x & kCoordMask), (int)(r.y & kCoordMask), (int)(r.z & kCoordMask)};
  if (!FULL) {
    V[0] -= (r.x & kNextTile) ? (kPT << 24) : 0;
    V[1] -= (r.y & kNextTile) ? (kPT << 24) : 0;
    V[2] -= (r.z & kNextTile) ? (kPT << 24) : 0;
  }
  int ix[3], iy[3], iz[3];
  float wx[3], wy[3], wz[3];
  tile_nodes<WIN>(V[0], ix, wx);
  tile_nodes<WIN>(V[1], iy, wy);
  tile_nodes<WIN>(V[2], iz, wz);
  tile_scatter<WIN, FULL>(acc, HI, ix, iy, iz, wx, wy, wz, vs, neg);
  if (INTER) {
    const int h = 1 << 23;  // half a cell
    tile_nodes<WIN>(V[0] - h, ix, wx);
    tile_nodes<WIN>(V[1] - h, iy, wy);
    tile_nodes<WIN>(V[2] - h, iz, wz);
    tile_scatter<WIN, FULL>(acc + kPT3, HI, ix, iy, iz, wx, wy, wz, vs, neg);
  }
}

// Threads of a tile's block. Interlaced, three blocks' accumulators (64 KB each) fit an SM, and the shared atomics
// need the warps: 512 threads keep 48 warps resident, 256 kept 24. Tiles of few particles (below 64 on average) have more
// to clear and to store than to add and run better with blocks of 256 (512^3, 16 a tile: TSC paint 1161 -> 1099 us; 64 a tile
// box 1397 -> 1319 but survey 821 -> 845). Without interlacing (32 KB) 256 threads keep as many warps in twice the blocks,
// whose clearing, adding and storing overlap (512^3 box: 4 a tile 337 -> 214 us, 64 587 -> 478, 1024 2416 -> 2300); meshes of
// up to 192^3 keep 512 for crowded tiles, whose few long chains of records decide (192^3 survey, TSC, 512 a tile 147 against
// 155 us, 1024 237 against 263). Meshes of at most kFewTiles tiles (96^3) leave SMs idle or with one block:
// 1024 threads shorten each tile's chain of records.
constexpr int kFewTiles = 216, kSmallTiles = 1728;
constexpr int kSparseTile = 64, kCrowdedTile = 512;  // particles per tile
template <bool INTER> int tile_paint_threads(int ntiles, int64_t count) {
  if (ntiles <= kFewTiles) return 1024;
  if (INTER) return count < (int64_t)kSparseTile * ntiles ? 256 : 512;
  return ntiles <= kSmallTiles && count >= (int64_t)kCrowdedTile * ntiles ? 512 : 256;
}

// One block per tile (every tile, so that empty tiles store their zeros): sums its records into
// shared 64-bit accumulators (lo words of both meshes, then hi words), then stores each cell of
// the tile once, four cells along z per 16-byte store. A tile without records stores zeros and
// skips the accumulators. With cached randoms meshes r1, r2 (batched mocks; r1 null: none) it stores
// cell - alpha * randoms cell instead: the same FMA as a pass of its own over the meshes, which
// would read and write each once more (135 us a mesh at 384^3).
template <int WIN, bool INTER, int NT>
__global__ void __launch_bounds__(NT, NT == 256 && !INTER ? 6 : (NT <= 512 ? 3 : 1)) k_ptile_paint(TileArgs ta, float* __restrict__ m1, float* __restrict__ m2,
                                                     int N, const double* __restrict__ fix,
                                                     const float* __restrict__ r1, const float* __restrict__ r2,
                                                     const double* __restrict__ alpha) {
  extern __shared__ __align__(16) unsigned acc[];  // lo [NM][kPT^3], then hi [NM][kPT^3]
  constexpr int NM = INTER ? 2 : 1;
  constexpr int HI = NM * kPT3;
  const int tile = blockIdx.x;
  const unsigned n = ta.cnt[tile];
  const unsigned o = ta.off[tile];
  const unsigned nf = ta.cursor[tile] - o;  // records that touch this tile only
  const int nts = N / kPT;
  const int tz = tile % nts, ty = (tile / nts) % nts, tx = tile / (nts * nts);
  // 16-byte group i of the tile: mesh, then cells (lx, ly, lz..lz+3); its mesh address
  auto group = [&](int i, int& mesh) {
    mesh = i / (kPT3 / 4);
    const int cell = (i - mesh * (kPT3 / 4)) * 4;
    const int lx = cell / (kPT * kPT), ly = (cell / kPT) % kPT, lz = cell % kPT;
    return ((int64_t)(tx * kPT + lx) * N + (ty * kPT + ly)) * N + tz * kPT + lz;
  };
  const float al = r1 ? (float)*alpha : 0.f;
  auto store = [&](int mesh, int64_t g, float4 v) {
    if (r1) {
      const float4 r = __ldg(reinterpret_cast<const float4*>((mesh ? r2 : r1) + g));
      v = make_float4(fmaf(-al, r.x, v.x), fmaf(-al, r.y, v.y), fmaf(-al, r.z, v.z), fmaf(-al, r.w, v.w));
    }
    *reinterpret_cast<float4*>((mesh ? m2 : m1) + g) = v;
  };
  if (n == 0) {
    for (int i = threadIdx.x; i < NM * kPT3 / 4; i += blockDim.x) {
      int mesh;
      const int64_t g = group(i, mesh);
      store(mesh, g, make_float4(0.f, 0.f, 0.f, 0.f));
    }
    return;  // uniform over the block: no barrier is left behind
  }
  const double sc = *fix;
  const float scale = (float)sc, inv = (float)(1.0 / sc);  // powers of two: exact
  for (int i = threadIdx.x; i < 2 * NM * kPT3 / 4; i += blockDim.x) reinterpret_cast<uint4*>(acc)[i] = make_uint4(0u, 0u, 0u, 0u);
  __syncthreads();
  // the others from the last warp on: a sparse tile's two short runs go to different warps
  for (unsigned q = threadIdx.x; q < nf; q += NT) tile_record<WIN, INTER, true>(acc, ta.sorted[o + q], scale);
  for (unsigned q = nf + (NT - 1 - threadIdx.x); q < n; q += NT) tile_record<WIN, INTER, false>(acc, ta.sorted[o + q], scale);
  __syncthreads();
  for (int i = threadIdx.x; i < NM * kPT3 / 4; i += blockDim.x) {
    int mesh;
    const int64_t g = group(i, mesh);
    const uint4 lo = reinterpret_cast<const uint4*>(acc)[i], hi = reinterpret_cast<const uint4*>(acc + HI)[i];
    auto cell = [&](unsigned l, unsigned h) {
      return ll2f_rn_int((long long)(((unsigned long long)h << 32) | l)) * inv;
    };
    store(mesh, g, make_float4(cell(lo.x, hi.x), cell(lo.y, hi.y), cell(lo.z, hi.z), cell(lo.w, hi.w)));
  }
}

namespace {
bool shared_tiles(int N) { return (N / kPT) * (N / kPT) * (N / kPT) <= kSharedTiles; }
// Blocks of 512 threads for `count` particles: with shared counts a few per SM, each with a long run of
// particles to share them; else enough to fill the SMs several times over.
int particle_blocks(int64_t count, bool shared, int nsm) {
  const int64_t need = (count + 511) / 512, cap = (shared ? 4 : 8) * (int64_t)nsm;
  return (int)(need < 1 ? 1 : (need < cap ? need : cap));
}
template <int WIN, bool INTER>
void ptile_prep_v(const PrepArgs& pa, int ncat, int64_t most, double* derived, const TileArgs& ta, int N, int nsm, cudaStream_t s) {
  const bool sh = shared_tiles(N);
  const dim3 grid(particle_blocks(most, sh, nsm), ncat);
  const size_t smem = sh ? (size_t)(N / kPT) * (N / kPT) * (N / kPT) * sizeof(unsigned) : 0;
  if (sh)
    k_ptile_prep<WIN, INTER, true><<<grid, 512, smem, s>>>(pa, derived, ta, N);
  else
    k_ptile_prep<WIN, INTER, false><<<grid, 512, 0, s>>>(pa, derived, ta, N);
}
}  // namespace

void launch_ptile_prep(const PaintArgs& a, int kind_a, const PaintArgs* b, int kind_b, int window, int interlaced,
                       double* derived, const TileArgs& ta, int N, int nsm, cudaStream_t s) {
  PrepArgs pa;
  pa.a[0] = a;
  pa.kind[0] = kind_a;
  pa.a[1] = b ? *b : a;
  pa.kind[1] = kind_b;
  // a catalog from a device descriptor (dc): its size is known on the device only
  const int64_t most = a.dc ? INT64_MAX / 2 : (b && b->count > a.count ? b->count : a.count);
  if (most <= 0) return;
  const int ncat = b ? 2 : 1;
  if (window == PSPEC_WINDOW_CIC) {
    if (interlaced)
      ptile_prep_v<PSPEC_WINDOW_CIC, true>(pa, ncat, most, derived, ta, N, nsm, s);
    else
      ptile_prep_v<PSPEC_WINDOW_CIC, false>(pa, ncat, most, derived, ta, N, nsm, s);
  } else {
    if (interlaced)
      ptile_prep_v<PSPEC_WINDOW_TSC, true>(pa, ncat, most, derived, ta, N, nsm, s);
    else
      ptile_prep_v<PSPEC_WINDOW_TSC, false>(pa, ncat, most, derived, ta, N, nsm, s);
  }
}

void launch_ptile_scan(const TileArgs& ta, int ntiles, cudaStream_t s) {
  k_ptile_scan<<<(ntiles + 1023) / 1024, 1024, 0, s>>>(ta, ntiles);
}

void launch_ptile_scatter(const TileArgs& ta, int64_t total, const DevCat* dc, const int* cur, int N, int nsm,
                          cudaStream_t s) {
  if (!dc && total <= 0) return;
  const bool sh = shared_tiles(N);
  const int nb = particle_blocks(dc ? INT64_MAX / 2 : total, sh, nsm);
  if (sh)
    k_ptile_scatter_shared<<<nb, 512, 2 * (size_t)(N / kPT) * (N / kPT) * (N / kPT) * sizeof(unsigned), s>>>(ta, total, dc, cur, N);
  else
    k_ptile_scatter<<<2 * nb, 256, 0, s>>>(ta, total, dc, cur, N);
}

template <int WIN, bool INTER>
static void ptile_paint_v(const TileArgs& ta, int64_t count, float* m1, float* m2, int N, const double* fix, const float* r1,
                          const float* r2, const double* alpha, cudaStream_t s) {
  const int ntiles = (N / kPT) * (N / kPT) * (N / kPT);
  const size_t smem = (size_t)(INTER ? 2 : 1) * kPT3 * sizeof(unsigned long long);
  auto go = [&](auto nt) {
    constexpr int NT = decltype(nt)::value;
    allow_smem(k_ptile_paint<WIN, INTER, NT>, smem);
    k_ptile_paint<WIN, INTER, NT><<<ntiles, NT, smem, s>>>(ta, m1, m2, N, fix, r1, r2, alpha);
  };
  switch (tile_paint_threads<INTER>(ntiles, count)) {
    case 256: go(std::integral_constant<int, 256>{}); break;
    case 512: go(std::integral_constant<int, 512>{}); break;
    default: go(std::integral_constant<int, 1024>{});
  }
}

void launch_ptile_paint(const TileArgs& ta, int64_t count, int window, int interlaced, float* m1, float* m2, int N,
                        const double* fix, const float* r1, const float* r2, const double* alpha, cudaStream_t s) {
  if (window == PSPEC_WINDOW_CIC) {
    if (interlaced)
      ptile_paint_v<PSPEC_WINDOW_CIC, true>(ta, count, m1, m2, N, fix, r1, r2, alpha, s);
    else
      ptile_paint_v<PSPEC_WINDOW_CIC, false>(ta, count, m1, m2, N, fix, r1, r2, alpha, s);
  } else {
    if (interlaced)
      ptile_paint_v<PSPEC_WINDOW_TSC, true>(ta, count, m1, m2, N, fix, r1, r2, alpha, s);
    else
      ptile_paint_v<PSPEC_WINDOW_TSC, false>(ta, count, m1, m2, N, fix, r1, r2, alpha, s);
  }
}

// ------------------------------------------------------------------ batched mocks
// rsums = (W_r, S_r, I_r, fixed-point scale of the randoms mesh painted alone) of the cached randoms.
__global__ void __launch_bounds__(kFinalThreads) k_randoms_sums(const double* pr, int nbr, double* rsums) {
  __shared__ double sum[8];
  all_column_sums(pr, 0, pr, nbr, sum);
  if (threadIdx.x != 0) return;
  rsums[0] = sum[4];
  rsums[1] = sum[5];
  rsums[2] = sum[6];
  rsums[3] = fix_scale(sum[7]);
}

__global__ void __launch_bounds__(kFinalThreads) k_catalog_final_cached(const double* pd, int nbd,
                                                                        const double* __restrict__ rsums, double* d) {
  __shared__ double sum[8];
  all_column_sums(pd, nbd, pd, 0, sum);
  if (threadIdx.x != 0) return;
  const double wd = sum[0], sd = sum[1], ad = sum[3];
  const double Wr = rsums[0], Sr = rsums[1], Ir = rsums[2];
  const double alpha = wd / Wr;
  d[D_WD] = wd;
  d[D_WR] = Wr;
  d[D_ALPHA] = alpha;
  d[D_I] = alpha * Ir;
  d[D_S] = sd + alpha * alpha * Sr;
  d[D_NONFINITE] = 0.0;
  d[D_WRAPPED] = 0.0;
  d[D_SD] = sd;
  d[D_SR] = Sr;
  d[D_IR] = Ir;
  d[D_FIX] = fix_scale(ad);  // the mock's data mesh is painted alone
}

template <typename T>
__global__ void k_axpy_randoms(T* __restrict__ m, const T* __restrict__ r, int64_t n, const double* __restrict__ d) {
  const T a = (T)d[D_ALPHA];
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    m[i] -= a * r[i];
}

__global__ void k_batch_outputs(const double* __restrict__ P, int n, const double* __restrict__ d,
                                const int* __restrict__ cur, const BatchOut* __restrict__ bo) {
  const int c = *cur;
  double* P_all = bo->P_all;
  double* sums_all = bo->sums_all;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    P_all[(int64_t)c * n + i] = P[i];
  if (blockIdx.x == 0 && threadIdx.x == 0 && sums_all) {
    sums_all[4 * c + 0] = d[D_ALPHA];
    sums_all[4 * c + 1] = d[D_I];
    sums_all[4 * c + 2] = d[D_S];
    sums_all[4 * c + 3] = d[D_WD];
  }
}

__global__ void k_advance(int* cur) {
  if (threadIdx.x == 0 && blockIdx.x == 0) *cur += 1;
}

void launch_randoms_sums(const double* part_r, int nb_r, double* rsums, cudaStream_t s) {
  k_randoms_sums<<<1, kFinalThreads, 0, s>>>(part_r, nb_r, rsums);
}
void launch_catalog_final_cached(const double* part_d, int nb_d, const double* rsums, double* derived,
                                 cudaStream_t s) {
  k_catalog_final_cached<<<1, kFinalThreads, 0, s>>>(part_d, nb_d, rsums, derived);
}
void launch_axpy_randoms(float* mesh, const float* rmesh, int64_t n, const double* derived, cudaStream_t s) {
  k_axpy_randoms<float><<<2048, 256, 0, s>>>(mesh, rmesh, n, derived);
}
void launch_axpy_randoms(double* mesh, const double* rmesh, int64_t n, const double* derived, cudaStream_t s) {
  k_axpy_randoms<double><<<2048, 256, 0, s>>>(mesh, rmesh, n, derived);
}
void launch_batch_outputs(const double* P, int n_ells, int nk, const double* derived, const int* cur,
                          const BatchOut* out, cudaStream_t s) {
  k_batch_outputs<<<(n_ells * nk + 127) / 128, 128, 0, s>>>(P, n_ells * nk, derived, cur, out);
}
void launch_advance(int* cur, cudaStream_t s) { k_advance<<<1, 32, 0, s>>>(cur); }

// ------------------------------------------------------------------ a6: finalise
struct EllList {
  int n;
  int ell[PSPEC_MAX_ELL / 2 + 1];
};

__global__ void k_finalize(const double* __restrict__ bins, const double* __restrict__ nmodes_in,
                           const double* __restrict__ ksum, int nk, EllList el, const double* __restrict__ derived,
                           double* P, double* kmean, double* nmodes, int cart) {
  // row 0: n_modes and k_mean; row 1 + i: P of ell[i] (FP64 divisions are long chains: one or two per thread)
  const int b = blockIdx.x * blockDim.x + threadIdx.x, i = (int)blockIdx.y - 1;
  if (b >= nk) return;
  const double n = nmodes_in[b];
  const double nan = __longlong_as_double(0x7ff8000000000000ULL);
  if (i < 0) {
    nmodes[b] = n;
    kmean[b] = n > 0.0 ? ksum[b] / n : nan;
    return;
  }
  const double I = derived[D_I], S = derived[D_S];
  const int ell = el.ell[i];
  double v;
  const double B0 = bins[SLOT_P0 * nk + b];
  if (ell == 0)
    v = (B0 / n - S) / I;
  else if (!cart)
    v = 4.0 * M_PI * bins[(SLOT_ELL0 + i) * nk + b] / (I * n);
  else {
    // Cartesian: A2, A4 = sum mult (khat . rhat)^2, ^4 terms; L_2 = (3mu^2-1)/2, L_4 = (35mu^4-30mu^2+3)/8
    const double A2 = bins[SLOT_ELL0 * nk + b], A4 = bins[(SLOT_ELL0 + 1) * nk + b];
    v = ell == 2 ? 2.5 * (3.0 * A2 - B0) / (I * n) : 1.125 * (35.0 * A4 - 30.0 * A2 + 3.0 * B0) / (I * n);
  }
  P[(int64_t)i * nk + b] = n > 0.0 ? v : nan;
}

void launch_finalize(const double* bins, const double* nmodes_in, const double* ksum, int nk, const int32_t* ells,
                     int n_ells, const double* derived, double* P, double* k_mean, double* n_modes, cudaStream_t s,
                     int cartesian) {
  EllList el;
  el.n = n_ells;
  for (int i = 0; i < n_ells; i++) el.ell[i] = ells[i];
  k_finalize<<<dim3((nk + 127) / 128, n_ells + 1), 128, 0, s>>>(bins, nmodes_in, ksum, nk, el, derived, P, k_mean, n_modes, cartesian);
}

// ------------------------------------------------------------------ a7: wedges
__global__ void k_wedges(const double* __restrict__ P, int n_ells, int nk, int n_mu, WedgeTab t, double* out) {
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= n_mu * nk) return;
  const int w = idx / nk, b = idx - w * nk;
  double s = 0.0;
  for (int i = 0; i < n_ells; i++) s += P[(int64_t)i * nk + b] * t.lbar[i * n_mu + w];
  out[idx] = s;
}

void launch_wedges(const double* P, int n_ells, int nk, int n_mu, const WedgeTab& t, double* out, cudaStream_t s) {
  const int n = n_mu * nk;
  if (n <= 0) return;
  k_wedges<<<(n + 127) / 128, 128, 0, s>>>(P, n_ells, nk, n_mu, t, out);
}

}  // namespace pspec
