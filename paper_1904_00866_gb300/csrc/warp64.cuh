// FP64 FORMULA of one node computed by a whole warp (FP32 / FP16 storage
// fixups), with logarithms and, near equilibrium, by the series
// (near64_warp): lane i < Q holds population i, so each lane evaluates one
// population's equilibrium factor, division and logarithms, and the sums
// over i are warp reductions.
//
// GB300 issues one FP64 warp instruction per ~64 cycles on each SM
// sub-partition.  A node collided on one lane (node64_prepare +
// alpha_formula64: ~2,400 FP64 instructions for D3Q27, most of them the 27
// divisions and logarithms) therefore holds its warp for ~75 us, and a
// fixup with a few thousand such nodes ends ~0.2 ms after its last node
// started, however they are spread.  Spread over the lanes the node takes
// ~460 FP64 warp instructions (divisions, logarithms and the reductions)
// and so ends ~6x sooner; in bulk, one node per lane costs fewer FP64
// instructions per node (~75), which the fixups use on long queues.
//
// The arithmetic is that of node64_prepare and alpha_formula64 (Eq. (8),
// the acceptance test after it, Eq. (9)), population by population; only
// the order of the sums over i differs (pairwise over the lanes), which
// moves Delta H by rounding only.
#pragma once
#include "node_fp64.cuh"
#include "series64.cuh"

namespace elbm {

// Velocity, weight and binary16 scale of the population a lane holds.
struct LanePop {
  int c[3];
  double w;
  float hscale, hscale_inv;
  bool on;   // lane < Q
};

template <class L>
__device__ __forceinline__ LanePop lane_pop(int lane) {
  LanePop r{{0, 0, 0}, 0.0, 1.0f, 1.0f, lane < L::Q};
#pragma unroll
  for (int q = 0; q < L::Q; ++q)
    if (q == lane) {
      r.c[0] = L::c(q, 0);
      r.c[1] = L::c(q, 1);
      r.c[2] = L::c(q, 2);
      r.w = L::w(q);
      r.hscale = L::hscale(q);
      r.hscale_inv = L::hscale_inv(q);
    }
  return r;
}

__device__ __forceinline__ double warp_sum64(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

__device__ __forceinline__ double warp_min64(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
    v = fmin(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// Result of formula64_warp (the same on every lane).
struct Warp64 {
  double rho, j[3], alpha;
  unsigned flags;   // NF_ACCEPT_* / NF_FORMULA, or NF_BAD_* (state invalid)
};

// All 32 lanes call this with f = f_i on lane i < Q (anything on the other
// lanes).  Writes the post-collision population of the lane through
// store(value) (lanes < Q only): f + alpha beta (f^eq - f), alpha rounded
// down to FP32 (the FP32 storage paths' convention), or f unchanged when
// the state is invalid.
template <class L, class Store>
__device__ __forceinline__ Warp64 formula64_warp(const LanePop& lp, double f,
                                                 double beta, Store store) {
  Warp64 r;
  r.flags = 0;
  const double fi = lp.on ? f : 0.0;
  if (__any_sync(0xffffffffu, lp.on && !(f > 0.0))) r.flags |= NF_BAD_NEG;
  r.rho = warp_sum64(fi);
  double u[3] = {0.0, 0.0, 0.0}, dp[3], dm[3], d0[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    r.j[a] = a < L::D ? warp_sum64((double)lp.c[a] * fi) : 0.0;
    if (a >= L::D) continue;
    u[a] = r.j[a] / r.rho;
    if (!(fabs(u[a]) < 1.0)) r.flags |= NF_BAD_NONFINITE;
    const double sg = 3.0 * u[a] * u[a] / (1.0 + sqrt(1.0 + 3.0 * u[a] * u[a]));
    dp[a] = 3.0 * u[a] + 2.0 * sg;
    dm[a] = -3.0 * u[a] + 2.0 * sg;
    d0[a] = -sg;
  }
  if (!(r.rho > 0.0) || !isfinite(r.rho)) r.flags |= NF_BAD_NONFINITE;
  r.alpha = 1.0;
  if (r.flags) {
    if (lp.on) store(f);
    return r;
  }
  double P = r.rho * lp.w;
#pragma unroll
  for (int a = 0; a < L::D; ++a) {
    const int ca = lp.c[a];
    P *= 1.0 + (ca == 1 ? dp[a] : (ca == -1 ? dm[a] : d0[a]));
  }
  const double x = lp.on ? (P - f) / f : 0.0;
  const double amax = warp_min64(x < 0.0 ? -1.0 / x : INFINITY);
  const double astar = fmin(2.0, amax);
  const double Li = log1p(x);
  const double B = warp_sum64(fi * x * Li);
  const double D1 = warp_sum64(fi * (Li - x));
  const double Dstar = warp_sum64(fi * phi64(astar * x)) - astar * B;
  double alpha;
  if (Dstar <= 0.0) {
    r.flags |= NF_ACCEPT_STAR;
    if (astar == 2.0) r.flags |= NF_ACCEPT_TWO;
    alpha = astar;
  } else {
    r.flags |= NF_FORMULA;
    alpha = Dstar - D1 > 0.0 ? astar + Dstar / (Dstar - D1) * (1.0 - astar)
                             : 1.0;
  }
  alpha = (double)__double2float_rd(alpha);
  r.alpha = alpha;
  if (lp.on) store(fma(alpha * beta, f * x, f));
  return r;
}

// Warp sums of a 62-bit non-negative integer v (0 on idle lanes) times
// c[] and of v itself: three 22-bit pieces, each summed by one 32-bit
// reduction.
__device__ __forceinline__ long long warp_sum_fixed(long long v, int c) {
  const int a = c * (int)(v & 0x3fffff), b = c * (int)((v >> 22) & 0x3fffff),
            d = c * (int)(v >> 44);
  const long long sa = __reduce_add_sync(0xffffffffu, a);
  const long long sb = __reduce_add_sync(0xffffffffu, b);
  const long long sd = __reduce_add_sync(0xffffffffu, d);
  return sa + sb * (1LL << 22) + sd * (1LL << 44);
}

// near64_formula of one node by the whole warp, one population per lane
// (f = f_i on lane i < Q): the same moments in 64-bit integers, the same
// n_i and double-float x_i; each lane sums its own series terms
// (Delta H(2) = sum_i n_i x_i^2 P2(x_i), Delta H(1) = sum_i n_i x_i P1(x_i))
// and three sums cross the warp.
//
// Why: a short list of nodes is bound by the time to fetch the code once.
// The one-node-per-lane form is a straight line of thousands of
// instructions (27 populations unrolled) that a warp runs a single time:
// ~25 us for D3Q27 whether it holds 1 node or 32.  This form is a tenth of
// that code and ~55 FP64 instructions (64 cycles each) per node, against
// ~460 of the logarithm form.
//
// True: settled, the lane's new population stored through store(value).
template <class L, class Store>
__device__ __forceinline__ bool near64_warp(const LanePop& lp, int lane,
                                            double f, double beta, Warp64& r,
                                            Store store) {
  constexpr unsigned kAll = 0xffffffffu;
  const int fh = __double2hiint(f);
  const int fmin = __reduce_min_sync(kAll, lp.on ? fh : 0x7fffffff);
  const int fmax = __reduce_max_sync(kAll, lp.on ? fh : (int)0x80000000);
  if (fmin < (200 << 20) || fmax > (1800 << 20)) return false;
  const int rexp = (fmax & 0x7ff00000) + (3 << 20);
  if (fmin < rexp - (15 << 20)) return false;
  const int top = rexp + (1 << 20) + 0xfffff;
  const long long v = lp.on ? to_fixed(f, top) : 0;
  const double rho = from_fixed(warp_sum_fixed(v, 1));
  if (!(__double2hiint(rho) >= (1023 << 20))) return false;
  // lane a (mod 3) works on axis a
  const long long jx = warp_sum_fixed(v, lp.c[0]),
                  jy = warp_sum_fixed(v, lp.c[1]),
                  jz = L::D == 3 ? warp_sum_fixed(v, lp.c[2]) : 0;
  const int ax = lane % 3;
  const double j = from_fixed(ax == 0 ? jx : (ax == 1 ? jy : jz));
  const double inv_rho = rcp64(rho);
  double u3, sv;
  if (__any_sync(kAll, !axis_near(j * inv_rho, u3, sv))) return false;
  constexpr double k6i = 1.0 / pow6(L::D);
  double P = rho * __hiloint2double(
                       __double2hiint(k6i) + rexp - ((62 + 1023) << 20),
                       __double2loint(k6i));
#pragma unroll
  for (int a = 0; a < L::D; ++a) {
    const double sa = __shfl_sync(kAll, sv, a), ua = __shfl_sync(kAll, u3, a);
    const int c = lp.c[a];
    P *= c == 0 ? fma(-4.0, sa, 4.0) : fma((double)c, ua, fma(2.0, sa, 1.0));
  }
  const double n = P - f;
  const int nmax = __reduce_max_sync(
      kAll, lp.on ? __double2hiint(n) & 0x7fffffff : 0);
  const int nexp = (nmax & 0x7ff00000) + (6 << 20);
  const int e_d = (nexp - rexp) >> 20;
  if (e_d < kSeriesNMin + 3) return false;
  const float d = __int_as_float((127 + e_d) << 23);
  // this lane's x (in units of d) and series terms; idle lanes add zeros
  const DF<float> zero = {0.0f, 0.0f}, one = {1.0f, 0.0f};
  const DF<float> nn = lp.on ? split_df(n, nexp - (127 << 20)) : zero;
  const DF<float> ff = lp.on ? split_df(f, rexp - (127 << 20)) : one;
  const DF<float> x = df_div(nn, ff);
  const int xm = __reduce_max_sync(kAll, __float_as_int(fabsf(x.hi)));
  if (!(__int_as_float(xm) * d <= kSeriesXMaxRounded)) return false;
  const DF<float> y = {x.hi * d, x.lo * d};   // exact
  float t2 = 0.0f, t1 = 0.0f;
#pragma unroll
  for (int k = kSeriesTop; k >= 7; --k) {
    t2 = fmaf(t2, y.hi, (float)series_c2(k));
    t1 = fmaf(t1, y.hi, (float)series_c1(k));
  }
  DF<float> p2 = {t2, 0.0f}, p1 = {t1, 0.0f};
#pragma unroll
  for (int k = 6; k >= 2; --k) {
    if (k >= 3)
      p2 = df_add(df_mul(p2, y),
                  DF<float>{df_hi(series_c2(k)), df_lo(series_c2(k))});
    p1 = df_add(df_mul(p1, y),
                DF<float>{df_hi(series_c1(k)), df_lo(series_c1(k))});
  }
  const DF<float> m2 = df_mul(nn, x), m3 = df_mul(m2, x);
  const DF<float> b2 = df_mul(m3, p2), b1 = df_mul(m2, p1);
  // sums of b2 d, b1 and m2 (units en d) over the lanes, FP64, halving the
  // set at the first two exchanges
  double s[4] = {f2d(b2.hi * d) + f2d(b2.lo * d), f2d(b1.hi) + f2d(b1.lo),
                 f2d(m2.hi), 0.0};
#pragma unroll
  for (int half = 2, o = 16; half >= 1; half >>= 1, o >>= 1) {
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int k = 0; k < half; ++k) {
      const double send = up ? s[k] : s[k + half];
      const double keep = up ? s[k + half] : s[k];
      s[k] = keep + __shfl_xor_sync(kAll, send, o);
    }
  }
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) s[0] += __shfl_xor_sync(kAll, s[0], o);
  const double D2 = __shfl_sync(kAll, s[0], 0), D1 = __shfl_sync(kAll, s[0], 8),
               M2 = __shfl_sync(kAll, s[0], 16);
  if (!(fabs(D2) > 2.842170943040401e-14 * M2)) return false;
  double alpha = 2.0;
  r.flags = NF_BAND;
  if (D2 <= 0.0) {
    r.flags |= NF_ACCEPT_STAR | NF_ACCEPT_TWO;
  } else {
    r.flags |= NF_FORMULA;
    const double den = D2 - D1, ri = rcp64(den);
    const double q = D2 * ri;
    alpha = 2.0 - fma(fma(-q, den, D2), ri, q);
  }
  alpha = (double)__double2float_rd(alpha);
  const double unit = __hiloint2double(rexp - (62 << 20), 0);
  r.alpha = alpha;
  r.rho = rho * unit;
  r.j[0] = __shfl_sync(kAll, j, 0) * unit;
  r.j[1] = __shfl_sync(kAll, j, 1) * unit;
  r.j[2] = L::D == 3 ? __shfl_sync(kAll, j, 2) * unit : 0.0;
  if (lp.on) store(fma(alpha * beta, n, f));
  return true;
}

}  // namespace elbm
