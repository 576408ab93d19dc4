// FP64 collision of a node near equilibrium (max |x_i| <= 1/48, or 1/32
// where alpha is rounded to FP32) without logarithms, for FP64 storage and
// the ROOT / SECANT modes.
//
// What bounds it: GB300 issues one FP64 warp instruction per 64 cycles on
// each SM sub-partition, against one FP32 or integer instruction per cycle.
// The literal evaluation of Eqs. (4), (8) and (9) (node_fp64.cuh) takes
// ~2,400 FP64 instructions for a D3Q27 FORMULA node, nearly all of them the
// logarithms and divisions of the entropy change, and ~17,000 for ROOT.
// Here FP64 keeps what has to carry 53 bits -- moments, equilibrium,
// n_i = f^eq_i - f_i and the relaxation, ~120 instructions per D3Q27 node --
// the moments' sums run in 64-bit integers, and the entropy change moves to
// double-float FP32 (df32.cuh).
//
// Why that loses nothing: alpha = 2 + O(x) enters f + alpha beta n through
// n = f x, so an error d(alpha) moves f by a fraction x d(alpha) of itself.
// Delta H(alpha) = sum_k c_k(alpha) M_k, M_k = sum_i n_i x_i^(k-1),
// c_k(alpha) = (-1)^k (alpha^k - k alpha) / (k (k-1)), has no k = 2 term at
// alpha = 2, so Delta H(2) is formed from its own leading term M_3 instead
// of as the difference of two O(x^2) sums: with x_i and M_2..M_6 in
// double-float (relative error ~2^-44) and M_7..M_14 in FP32, Delta H(2) is
// off by ~1e-13 x^3 rho plus 2e-7 x^7 rho, against ~1e-16 x^2 rho of the
// logarithm form.  The range ends where the second term reaches that.
// Measured against 160 bits over max |x| = 1e-11 .. 0.024, 320 states per
// lattice: alpha off by at most 8.5e-16 (D2Q9) and 7.7e-16 (D3Q27), the
// logarithm form's by 1.8e-15 and 3.0e-15; the new populations by 1.1e-15
// and 1.3e-15 of f, the logarithm form's by 1.1e-15 and 1.8e-15.  At 1/32
// alpha would be off by 1.1e-14.  The series is cut after k = 14:
// 2^15 x^15 / 210 < 3e-20 x^2 at x = 1/48.
//
// Numbers are scaled by powers of two before they become FP32 (n_i by that
// of max |n_i|, f_i by that of max f_i), so nothing under- or overflows.
// Conversions between FP64 and FP32 are integer shifts: the conversion
// instructions issue on the FP64 pipe.
//
// Nodes outside the range (|x_i| too large, |u_a| >= 1/4, f_i below 2^-12 of
// the largest, every |n_i| below 2^-42 of it, invalid states) report false
// and take the logarithm path.
#pragma once
#include "df32.cuh"
#include "fp16_storage.cuh"
#include "node_fp32.cuh"
#include "node_fp64.cuh"

namespace elbm {

constexpr int kSeriesTop = 14;             // last moment of the series
// Largest |x_i| it takes.  Where alpha is rounded to FP32 afterwards (FP32 /
// FP16 storage) an error of 1e-14 does not matter and the range is wider, as
// the fixup's open nodes between the two would cost a logarithm form each
// (189 x 107 x 83, 20 steps: 2.95 ms with 1/48, 2.85 with 1/32).
constexpr float kSeriesXMax = 1.0f / 48.0f;
constexpr float kSeriesXMaxRounded = 1.0f / 32.0f;
// Exponent of max |n_i| over that of max f_i below which f^eq == f to within
// the rounding of either form: whether a node counts as degenerate, and the
// sign of Delta H(2) ~ x M_2 / 3 against the logarithm form's 1.1e-14 M_2,
// are then decided by rounding, and the logarithm form (max |n_i| up to 27
// times 20 ulp of the largest f_i at a node it finds degenerate) keeps that
// decision.  Only states at equilibrium get there: the first step after
// initialisation, a fluid at rest.
constexpr int kSeriesNMin = -42;

// (double)v for normal or zero v, by shifting the exponent and mantissa
__device__ __forceinline__ double f2d(float v) {
  const unsigned b = __float_as_uint(v);
  const unsigned a = b & 0x7fffffffu;
  const unsigned hi = a < 0x00800000u
                          ? 0u
                          : ((b & 0x80000000u) | ((a >> 3) + (896u << 20)));
  return __hiloint2double((int)hi, (int)(a < 0x00800000u ? 0u : b << 29));
}

// v truncated to FP32; 0 below the FP32 range, callers stay under its top
__device__ __forceinline__ float d2f_trunc(double v) {
  const int h = __double2hiint(v);
  const int a = (h & 0x7fffffff) - (896 << 20);
  const unsigned m = __funnelshift_l((unsigned)__double2loint(v), (unsigned)a, 3);
  return a < (1 << 20) ? 0.0f
                       : __uint_as_float(m | ((unsigned)h & 0x80000000u));
}

// v 2^-(adj >> 20) as hi + lo: hi the upper 24 bits, lo the next 23 (the
// shift moves the FP64 exponent bias to FP32's as well).  Values that
// would leave lo below the FP32 range count as zero; they are 2^-100 of
// the largest of their kind.
__device__ __forceinline__ DF<float> split_df(double v, int adj) {
  const int h = __double2hiint(v);
  const unsigned l = (unsigned)__double2loint(v);
  const int a = (h & 0x7fffffff) - adj;
  const unsigned s = (unsigned)h & 0x80000000u;
  const unsigned hb = __funnelshift_l(l, (unsigned)a, 3) | s;
  // lo = 2^(E-23) 0.m with m the 29 bits that did not fit (23 kept)
  const unsigned base = (hb & 0xff800000u) - (23u << 23);
  const float lo =
      __uint_as_float(base | ((l & 0x1fffffffu) >> 6)) - __uint_as_float(base);
  const bool in = a >= (25 << 20);
  return {in ? __uint_as_float(hb) : 0.0f, in ? lo : 0.0f};
}

// Stored value of population i as FP64.
template <class L, class T>
__device__ __forceinline__ double load64(T v, int i, double rho0,
                                         bool unshifted) {
  if constexpr (sizeof(T) == 8) {
    return v;
  } else if constexpr (sizeof(T) == 2) {
    return fma(L::w(i), rho0, f2d(__half2float(v) * L::hscale_inv(i)));
  } else {
    const double d = f2d(v);
    return unshifted ? d : fma(L::w(i), rho0, d);
  }
}

__host__ __device__ constexpr double pow6(int d) {
  return d == 0 ? 1.0 : 6.0 * pow6(d - 1);
}

// Population with velocity (cx, cy, cz).
template <class L>
__host__ __device__ constexpr int pop_index(int cx, int cy, int cz) {
  for (int i = 0; i < L::Q; ++i)
    if (L::c(i, 0) == cx && L::c(i, 1) == cy && L::c(i, 2) == cz) return i;
  return 0;
}

// Moments of x_i scaled by powers of two: sum_i n_i x_i^(k-1) = en d^(k-1)
// m[k] with en, d powers of two.
struct Series64 {
  DF<float> m[7];               // k = 2..6
  float t[kSeriesTop + 1];      // k = 7..kSeriesTop
  int e_n, e_d;                 // en = 2^e_n, d = 2^e_d
};

// 1 / y for positive normal y with a normal reciprocal: PTX's approximate
// reciprocal r and one step of Householder's third-order iteration for 1 / y
// (A. S. Householder, The Numerical Treatment of a Single Nonlinear Equation,
// 1970), r (1 + e + e^2) with e = 1 - y r.  |e| <= 2^-19 leaves e^3 < 2^-57 and
// one rounding of the result: within an ulp of 1 / y (tests/test_gpu_rcp64.py),
// 3 FP64 instructions where a division takes about 10.
__device__ __forceinline__ double rcp64(double y) {
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(y));
  const double e = fma(-y, r, 1.0);
  return fma(r, fma(e, e, e), r);
}

// A positive FP64 value as a 64-bit integer in units of 2^(e - 62), e + 1 =
// top >> 20 its biased reference exponent (v < 2^(e + 1)); bits below the
// unit are dropped.
__device__ __forceinline__ long long to_fixed(double v, int top) {
  const unsigned h = (unsigned)__double2hiint(v);
  const unsigned l = (unsigned)__double2loint(v);
  const unsigned mh = __funnelshift_l(l, h, 11) | 0x80000000u, ml = l << 11;
  const unsigned sh = (unsigned)(top - (int)h) >> 20;   // < 32 (range check)
  const unsigned lo = __funnelshift_r(ml, mh, sh), hi = mh >> sh;
  return (long long)(((unsigned long long)hi << 32) | lo);
}
// (double)v, rounded once: (2^84 + 2^63 + upper half) - (2^84 + 2^63 + 2^52)
// is exact, and the sum with 2^52 + lower half is the one rounding
__device__ __forceinline__ double from_fixed(long long v) {
  const unsigned hi = (unsigned)((unsigned long long)v >> 32) ^ 0x80000000u;
  const double dh = __hiloint2double(0x45300000, (int)hi) -
                    __hiloint2double(0x45300000, (int)0x80100000);
  return dh + __hiloint2double(0x43300000, (int)(unsigned)v);
}

template <class L>
struct Near64 {
  double f[L::Q];
  double n[L::Q];               // f^eq_i - f_i
  double rho, inv_rho;          // in units of `unit`
  double j[3];
  double unit;
};

// 3u and s = sqrt(1 + 3u^2) - 1 of one axis; false: |u| >= kUMax32.  One
// Newton step on s^2 + 2s - 3u^2 = 0 from the FP32 value, whose relative error
// (< 2^-20) the step squares; the reciprocal of its slope is refined once.
__device__ __forceinline__ bool axis_near(double u, double& u3, double& sv) {
  u3 = 3.0 * u;
  const float uf = d2f_trunc(u);
  const float yf = fmaf(3.0f * uf, uf, 1.0f);
  const float s0f = 3.0f * uf * uf * rcp_approx(1.0f + yf * rsqrt_approx(yf));
  const double s0 = f2d(s0f);
  const double rs = f2d(rcp_approx(fmaf(2.0f, s0f, 2.0f)));
  const double g = fma(s0, s0 + 2.0, -u3 * u);
  const double ri = fma(rs, fma(-fma(2.0, s0, 2.0), rs, 1.0), rs);
  sv = fma(-g, ri, s0);
  return fabsf(uf) < kUMax32;
}

// Moments, n_i and the scaled x moments of a node whose f[] is filled.
// False: the node is outside the series' range, max |x_i| <= xmax.
template <class L>
__device__ __forceinline__ bool near64_prepare(Near64<L>& s, Series64& r,
                                               float xmax) {
  constexpr int Z = L::D == 3 ? 1 : 0;
  int fmin = 0x7fffffff, fmax = (int)0x80000000;
#pragma unroll
  for (int i = 0; i < L::Q; ++i) {
    const int h = __double2hiint(s.f[i]);
    fmin = min(fmin, h);
    fmax = max(fmax, h);
  }
  // every f_i within [2^-12, 1] of the largest and far from the ends of
  // the FP64 range (also excludes f <= 0, NaN, inf)
  if (fmin < (200 << 20) || fmax > (1800 << 20)) return false;
  const int rexp = (fmax & 0x7ff00000) + (3 << 20);
  if (fmin < rexp - (15 << 20)) return false;
  // Mass and momentum in 64-bit integers: exact but for the bits of a
  // population below 2^-59 of the largest one's power of two (27 of them stay
  // below half an ulp of the mass), and off the FP64 pipe (49 additions for
  // D3Q27).  Within the series' range f_0 >= 0.2 rho, so rho
  // stays below 2^4 of the largest f_i's power of two; a node for which it
  // does not overflows, and its f^eq then differs from f far beyond xmax.
  const int top = rexp + (1 << 20) + 0xfffff;
  long long jx = 0, jy = 0;
  long long sy[3];
#pragma unroll
  for (int cz = -Z; cz <= Z; ++cz) {
    long long sx[3];
#pragma unroll
    for (int cy = -1; cy <= 1; ++cy) {
      const long long p = to_fixed(s.f[pop_index<L>(1, cy, cz)], top);
      const long long m = to_fixed(s.f[pop_index<L>(-1, cy, cz)], top);
      jx += p - m;
      sx[cy + 1] = (p + m) + to_fixed(s.f[pop_index<L>(0, cy, cz)], top);
    }
    jy += sx[2] - sx[0];
    sy[cz + 1] = (sx[2] + sx[0]) + sx[1];
  }
  const double rho =
      from_fixed(Z ? (sy[2] + sy[0]) + sy[1] : sy[1]);
  s.rho = rho;
  s.j[0] = from_fixed(jx);
  s.j[1] = from_fixed(jy);
  s.j[2] = Z ? from_fixed(sy[2] - sy[0]) : 0.0;
  s.unit = __hiloint2double(rexp - (62 << 20), 0);
  if (!(__double2hiint(rho) >= (1023 << 20))) return false;
  s.inv_rho = rcp64(rho);
  // rho / 6^D; the factors below carry weights 4 (rest) and 1 per axis,
  // which are exact
  constexpr double k6i = 1.0 / pow6(L::D);
  const double r6 =
      rho * __hiloint2double(__double2hiint(k6i) + rexp - ((62 + 1023) << 20),
                             __double2loint(k6i));

  double psi[3][3];
  bool slow = false;
#pragma unroll
  for (int a = 0; a < L::D; ++a) {
    double u3, sv;
    slow = !axis_near(s.j[a] * s.inv_rho, u3, sv) || slow;
    const double b = fma(2.0, sv, 1.0);
    psi[a][2] = b + u3;
    psi[a][0] = b - u3;
    psi[a][1] = fma(-4.0, sv, 4.0);
  }
  if (slow) return false;
  int nmax = 0;
#pragma unroll
  for (int cx = -1; cx <= 1; ++cx) {
    const double px = r6 * psi[0][cx + 1];
#pragma unroll
    for (int cy = -1; cy <= 1; ++cy) {
      if (Z == 0) {
        const int i = pop_index<L>(cx, cy, 0);
        s.n[i] = fma(px, psi[1][cy + 1], -s.f[i]);
        nmax = max(nmax, __double2hiint(s.n[i]) & 0x7fffffff);
      } else {
        const double pxy = px * psi[1][cy + 1];
#pragma unroll
        for (int cz = -1; cz <= 1; ++cz) {
          const int i = pop_index<L>(cx, cy, cz);
          s.n[i] = fma(pxy, psi[2][cz + 1], -s.f[i]);
          nmax = max(nmax, __double2hiint(s.n[i]) & 0x7fffffff);
        }
      }
    }
  }
  // n_i scaled to at most 2^-5, so that |n_i / f_i| <= 2^5 and typically
  // ~2^-4: the products up to k = 14 stay inside the FP32 range
  const int nexp = (nmax & 0x7ff00000) + (6 << 20);
  r.e_n = (nexp >> 20) - 1023;
  r.e_d = (nexp - rexp) >> 20;
  if (r.e_d < kSeriesNMin + 3) return false;
  const float d = __int_as_float((127 + r.e_d) << 23);

  const int adjn = nexp - (127 << 20), adjf = rexp - (127 << 20);
  constexpr int P = npairs<L>();
  DF<float2> m2, m3, m4, m5, m6;
  float2 tt[kSeriesTop + 1];
  float2 xm;
  m2 = m3 = m4 = m5 = m6 = DF<float2>{f2(0.0f), f2(0.0f)};
#pragma unroll
  for (int k = 7; k <= kSeriesTop; ++k) tt[k] = f2(0.0f);
  xm = f2(0.0f);
  auto accum = [](DF<float2>& m, const DF<float2>& v) {
    const DF<float2> t = two_sum(m.hi, v.hi);
    m.hi = t.hi;
    m.lo = add_(m.lo, add_(t.lo, v.lo));
  };
  // product by x kept as an unnormalised double-float (|lo| stays below
  // a few ulp of hi)
  auto times = [](const DF<float2>& v, const DF<float2>& x) {
    const float2 h = mul_(v.hi, x.hi);
    const float2 e = fma_(v.hi, x.hi, neg_(h));
    return DF<float2>{h, fma_(v.hi, x.lo, fma_(v.lo, x.hi, e))};
  };
#pragma unroll
  for (int k = 0; k <= P; ++k) {
    // populations 2k-1 and 2k in the two lanes; the rest population pairs
    // with a zero
    const int i0 = k == 0 ? 0 : 2 * k - 1, i1 = 2 * k;
    const DF<float> na = split_df(s.n[i0], adjn), fa = split_df(s.f[i0], adjf);
    DF<float> nb = {0.0f, 0.0f}, fb = {1.0f, 0.0f};
    if (k > 0) {
      nb = split_df(s.n[i1], adjn);
      fb = split_df(s.f[i1], adjf);
    }
    const DF<float2> n2 = df_pair(na, nb), ff = df_pair(fa, fb);
    // x = n / f: FP32 quotient and the corrected residual
    const float2 rf = rcp_approx2(ff.hi);
    DF<float2> x;
    x.hi = mul_(n2.hi, rf);
    {
      const float2 p = mul_(x.hi, ff.hi);
      const float2 pe = fma_(x.hi, ff.hi, neg_(p));
      const float2 res = fma_(neg_(x.hi), ff.lo,
                              add_(sub_(sub_(n2.hi, p), pe), n2.lo));
      x.lo = mul_(res, rf);
    }
    xm = make_float2(fmaxf(xm.x, fabsf(x.hi.x)), fmaxf(xm.y, fabsf(x.hi.y)));
    DF<float2> t = times(n2, x);
    accum(m2, t);
    t = times(t, x);
    accum(m3, t);
    t = times(t, x);
    accum(m4, t);
    t = times(t, x);
    accum(m5, t);
    t = times(t, x);
    accum(m6, t);
    float2 w = t.hi;
#pragma unroll
    for (int q = 7; q <= kSeriesTop; ++q) {
      w = mul_(w, x.hi);
      tt[q] = add_(tt[q], w);
    }
  }
  if (!(fmaxf(xm.x, xm.y) * d <= xmax)) return false;
  auto fold = [](const DF<float2>& m) {
    return df_add(fast_two_sum(m.hi.x, m.lo.x), fast_two_sum(m.hi.y, m.lo.y));
  };
  r.m[2] = fold(m2);
  r.m[3] = fold(m3);
  r.m[4] = fold(m4);
  r.m[5] = fold(m5);
  r.m[6] = fold(m6);
#pragma unroll
  for (int k = 7; k <= kSeriesTop; ++k) r.t[k] = tt[k].x + tt[k].y;
  return true;
}

// c_k(2) = (-1)^k (2^k - 2k) / (k (k-1)) and c_k(1) = (-1)^(k+1) / k.
__host__ __device__ constexpr double series_c2(int k) {
  double p = 1.0;
  for (int q = 0; q < k; ++q) p *= 2.0;
  return (k % 2 ? -1.0 : 1.0) * (p - 2.0 * k) / (k * (k - 1.0));
}
__host__ __device__ constexpr double series_c1(int k) {
  return (k % 2 ? 1.0 : -1.0) / k;
}

// sum_{k = K0}^{kSeriesTop} c_k m[k] d^(k-K0), Horner from the top: FP32
// above k = 6, double-float below.
template <int K0, bool TWO>
__device__ __forceinline__ DF<float> series_sum(const Series64& r, float d) {
  constexpr auto c = [](int k) { return TWO ? series_c2(k) : series_c1(k); };
  float t = 0.0f;
#pragma unroll
  for (int k = kSeriesTop; k >= 7; --k) t = fmaf(t, d, (float)c(k) * r.t[k]);
  DF<float> s = {t, 0.0f};
#pragma unroll
  for (int k = 6; k >= K0; --k) {
    const DF<float> ck = {df_hi(c(k)), df_lo(c(k))};
    // d is a power of two: exact
    s = df_add(DF<float>{s.hi * d, s.lo * d}, df_mul(r.m[k], ck));
  }
  return s;
}

// Eqs. (8)-(9) of a node within the series' range (alpha_max > 2 there).
__device__ __forceinline__ double alpha_formula_near(const Series64& r,
                                                     unsigned& flags) {
  const float d = __int_as_float((127 + r.e_d) << 23);
  // Delta H(2) = en d^2 b2, Delta H(1) = en d b1
  const DF<float> b2 = series_sum<3, true>(r, d);
  if (b2.hi <= 0.0f) {
    flags |= NF_ACCEPT_STAR | NF_ACCEPT_TWO;
    return 2.0;
  }
  flags |= NF_FORMULA;
  const DF<float> b1 = series_sum<2, false>(r, d);
  const DF<float> D2 = {b2.hi * d, b2.lo * d};
  const DF<float> den = df_add(D2, df_neg(b1));
  if (!(den.hi > 0.0f)) return 1.0;   // f == f^eq to rounding
  const DF<float> t = df_div(D2, den);
  return (2.0 - f2d(t.hi)) - f2d(t.lo);
}

// The FORMULA of a node the FP32 stages left open (FP32 / FP16 storage): the
// series decision, taken only where the logarithm form (node_fp64.cuh,
// warp64.cuh) takes the same branch, and alpha rounded down to FP32.  The
// logarithm form's Delta H(2) is off by less than 100 u M_2 = 1.1e-14 M_2
// (u = 2^-53; 27 terms f phi(2 x) of at most 2 f x^2, the products f x L,
// and x off by 20 u), the series' by less than 20 u M_2, so a value beyond
// 2^-45 M_2 has the same sign in both, and the two alphas differ by less
// than 1e-13.  False: out of the series' range or within that distance of
// zero -- the logarithm form decides.
template <class L>
__device__ __forceinline__ bool near64_formula(Near64<L>& s, double& alpha,
                                               unsigned& flags) {
  Series64 r;
  if (!near64_prepare(s, r, kSeriesXMaxRounded)) return false;
  const float d = __int_as_float((127 + r.e_d) << 23);
  const DF<float> b2 = series_sum<3, true>(r, d);
  if (!(fabsf(b2.hi) * d > 2.842170943040401e-14f * r.m[2].hi)) return false;
  alpha = (double)__double2float_rd(alpha_formula_near(r, flags));
  return true;
}

// Delta H(alpha) = alpha (sum_k A_k alpha^(k-1) - T) for alpha <= 4, with
// A_k = (-1)^k M_k / (k (k-1)), T = sum_k k A_k.  Everything is in units of
// en d (M_2 is of order d^0 then).  The terms k >= 7 are at most
// 2^7 x^5 / 42 of the leading one: FP32 carries them.
struct Poly64 {
  double A[7], T;
  float a[kSeriesTop + 1], Tf;
  double unit;

  // FP32 value of sum_k a_k alpha^(k-1) - T
  __device__ __forceinline__ float q32(float al) const {
    float v = a[kSeriesTop];
#pragma unroll
    for (int k = kSeriesTop - 1; k >= 2; --k) v = fmaf(v, al, a[k]);
    return fmaf(v, al, -Tf);
  }
  __device__ __forceinline__ double q64(double al) const {
    const float af = d2f_trunc(al);
    float v = a[kSeriesTop];
#pragma unroll
    for (int k = kSeriesTop - 1; k >= 7; --k) v = fmaf(v, af, a[k]);
    double w = f2d(v * af);
#pragma unroll
    for (int k = 6; k >= 2; --k) w = k == 6 ? w + A[k] : fma(w, al, A[k]);
    return fma(w, al, -T);
  }
  __device__ __forceinline__ double dH(double al) const {
    return al * (q64(al) * unit);
  }
};

__device__ __forceinline__ Poly64 poly_near(const Series64& r) {
  Poly64 p;
  float tf = 0.0f;
#pragma unroll
  for (int k = kSeriesTop; k >= 2; --k) {
    const float ck = (float)((k % 2 ? -1.0 : 1.0) / (k * (k - 1.0)));
    // d^(k-2); far below the FP32 range it multiplies terms that vanish
    // beside k = 2
    const float dk =
        __int_as_float((127 + max((k - 2) * r.e_d, -120)) << 23);
    p.a[k] = (k <= 6 ? r.m[k].hi : r.t[k]) * ck * dk;
    if (k >= 7) tf = fmaf((float)k, p.a[k], tf);
  }
  double T = f2d(tf);
  float Tf = tf;
#pragma unroll
  for (int k = 6; k >= 2; --k) {
    const double c = (k % 2 ? -1.0 : 1.0) / (k * (k - 1.0));
    const int e = max((k - 2) * r.e_d, -1000);
    const double cd = __hiloint2double(__double2hiint(c) + (e << 20),
                                       __double2loint(c));
    p.A[k] = (f2d(r.m[k].hi) + f2d(r.m[k].lo)) * cd;
    T = fma((double)k, p.A[k], T);
    Tf = fmaf((float)k, p.a[k], Tf);
  }
  p.T = T;
  p.Tf = Tf;
  p.unit = __hiloint2double((1023 + max(r.e_n + r.e_d, -1022)) << 20, 0);
  return p;
}

// Eq. (4) by bisection on [1, alpha_max], stop rule -1e-13 <= dH <= 0, as
// alpha_root64.  Delta H is convex, Delta H(0) = 0 and its minimum lies at
// alpha = 1, so it increases on the bracket.  Most of the ~45 midpoints are
// decided without FP64: beyond alpha = 4 Delta H is positive (|x| <= 1/32:
// Delta H(4) >= 2 M_2), and elsewhere the FP32 value decides when its
// distance from 0 and from the stop rule's -1e-13 exceeds its error
// (kErr M_2, a few hundred FP32 roundings).  The rest, at most log2 of the
// interval that leaves open over the stop interval (~10), takes the Taylor
// polynomial of the FP64 series about the FP32 root.
template <class L>
__device__ __forceinline__ double alpha_root_near(const Near64<L>& s,
                                                  const Series64& r,
                                                  unsigned& flags, int& iters) {
  constexpr float kErr = 3.0517578125e-05f;    // 2^-15
  constexpr float kTaylor = 6.103515625e-05f;  // 2^-14
  const Poly64 p = poly_near(r);
  double amax;
  {   // alpha_max = min over n_i < 0 of -f_i / n_i; the candidate is found
      // in FP32 and divided once in FP64
    double fb = 1.0, nb = 0.0;
    float best = 0.0f;
    const int adjn = (r.e_n + 1023 - 127) << 20;
    const int adjf = adjn - (r.e_d << 20);
#pragma unroll
    for (int i = 0; i < L::Q; ++i) {
      const float x = split_df(s.n[i], adjn).hi *
                      rcp_approx(split_df(s.f[i], adjf).hi);
      if (x < best) {
        best = x;
        fb = s.f[i];
        nb = s.n[i];
      }
    }
    if (best >= 0.0f) {   // no x_i < 0 resolved: f^eq == f
      flags |= NF_DEGENERATE;
      return 2.0;
    }
    amax = -fb / nb;
  }
  // FP32 root near 2, with the first two derivatives there
  float ar = 2.0f, q2 = 0.0f;
#pragma unroll
  for (int it = 0; it < 3; ++it) {
    float v = p.a[kSeriesTop], dv = 0.0f;
    q2 = 0.0f;
#pragma unroll
    for (int k = kSeriesTop - 1; k >= 2; --k) {
      q2 = fmaf(q2, ar, dv);
      dv = fmaf(dv, ar, v);
      v = fmaf(v, ar, p.a[k]);
    }
    q2 = fmaf(q2, ar, dv);   // half the second derivative
    dv = fmaf(dv, ar, v);
    v = fmaf(v, ar, -p.Tf);
    if (it < 2) ar -= __fdividef(v, dv);
  }
  ar = fminf(fmaxf(ar, 1.5f), 2.5f);
  // FP64 value and slope there
  const double ard = f2d(ar);
  double q0, q1;
  {
    float v = p.a[kSeriesTop], dv = 0.0f;
#pragma unroll
    for (int k = kSeriesTop - 1; k >= 7; --k) {
      dv = fmaf(dv, ar, v);
      v = fmaf(v, ar, p.a[k]);
    }
    double dw = f2d(dv), w = f2d(v);
#pragma unroll
    for (int k = 6; k >= 2; --k) {
      dw = fma(dw, ard, w);
      w = fma(w, ard, p.A[k]);
    }
    q1 = fma(dw, ard, w);
    q0 = fma(w, ard, -p.T);
  }
  // the stop rule in units of the polynomial (may overflow to inf: every
  // value <= 0 stops then)
  const float uf = __int_as_float(
      (127 + min(max(r.e_n + r.e_d, -120), 120)) << 23);
  const float tol = __fdividef(1e-13f, uf);
  const float err = kErr * fabsf(r.m[2].hi);
  double lo = 1.0, hi = amax;
  for (int k = 0; k < kRootMaxIters; ++k) {
    const double mid = 0.5 * (lo + hi);
    ++iters;
    bool up = true;
    // positive FP64 values order like their bits
    if (__double2hiint(mid) < 0x40100000) {
      const float mf = d2f_trunc(mid);
      const float q = p.q32(mf);
      const float tl = __fdividef(tol, mf);   // rule: -tl <= q <= 0
      if (q > err) {
        up = true;
      } else if (q < -tl - err) {
        up = false;
      } else if (q < -err && q > err - tl) {
        return mid;
      } else {
        double d;
        if (fabsf(mf - ar) < kTaylor) {
          const double h = mid - ard;
          d = mid * (fma(h, fma(h, f2d(q2), q1), q0) * p.unit);
        } else {
          d = p.dH(mid);
        }
        if (d >= -kRootTol && d <= 0.0) return mid;
        up = d > 0.0;
      }
    }
    if (up)
      hi = mid;
    else
      lo = mid;
    // hi - lo < 1e-15 hi needs hi and lo within 9 ulp
    const long long ulps = __double_as_longlong(hi) - __double_as_longlong(lo);
    if (ulps < 16 && hi - lo < 1e-15 * hi) return lo;
  }
  flags |= NF_ROOT_CAP;
  return lo;
}

// Modified secant iteration, as alpha_secant64.
__device__ __forceinline__ double alpha_secant_near(const Series64& r,
                                                    int n_iter, unsigned& flags,
                                                    int& iters) {
  const float d = __int_as_float((127 + r.e_d) << 23);
  const DF<float> b2 = series_sum<3, true>(r, d);
  if (b2.hi <= 0.0f) {
    flags |= NF_ACCEPT_STAR | NF_ACCEPT_TWO;
    return 2.0;
  }
  flags |= NF_FORMULA;
  const DF<float> b1 = series_sum<2, false>(r, d);
  const Poly64 p = poly_near(r);
  const double Dstar = p.unit * (f2d(b2.hi * d) + f2d(b2.lo * d));
  const double D1 = p.unit * (f2d(b1.hi) + f2d(b1.lo));
  if (!(Dstar - D1 > 0.0)) return 1.0;
  double a = 1.0, da = D1;
  for (int k = 0; k < n_iter; ++k) {
    const double an = 2.0 + Dstar / (Dstar - da) * (a - 2.0);
    const double dn = p.dH(an);
    ++iters;
    if (dn > 0.0) break;
    a = an;
    da = dn;
    if (da >= -kRootTol) break;
  }
  return a;
}

}  // namespace elbm
