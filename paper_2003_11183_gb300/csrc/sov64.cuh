// The float64 step of eq. (2) and its tables.
//
// GB300 issues one float64 instruction of a warp in 16 cycles of its SM (two lanes a
// cycle), so a step is as long as the float64 instructions it takes: about 870 a
// variable when Phi, log Phi and Phi^-1 come from erfc, erfcx, log, exp and a refined
// rational start, their branches diverging within a warp.  Both functions are read here from
// tables of local polynomials of degree 8, in shared memory: a look-up of ten doubles at a
// lane's own place costs a few cycles, the polynomial eight FMAs, and the whole step about
// 40 float64 instructions on one path.  Measured with it, the spread of the samples' warps over the SMs and the
// products' padding left out: n = 256, 20 x 500 samples, tiles of 64: 7.21 -> 1.71 ms a solve; n = 4,096, 20 x 1,000,
// tiles of 64: 245 -> 67.4 ms; errors against 64-bit references no larger (1.3e-16 and 8.3e-16 of the logs).
//   A  Phi(-x) on [0, 13]: around x_j = j / 64, from the Taylor series (Hermite polynomials times
//      phi(x_j)) of degree 9 with its last term economised (Lanczos: replaced by its Chebyshev
//      remainder of 1.2e-17 relative);
//   B  Phi^-1(p) on (2^-41, 1/2]: 16 intervals an octave, around their midpoints, from the Taylor
//      series of degree 10 (the derivatives of Phi^-1 by the recurrence of G. Steinbrecher and W. T. Shaw,
//      Quantile mechanics, European J. Appl. Math. 19 (2008)), two terms economised.
// The leading coefficients, which carry the result's accuracy, are worked out in pairs of
// doubles (Phi(-x) by its power series below 4 and the continued fraction of the Mills ratio above;
// Phi^-1 by a Newton step on that), so that table values are rounded once.
#pragma once
#include "common.cuh"

namespace tlrmvn {

constexpr int T64_A = 833;             // entries of table A: x = 0, 1/64, ..., 13
constexpr int T64_OCT = 40;            // octaves of table B: [2^-41, 2^-40) up to [1/4, 1/2)
constexpr int T64_B = T64_OCT * 16;
constexpr int T64_W = 10;              // doubles an entry (nine coefficients and one spare: 16-byte loads)
constexpr int T64_DOUBLES = (T64_A + T64_B) * T64_W;

// ---- pairs of doubles (T. J. Dekker, Numer. Math. 18 (1971); products by FMA) ------------------------
struct DD {
  double h, l;
};
__device__ __forceinline__ DD dd_two_sum(double a, double b) {
  const double s = __dadd_rn(a, b), t = __dsub_rn(s, a);
  return DD{s, __dadd_rn(__dsub_rn(a, __dsub_rn(s, t)), __dsub_rn(b, t))};
}
__device__ __forceinline__ DD dd_fast(double a, double b) {  // |a| >= |b|
  const double s = __dadd_rn(a, b);
  return DD{s, __dsub_rn(b, __dsub_rn(s, a))};
}
__device__ __forceinline__ DD dd_add(DD a, DD b) {
  DD s = dd_two_sum(a.h, b.h);
  const DD t = dd_two_sum(a.l, b.l);
  s = dd_fast(s.h, __dadd_rn(s.l, t.h));
  return dd_fast(s.h, __dadd_rn(s.l, t.l));
}
__device__ __forceinline__ DD dd_mul(DD a, DD b) {
  const double p = __dmul_rn(a.h, b.h);
  const double e = __fma_rn(a.h, b.l, __fma_rn(a.l, b.h, __fma_rn(a.h, b.h, -p)));
  return dd_fast(p, e);
}
__device__ __forceinline__ DD dd_div(DD a, DD b) {
  const double q = __ddiv_rn(a.h, b.h);
  DD r = dd_mul(DD{-q, 0.0}, b);
  r = dd_add(a, r);
  return dd_fast(q, __ddiv_rn(r.h, b.h));
}
// exp(z) for z in [-100, 0]: z = k ln 2 + 64 s, the series of exp(s), squared six times
__device__ inline DD dd_exp(DD z) {
  const DD ln2{6.931471805599452862e-01, 2.319046813846299616e-17};
  const double k = rint(z.h * 1.4426950408889634);
  DD r = dd_add(z, dd_mul(DD{-k, 0.0}, ln2));
  r.h *= 0.015625;
  r.l *= 0.015625;
  DD s{1.0, 0.0};
  for (int n = 16; n >= 1; n--) s = dd_add(DD{1.0, 0.0}, dd_div(dd_mul(r, s), DD{(double)n, 0.0}));
  for (int n = 0; n < 6; n++) s = dd_mul(s, s);
  const double p = scalbn(1.0, (int)k);
  return DD{s.h * p, s.l * p};
}
// (Phi(-x), phi(x)) for x in [0, 13]
__device__ inline void dd_phi(double x, DD& Phi, DD& phi) {
  const DD rsqrt2pi{3.989422804014327029e-01, -2.492327202277730079e-17};
  const double x2 = __dmul_rn(x, x), xe = __fma_rn(x, x, -x2);
  phi = dd_mul(rsqrt2pi, dd_exp(DD{-0.5 * x2, -0.5 * xe}));
  if (x < 4.0) {  // 1/2 - phi (x + x^3/3 + x^5/15 + ...)
    DD t{x, 0.0}, s{x, 0.0};
    for (int k = 1; k < 200 && t.h > 1e-34 * s.h; k++) {
      t = dd_div(dd_mul(t, DD{x2, xe}), DD{2.0 * k + 1.0, 0.0});
      s = dd_add(s, t);
    }
    s = dd_mul(s, phi);
    Phi = dd_add(DD{0.5, 0.0}, DD{-s.h, -s.l});
  } else {  // phi / (x + 1/(x + 2/(x + 3/...)))
    DD f{x, 0.0};
    for (int k = 80; k >= 1; k--) f = dd_add(DD{x, 0.0}, dd_div(DD{(double)k, 0.0}, f));
    Phi = dd_div(phi, f);
  }
}

// midpoint of interval j of table B and half its width
__device__ __forceinline__ void t64_interval(int j, double& mid, double& half) {
  const double low = scalbn(1.0, j / 16 - T64_OCT - 1);
  half = low * 0.03125;
  mid = low * (1.0 + (j % 16) * 0.0625) + half;
}

// c[0..deg] in powers of d on |d| <= w, economised to degree 8
__device__ inline void t64_economise(double* c, int deg, double w) {
  for (int n = deg; n > 8; n--) {
    // c_n d^n = c_n w^n t^n with t = d / w; t^n minus its Chebyshev part T_n / 2^(n-1) has degree n - 2
    double tc[12] = {}, ta[12] = {}, tb[12] = {};  // coefficients of T_n, T_(k-1), T_(k-2)
    ta[1] = 1.0;
    tb[0] = 1.0;
    for (int k = 2; k <= n; k++) {
      for (int i = 0; i <= k; i++) tc[i] = (i ? 2.0 * ta[i - 1] : 0.0) - tb[i];
      for (int i = 0; i <= k; i++) {
        tb[i] = ta[i];
        ta[i] = tc[i];
      }
    }
    const double lead = tc[n];
    for (int i = n - 2; i >= 0; i -= 2) {
      double s = c[n] * (-tc[i] / lead);
      for (int q = i; q < n; q++) s *= w;
      c[i] += s;
    }
    c[n] = 0.0;
  }
}

static __global__ void __launch_bounds__(32) k_tables64(double* out) {
  const int t = blockIdx.x * 32 + threadIdx.x;
  if (t >= T64_A + T64_B) return;
  double c[12] = {};
  double lo = 0.0;  // low part of the leading coefficient
  int deg;
  double w;
  if (t < T64_A) {
    const double x = t / 64.0;
    DD P, f;
    dd_phi(x, P, f);
    c[0] = P.h;
    lo = P.l;
    double a = 0.0, b = 1.0, fact = 1.0, sg = -1.0;  // He_(k-2), He_(k-1)
    deg = 9;
    w = 1.0 / 128.0;
    for (int k = 1; k <= deg; k++, sg = -sg) {
      fact *= k;
      c[k] = sg * b * f.h / fact;
      const double n = x * b - (k - 1) * a;
      a = b;
      b = n;
    }
  } else {
    double p;
    t64_interval(t - T64_A, p, w);
    double y = ndtri_lower(p, log(p));
    DD P, f;
    dd_phi(-y, P, f);
    const DD r = dd_add(P, DD{-p, 0.0});
    const DD n = dd_two_sum(y, -(r.h / f.h));  // Newton: the correction's own error is second order
    y = n.h;
    c[0] = n.h;
    lo = n.l;
    double Pn[12] = {1.0}, fact = 1.0, pw = 1.0;
    deg = 10;
    const double yp = 1.0 / f.h;
    for (int k = 1; k <= deg; k++) {
      fact *= k;
      pw *= yp;
      double v = 0.0;
      for (int i = k - 1; i >= 0; i--) v = v * y + Pn[i];
      c[k] = v * pw / fact;
      double q[12] = {};  // P_(k+1) = P_k' + k y P_k
      for (int i = 0; i < k; i++) {
        if (i > 0) q[i - 1] += i * Pn[i];
        q[i + 1] += k * Pn[i];
      }
      for (int i = 0; i < 12; i++) Pn[i] = q[i];
    }
  }
  const double c0 = c[0];
  c[0] = 0.0;
  t64_economise(c, deg, w);
  c[0] = c0 + (c[0] + lo);
  for (int k = 0; k < T64_W; k++) out[(size_t)t * T64_W + k] = k <= 8 ? c[k] : 0.0;
}

// ---- the step -----------------------------------------------------------------------------------
__device__ __forceinline__ double t64_poly(const double* __restrict__ e, double d) {
  const double2* e2 = reinterpret_cast<const double2*>(e);
  const double2 a = e2[0], b = e2[1], c = e2[2], f = e2[3];
  double r = e[8];
  r = fma(r, d, f.y);
  r = fma(r, d, f.x);
  r = fma(r, d, c.y);
  r = fma(r, d, c.x);
  r = fma(r, d, b.y);
  r = fma(r, d, b.x);
  r = fma(r, d, a.y);
  return fma(r, d, a.x);
}
// Phi(-x) for 0 <= x <= 13 (T: the tables in shared memory)
__device__ __forceinline__ double t64_phi(const double* T, double x) {
  const double big = 105553116266496.0;  // 1.5 * 2^46: the sum's unit is 1/64
  const double s = x + big;
  return t64_poly(T + (__double2loint(s) & 1023) * T64_W, x - (s - big));
}
// the same with half the dependent steps (and three more products), for a few threads that wait on it
__device__ __forceinline__ double t64_phi_wide(const double* T, double x) {
  const double big = 105553116266496.0;
  const double s = x + big, d = x - (s - big), d2 = d * d, d4 = d2 * d2;
  const double* e = T + (__double2loint(s) & 1023) * T64_W;
  const double a = fma(e[1], d, e[0]), b = fma(e[3], d, e[2]), c = fma(e[5], d, e[4]), f = fma(e[7], d, e[6]);
  const double hi = fma(e[8], d4, fma(f, d2, c));
  return fma(hi, d4, fma(b, d2, a));
}
// Phi^-1(p) for 2^-41 <= p <= 1/2
__device__ __forceinline__ double t64_ndtri(const double* T, double p) {
  const int hi = min(__double2hiint(p), 0x3FDFFFFF);  // (1/2 itself: the end of the last interval)
  const int j = (hi >> 16) - ((1023 - T64_OCT - 1) << 4);
  const double mid = __hiloint2double((hi & 0x7FFF0000) | 0x8000, 0);
  return t64_poly(T + (T64_A + j) * T64_W, p - mid);
}

// Lattice value (w, 1 - w), exactly, as lattice_w gives it, through the bits of the doubles instead of conversions:
// num 2^-53 = (hi 2^32 + lo) 2^-53.
__device__ __forceinline__ void lattice_w64(uint64_t x, int periodize, double& w, double& wc) {
  uint64_t num;
  if (periodize) {
    const int64_t d = (int64_t)(2 * (x >> 11) + 1) - (int64_t(1) << 53);
    num = (uint64_t)(d < 0 ? -d : d);
  } else {
    num = 2 * (x >> 12) + 1;
  }
  const double a = __hiloint2double(0x41E00000, (int)(num >> 32));  // 2^31 + hi 2^-21
  const double b = __hiloint2double(0x3FE00000, (int)(uint32_t)num);  // 1/2 + lo 2^-53
  w = (a - 2147483648.5) + b;
  wc = 1.0 - w;  // (a multiple of 2^-53 below 1: exact)
}

// (y, log of the probability) of a lane off the tables
static __device__ __noinline__ double2 sov_step_rare_f64(double at, double bt, double w, double wc) {
  double ld, y;
  sov_step<double>(at, bt, w, wc, ld, y);
  if (at == -INFINITY && bt > 13.0) {
    // log1p(-h) = -h for h = Phi(-bt) = erfc(t) / 2, t = bt / sqrt(2): t's rounding, which erfc multiplies by 2 t^2
    // (1.5e-13 at bt = 37), taken back to first order
    const double t = bt * 0.70710678118654752440;
    const double e = fma(bt, 0.70710678118654752440, -t) + bt * -4.833646656726456726e-17;
    ld = bt < 39.0 ? -0.5 * erfc(t) * (1.0 - (2.0 * t + 1.0 / t) * e) : 0.0;
  }
  if (ld == -INFINITY && isnan(y)) y = 0.0;  // (an infinite limit: the sample counts as zero, whatever y is)
  return make_double2(y, ld);
}

// One variable of eq. (2): multiplies its probability into prod (in [1, 2) at the call; the caller renormalises) or
// adds its log to lsum; returns y.  zero_so_far: the sample's log P is still above -1e-20, so that even a
// probability's complement below Phi(-13) = 6e-39 counts (else it cannot reach the last bit).
template <bool ONE>
__device__ __forceinline__ double sov_step_f64(const double* T, double at, double bt, double w, double wc,
                                               bool zero_so_far, double& prod, double& lsum) {
  const double xb = fabs(bt);
  const bool nb = bt < 0.0;
  const double hb = xb <= 13.0 ? t64_phi(T, xb) : 0.0;
  double u, uc, f, c;
  bool rare, near1;
  if (ONE) {
    const double m = 1.0 - hb;
    f = nb ? hb : m;
    u = w * f;
    uc = fma(wc, f, nb ? m : hb);
    c = hb;
    near1 = bt > 3.09;  // c < 1e-3
    rare = !(bt >= -13.0) || (bt > 13.0 && zero_so_far);  // (a NaN too)
  } else {
    const double xa = fabs(at);
    const bool na = at < 0.0;
    const double ha = xa <= 13.0 ? t64_phi(T, xa) : 0.0;
    const double ma = 1.0 - ha;
    f = nb ? hb - ha : (na ? ma - hb : ha - hb);
    u = fma(w, f, na ? ha : ma);
    uc = fma(wc, f, nb ? 1.0 - hb : hb);
    c = ha + hb;
    near1 = at < -3.3 && bt > 3.3;
    // (both limits in one tail beyond the table, a zero-width interval; a NaN, which its side's zero hides from f)
    rare = !(at <= bt) || !(f > 1e-37) || (near1 && c == 0.0 && zero_so_far);
  }
  const double p = fmin(u, uc);
  rare = rare || !(p >= 4.6e-13);  // 2^-41 = 4.547e-13
  if (rare) {
    const double2 r = sov_step_rare_f64(ONE ? -INFINITY : at, bt, w, wc);
    lsum += r.y;
    return r.x;
  }
  if (near1)  // log1p(-c) to c^5: the next term is below 2e-16 c
    lsum = fma(-c, fma(c, fma(c, fma(c, fma(c, 0.2, 0.25), 0.3333333333333333), 0.5), 1.0), lsum);
  else
    prod *= f;
  const double z = t64_ndtri(T, p);
  return u <= uc ? z : -z;
}

}  // namespace tlrmvn
