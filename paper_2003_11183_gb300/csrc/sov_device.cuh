// Device functions of the float32 integrand and of the Student-t scale, shared
// by the single-problem integrand (prob.cu) and the batched persistent kernel (batch.cu).
#pragma once
#include "common.cuh"

namespace tlrmvn {

// ---- Student-t scale (Algorithm 7): chi_nu^-1(w0)/sqrt(nu) ------------------------
// Regularised incomplete gamma P(a,x) and Q(a,x) = 1 - P: power series below
// x = a + 1, Legendre continued fraction (modified Lentz) above; lga = log Gamma(a), x > 0.
// Both need some 8.5 sqrt(a) terms near x = a.  f1: the derivative of P.
__device__ inline void gamma_pq(double a, double lga, double x, double& P, double& Q, double& f1) {
  // log of x^a e^-x / Gamma(a); for large a by Stirling's series around x = a, where the logs' rounding would count
  const double u = (x - a) / a;
  const double lpref = a > 1000.0 ? 0.5 * log(a * 0.15915494309189535) - (1.0 - 1.0 / (30.0 * a * a)) / (12.0 * a) -
                                        a * (u - log1p(u))
                                  : a * log(x) - x - lga;
  const double pref = exp(lpref);
  f1 = pref / x;
  const int terms = 2000 + (int)fmin(10.0 * sqrt(a), 200000.0);
  if (x < a + 1.0) {
    double ap = a, term = 1.0 / a, sum = term;
    for (int it = 0; it < terms; it++) {
      ap += 1.0;
      term *= x / ap;
      sum += term;
      if (fabs(term) <= fabs(sum) * 1.2e-16) break;
    }
    P = sum * pref;
    Q = 1.0 - P;
  } else {
    const double tiny = 1e-300;
    double bq = x + 1.0 - a, c = 1.0 / tiny, d = 1.0 / bq, h = d;
    for (int i = 1; i < terms; i++) {
      double an = -i * (i - a);
      bq += 2.0;
      d = an * d + bq;
      if (fabs(d) < tiny) d = tiny;
      c = bq + an / c;
      if (fabs(c) < tiny) c = tiny;
      d = 1.0 / d;
      double del = d * c;
      h *= del;
      if (fabs(del - 1.0) <= 4.5e-16) break;  // a few ulp: exact equality may never occur
    }
    Q = pref * h;
    P = 1.0 - Q;
  }
}

// x with P(a, x) = p (q = 1 - p exactly): Halley steps, kept between the points known to lie on either side of it.
// Start: Wilson-Hilferty's cube, or, where its base is small and it lies far too low or is negative, the leading term of
// the series, p = x^a / Gamma(a + 1), which never lies above x.
__device__ inline double gamma_p_inv(double a, double p, double q) {
  const double z = ndtri2(p, q, log(p)), t = 1.0 / (9.0 * a), lga = lgamma(a);
  const double base = 1.0 - t + z * sqrt(t);
  double x = a * base * base * base, lo = 0.0, hi = INFINITY;
  if (base < 0.5) {
    const double x0 = exp((log(p) + lga + log(a)) / a);
    x = fmax(x, x0);
    lo = 0.999999 * x0;
  }
  if (!(x > 0.0)) return x;  // (below the smallest double)
  for (int it = 0; it < 100; it++) {
    double P, Q, f1;
    gamma_pq(a, lga, x, P, Q, f1);
    const double f = (p < 0.5) ? (P - p) : (q - Q);
    if (f < 0.0) lo = x;
    else hi = x;
    const double dx = f / f1;
    const double corr = 0.5 * dx * ((a - 1.0) / x - 1.0);
    const double step = (fabs(corr) < 0.5) ? dx / (1.0 - corr) : dx;
    double xn = x - step;
    // Halley converges cubically: once a step is below 1e-12 x the next iterate
    // is exact to rounding, so stop there instead of chasing the last ulp
    const bool done = fabs(xn - x) <= 1e-12 * x;
    if (!done && !(xn > lo && xn < hi)) xn = hi < INFINITY ? 0.5 * (lo + hi) : 2.0 * x;  // (also where f1 underflows)
    x = xn;
    if (done) break;
  }
  return x;
}

// ---- float32 integrand helpers ------------------------------------------------------
// Lattice value as floats for the float32 integrands: the cell midpoint of the
// point's top 32 bits, (h + 1/2) / 2^32 with h = x >> 32, through the tent map
// when periodised, w = |2 (h + 1/2) / 2^32 - 1| = |2 d + 1| / 2^32 with d = h - 2^31, and
// 1 - w = |2 h' + 1| / 2^32 with h' = h read as a signed integer.  Integer
// arithmetic and two 32-bit conversions only (the float path issues no float64
// instruction).  It differs from the exact value of the 53-bit definition
// (lattice_w) by at most 2^-32 (2^-33 without the tent map): within half a
// float32 ulp for w >= 2^-8, and a relative 2^-32 / w below that.
__device__ __forceinline__ void lattice_wf(uint64_t x, int periodize, float& w, float& wc) {
  const uint32_t h = (uint32_t)(x >> 32);
  if (periodize) {
    w = fabsf(fmaf((float)(int32_t)(h ^ 0x80000000u), 4.656612873077393e-10f, 2.3283064365386963e-10f));
    wc = fabsf(fmaf((float)(int32_t)h, 4.656612873077393e-10f, 2.3283064365386963e-10f));
  } else {
    w = fmaf((float)h, 2.3283064365386963e-10f, 1.1641532182693481e-10f);                  // (h + 1/2) / 2^32
    wc = fmaf((float)(0xFFFFFFFFu - h), 2.3283064365386963e-10f, 1.1641532182693481e-10f);
  }
}

// eq. (2) for one variable in float32.  The one-sided case (at = -inf), which is
// the whole integrand for upper-limit problems, has a branch-free fast path for
// bt >= -12 (Phi(bt) > 1.7e-33): one complementary error function of |bt|, one
// log, and the library's float quantile (ndtri_f32); samples of one
// warp take the same instructions whatever the sign of their limit.  log Phi(bt)
// near 1 uses Goldberg's form of log1p (D. Goldberg, What every computer
// scientist should know about floating-point arithmetic, 1991, Theorem 4):
// log1p(-c) = log(s) * (-c) / (s - 1) with s = fl(1 - c).  Quantiles whose
// probability is below 1e-30 take the log of that probability from logs of its
// factors, and limits below -12 go through the log-domain code.
__device__ __forceinline__ void sov_step_f32(float at, float bt, float w, float wc, float& ld, float& y) {
  const float rs2 = (float)TLR_RSQRT2;
  if (at == -INFINITY && bt != INFINITY) {
    if (bt >= -12.0f) {
      const float h = 0.5f * erfcf(fabsf(bt) * rs2);  // Phi(-|bt|)
      const bool neg = bt < 0.0f;
      const float ph = neg ? h : 1.0f - h;  // Phi(bt)
      const float pc = neg ? 1.0f - h : h;  // 1 - Phi(bt)
      const float s1 = 1.0f - pc;
      const float lg = logf(neg ? ph : s1);
      ld = neg ? lg : ((s1 == 1.0f) ? -pc : lg * (-pc / (s1 - 1.0f)));
      const float u = w * ph, uc = pc + wc * ph;  // u + uc = 1
      const bool lower = u <= uc;
      const float pp = lower ? u : uc;
      float lpp = 0.0f;
      if (pp < 1e-30f) lpp = logf(w) + ld;  // (u underflows: its log from the logs of its factors)
      const float z = ndtri_f32(pp, lpp);
      y = lower ? z : -z;
      return;
    }
    const float t = -bt * rs2;
    const float le = logf(0.5f * erfcxf(t)) - t * t;  // log Phi(bt)
    const float lu = logf(w) + le;                      // log u, u = w Phi(bt) < 1/2
    y = ndtri_lower(expf(lu), lu);
    ld = le;
    return;
  }
  sov_step<float>(at, bt, w, wc, ld, y);
}

// Phi(-x) in float32 for x >= 0 (zero beyond 13, where it falls below the normal floats; NaN for a NaN), straight-line:
// exp(-x^2/2) R(x), with R half the scaled complementary error function as a degree-9 polynomial in
// 1 / (2.5 + x) (coefficients from csrc/fit_mills.py; its even and odd halves side by side), and the
// exponential from x^2 in two parts, x^2 + er exactly: -(x^2 + er) log2(e)/2 = n + f with n the nearest
// integer, 2^f by the hardware and 2^n added to the exponent.  Relative error 4.0e-7 at most and 8e-8 rms with
// an exact 2^f and reciprocal.
__device__ __forceinline__ float phi_neg_f32(float x) {
  x = min_nan(x, 13.0f);
  const float x2 = x * x, er = fmaf(x, x, -x2);
  const float kf = fmaf(x2, -7.213475108e-01f, 12582912.0f);  // the integer n in the low bits
  float f = fmaf(x2, -7.213475108e-01f, 12582912.0f - kf);
  f = fmaf(x2, -9.629815168e-09f, f);
  f = fmaf(er, -7.213475108e-01f, f);
  const float e = __int_as_float(__float_as_int(ex2_ftz(f)) + (__float_as_int(kf) << 23));
  const float t = rcp_ftz(x + 2.5f), t2 = t * t;
  float p = -6.734211731e+01f, q = 3.024349689e+00f;
  p = fmaf(p, t2, -9.483559418e+01f);
  q = fmaf(q, t2, 1.291362152e+02f);
  p = fmaf(p, t2, -7.301989794e-01f);
  q = fmaf(q, t2, 2.569419479e+01f);
  p = fmaf(p, t2, 9.710934162e-01f);
  q = fmaf(q, t2, 2.507573128e+00f);
  p = fmaf(p, t2, -1.405569856e-05f);
  q = fmaf(q, t2, 3.998731673e-01f);
  return mul_ftz(e, fmaf(q, t, p));
}

// The same step for a caller that keeps the sample's probability as a running
// product: returns y, a factor f to multiply into the product and a log added to
// the separate sum lsum.  The fast path's factor is the probability, except when its
// complement c is below 3e-4, where fl(1 - c) would lose c's digits: then f = 1 and
// log1p(-c) is added as -c - c^2/2 (the next term is below 4e-8 c).  f is at least
// 2.5e-19, so that a caller may multiply two into a product in [1, 2).
//
// The fast path is straight-line code for every lane, and one branch follows for
// the lanes it does not serve (limits in the deep tail; a quantile below 8.4e-5, a
// lane in 6,000; a NaN, whose log must reach lsum, for the product's renormalisation drops it): the chain from a variable's sum to its y is what bounds the
// sweeps, and branches cut it (the one-sided case, the quantile's tail when that
// started at 0.0017 and one warp in ten took it, the underflow test) and keep the compiler from
// filling its waits.  With u = Phi(at) + w (Phi(bt) - Phi(at)) and uc = 1 - u both accurate, the
// quantile takes 4 p (1 - p) = 4 u uc and 1 - 2p = +-(uc - u) from them directly: no
// minimum, comparison or select on the way to y.

// (y, the step's log) of a lane off the fast path, the only one whose y may be large: cut to CAP in size (0: not)
template <int CAP>
static __device__ __noinline__ float2 sov_step_rare_f32(float at, float bt, float w, float wc, float pp, bool deep) {
  if (!deep) return make_float2(ndtri_tail_f32(__logf(pp)), 0.0f);
  float ld, y;
  sov_step_f32(at, bt, w, wc, ld, y);
  if (CAP) y = fminf(fmaxf(y, (float)-CAP), (float)CAP);
  return make_float2(y, ld);
}

// The one-sided (at = -inf) case.
template <int CAP = 0>
__device__ __forceinline__ void sov_step_f32_upper(float bt, float w, float wc, float& f, float& lsum, float& y) {
  const float h = phi_neg_f32(fabsf(bt)), m = 1.0f - h;  // Phi(-|bt|), Phi(|bt|)
  const bool neg = bt < 0.0f, near1 = bt > 3.5f;
  const float ph = neg ? h : m, pc = neg ? m : h;  // Phi(bt), 1 - Phi(bt)
  const float c = near1 ? h : 0.0f;
  f = near1 ? 1.0f : ph;
  lsum = fmaf(-c, fmaf(0.5f, c, 1.0f), lsum);
  const float u = w * ph, uc = fmaf(wc, ph, pc);
  const float L = lg2_ftz(u * uc);  // log2(4 u uc) - 2
  y = ndtri_poly_f32(L + 5.0f) * (uc - u);
  if (!(L >= NDTRI_LMIN - 2.0f)) {
    // (a deep limit always comes here: u < Phi(-8.9) = 2.8e-19; above it pp > 3e-29; and a NaN, as a deep one)
    const bool deep = !(bt >= -8.9f);
    const float2 r = sov_step_rare_f32<CAP>(-INFINITY, bt, w, wc, fminf(u, uc), deep);
    y = (deep || u <= uc) ? r.x : -r.x;
    f = deep ? 1.0f : f;
    lsum += r.y;
  }
}

// Any interval.  With both limits on one side of 0 the probability is the difference of the two smaller tails.
template <int CAP = 0>
__device__ __forceinline__ void sov_step_f32_prod(float at, float bt, float w, float wc, float& f, float& lsum,
                                                  float& y) {
  const float ha = phi_neg_f32(fabsf(at)), hb = phi_neg_f32(fabsf(bt)), ma = 1.0f - ha;
  const bool na = at < 0.0f, nb = bt < 0.0f, near1 = fminf(-at, bt) > 3.6f;
  const float d = na ? ha : ma, ec = nb ? 1.0f - hb : hb;  // Phi(at), 1 - Phi(bt)
  const float diff = nb ? hb - ha : (na ? ma - hb : ha - hb);
  const float c = near1 ? ha + hb : 0.0f;
  f = near1 ? 1.0f : diff;
  lsum = fmaf(-c, fmaf(0.5f, c, 1.0f), lsum);
  const float u = fmaf(w, diff, d), uc = fmaf(wc, diff, ec);
  const float L = lg2_ftz(u * uc);
  y = ndtri_poly_f32(L + 5.0f) * (uc - u);
  const bool deep = !(diff >= 2.5e-19f);  // (also a zero-width interval and, through the comparison, a NaN)
  if (deep || L < NDTRI_LMIN - 2.0f) {
    const float2 r = sov_step_rare_f32<CAP>(at, bt, w, wc, fminf(u, uc), deep);
    y = (deep || u <= uc) ? r.x : -r.x;
    f = deep ? 1.0f : f;
    lsum += r.y;
  }
}

}  // namespace tlrmvn
