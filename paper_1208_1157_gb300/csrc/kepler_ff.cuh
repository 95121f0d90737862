// Universal-variable Kepler drift with the FP64 pipe kept for the root and the state.
//
// In s = chi/sqrt(mu) the equation of `kepler_drift` (mvs_impl.cuh) reads, with beta = 2 mu/r0 -
// v0^2, zeta = mu - beta r0, sigma = r0.v0 and G_k = s^k c_k(beta s^2) (Stumpff 1962; the form
// of Rein & Tamayo 2015, Sec. 2.3),
//   F(s) = r0 s + sigma G2 + zeta G3 - h = 0,  F' = |r(s)|,  F'' = sigma G0 + zeta G1.
//   - Start: the fourth-order Taylor series and two Halley steps in FP32 (some 90 FP32
//     instructions, the time of two FP64 ones): s to 2^-22, of 24 bits.
//   - One evaluation of F and F' there in FP64, the Stumpff series' terms from z^2 on as pairs
//     (weight z^2/360).
//   - The correction d = -F/F' (1 + ...) to third order, and the G_k at s + d by their Taylor
//     step, as pairs: |d| <= 2^-19 |s|, so a pair's 2^-45 is far below the rounding of the one
//     DFMA that adds it.
//   - f, g and the new state in FP64; 1/|r| there from the hardware's root and its series.
// 54 FP64 instructions, against 150 of `kepler_drift` with one iteration (and 45 more for every
// further one that a lane of the warp needs).  Conditions, per lane: |z| < 1 (a radian of
// eccentric anomaly), |d| <= 2^-19 |s|, the dropped term below 2^-54 |s|, nothing near the ends
// of FP32's range; otherwise the caller takes `kepler_drift`.
#pragma once
#include "ff.cuh"

namespace swarm {

// 1/sqrt(a): the hardware's root y of the upper word (21 bits, so y^2 is exact), and the
// series of (1 - t)^(-1/2), t = 1 - a y^2
__device__ __forceinline__ double rsqrt_ff(const F64k &k, double a) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(a));
  y = __hiloint2double(__double2hiint(y), 0);
  const ff t = ff_from(fma(-a, kmul(k, y, y), k.one));
  const ff w = fast_two_sum(0.5f, __fmul_rn(t.h, __fmaf_rn(0.3125f, t.h, 0.375f)));
  return fma(ff_double(ff_mul(t, w)), y, y);
}

// c2 and c3 in FP32, |z| <= 1 (the dropped terms are below 2^-24)
__device__ __forceinline__ void stumpff23_f32(float z, float &c2, float &c3) {
  c2 = __fmaf_rn(z, -1.0f / 479001600.0f, 1.0f / 3628800.0f);
  c2 = __fmaf_rn(-z, c2, 1.0f / 40320.0f);
  c2 = __fmaf_rn(-z, c2, 1.0f / 720.0f);
  c2 = __fmaf_rn(-z, c2, 1.0f / 24.0f);
  c2 = __fmaf_rn(-z, c2, 0.5f);
  c3 = __fmaf_rn(z, -1.0f / 6227020800.0f, 1.0f / 39916800.0f);
  c3 = __fmaf_rn(-z, c3, 1.0f / 362880.0f);
  c3 = __fmaf_rn(-z, c3, 1.0f / 5040.0f);
  c3 = __fmaf_rn(-z, c3, 1.0f / 120.0f);
  c3 = __fmaf_rn(-z, c3, 1.0f / 6.0f);
}
// c - z (d - z (e - z r)) as a pair: r FP32 (weight z^3 e.../c, below 2^-19 of c)
__device__ __forceinline__ ff stumpff_tail(const ff &z, float r, const ff &e, const ff &d, const ff &c) {
  ff y = fast_two_sum(e.h, __fmul_rn(-z.h, r));
  y.l = __fadd_rn(y.l, e.l);
  ff p = ff_mul_raw(z, y);
  y = fast_two_sum(d.h, -p.h);
  y.l = __fadd_rn(y.l, __fsub_rn(d.l, p.l));
  p = ff_mul_raw(z, y);
  y = fast_two_sum(c.h, -p.h);
  return fast_two_sum(y.h, __fadd_rn(y.l, __fsub_rn(c.l, p.l)));
}
// c2 and c3 of |z| < 1, to FP64 rounding
__device__ __forceinline__ void stumpff23_ff(double z, double &c2, double &c3) {
  const ff zf = ff_norm(ff_from(z));
  float r = __fmaf_rn(zf.h, -1.0f / 6402373705728000.0f, 1.0f / 20922789888000.0f);
  r = __fmaf_rn(-zf.h, r, 1.0f / 87178291200.0f);
  r = __fmaf_rn(-zf.h, r, 1.0f / 479001600.0f);
  const ff a = stumpff_tail(zf, r, ff_const(1.0 / 3628800.0), ff_const(1.0 / 40320.0), ff_const(1.0 / 720.0));
  c2 = fma(-z, fma(-z, ff_double(a), 1.0 / 24.0), 0.5);
  r = __fmaf_rn(zf.h, -1.0f / 121645100408832000.0f, 1.0f / 355687428096000.0f);
  r = __fmaf_rn(-zf.h, r, 1.0f / 1307674368000.0f);
  r = __fmaf_rn(-zf.h, r, 1.0f / 6227020800.0f);
  const ff b = stumpff_tail(zf, r, ff_const(1.0 / 39916800.0), ff_const(1.0 / 362880.0), ff_const(1.0 / 5040.0));
  c3 = fma(-z, fma(-z, ff_double(b), 1.0 / 120.0), 1.0 / 6.0);
}

// The drift of (r, v) by h; rq = 1/|r| and r2 = |r|^2 on entry (and, of the new r, on return).
// A lane whose conditions do not hold is left as it was and gets false; so is the lane of the
// centre of mass (`star`), or with FREE it moves uniformly.
template <bool FREE>
__device__ __forceinline__ bool kepler_drift_ff(const F64k &k, bool star, double mu, double (&r)[3], double (&v)[3],
                                                double h, double &rq, double &r2) {
  const double u = rq;
  const double r0 = kmul(k, r2, u);
  const double sig = fma(r[2], v[2], fma(r[1], v[1], kmul(k, r[0], v[0])));
  const double v2 = fma(v[2], v[2], fma(v[1], v[1], kmul(k, v[0], v[0])));
  const double beta = fma(kmul(k, mu, u), 2.0, -v2);
  const double zeta = fma(-beta, r0, mu);

  const float hf = f_from(h), r0f = f_from(r0), sf = f_from(sig), zf = f_from(zeta), bf = f_from(beta);
  float s1;
  {
    const float uf = f_from(u), muu = f_from(mu) * uf;
    const float su = sf * uf, su2 = su * su, A = f_from(v2) - muu, hu = hf * uf;
    const float t4 = su * (1.0f / 24.0f) * __fmaf_rn(-15.0f, su2, __fmaf_rn(9.0f, A, muu));
    const float t3 = (-1.0f / 6.0f) * __fmaf_rn(-3.0f, su2, A);
    s1 = __fmaf_rn(hu, __fmaf_rn(hu, __fmaf_rn(hu, t4, t3), -0.5f * su), 1.0f) * hu;
  }
#pragma unroll
  for (int i = 0; i < 2; i++) {  // Halley
    const float ss = s1 * s1, z = bf * ss;
    float c2, c3;
    stumpff23_f32(z, c2, c3);
    const float G0 = __fmaf_rn(-z, c2, 1.0f), G1 = s1 * __fmaf_rn(-z, c3, 1.0f), G2 = ss * c2, G3 = ss * s1 * c3;
    const float F = __fmaf_rn(sf, G2, __fmaf_rn(zf, G3, __fmaf_rn(r0f, s1, -hf)));
    const float dF = __fmaf_rn(sf, G1, __fmaf_rn(zf, G2, r0f)), ddF = __fmaf_rn(sf, G0, zf * G1);
    s1 -= __fdividef(F * dF, __fmaf_rn(-0.5f * F, ddF, dF * dF));
  }
  // exactly (a normal number, see the last condition)
  const int sb = __float_as_int(s1);
  const double s = __hiloint2double((((sb & 0x7fffffff) >> 3) + (896 << 20)) | (sb & 0x80000000), sb << 29);

  const double ss = kmul(k, s, s), z = kmul(k, beta, ss);
  double c2, c3;
  stumpff23_ff(z, c2, c3);
  double G1 = kmul(k, s, fma(-z, c3, 1.0)), G2 = kmul(k, ss, c2), G3 = kmul(k, kmul(k, ss, s), c3);
  const double F = fma(sig, G2, fma(zeta, G3, fma(r0, s, -h)));
  const double dF = fma(sig, G1, fma(zeta, G2, r0));  // |r(s)|
  const ff g2 = ff_from(G2), g1 = ff_from(G1), df = ff_from(dF), ef = ff_from(F);
  const ff bG2 = ff_mul(ff_from(beta), g2);
  const ff g0 = ff_sub(ff_make(1.0f, 0.0f), bG2);
  const float inv = __frcp_rn(df.h);
  const float ddF = __fmaf_rn(sf, g0.h, zf * g1.h), dddF = __fmaf_rn(zf, g0.h, -bf * sf * g1.h);
  const float q0 = ef.h * inv;
  const float e2 = 0.5f * ddF * inv;  // F''/2F'
  // F/F' to 2^-44, times 1 + q F''/2F'
  const float q1 = (__fmaf_rn(-q0, df.h, ef.h) + __fmaf_rn(-q0, df.l, ef.l)) * inv;
  const ff d = fast_two_sum(-q0, -__fmaf_rn(q0 * q0, e2, q1));
  const float d2 = d.h * d.h, as = fabsf(s1);
  const float cub = __fmaf_rn(2.0f * e2, e2, fabsf(dddF * inv) * (1.0f / 6.0f));
  const bool ok = abs_below_pow2(z, 0) && fabsf(d.h) <= 0x1p-19f * as && cub * d2 * fabsf(d.h) <= 0x1p-54f * as &&
                  as > 0x1p-100f && as < 0x1p50f && abs_below_pow2(F, 100) && abs_below_pow2(dF, 100) &&
                  abs_below_pow2(v2, 80) && abs_below_pow2(r2, 40) && !abs_below_pow2(r2, -40);
  const float hd2 = 0.5f * d2;
  {
    const ff w1 = ff_mul_raw(g0, d), w2 = ff_mul_raw(g1, d), w3 = ff_mul_raw(g2, d);
    G1 = ff_addto(G1, fast_two_sum(w1.h, __fmaf_rn(-bf * g1.h, hd2, w1.l)));
    G2 = ff_addto(G2, fast_two_sum(w2.h, __fmaf_rn(g0.h, hd2, w2.l)));
    G3 = ff_addto(G3, fast_two_sum(w3.h, __fmaf_rn(g1.h, hd2, w3.l)));
  }
  const double mG2 = kmul(k, mu, G2);
  const double f = fma(-mG2, u, 1.0), g = fma(-mu, G3, h);
  double rn[3];
#pragma unroll
  for (int c = 0; c < 3; c++) {  // f r + g v; a free body h v + r
    const bool free = FREE && star;
    const double a = free ? h : f, x = free ? v[c] : r[c], b = free ? k.one : g, y = free ? r[c] : v[c];
    rn[c] = fma(a, x, kmul(k, b, y));
  }
  const double rn2 = fma(rn[2], rn[2], fma(rn[1], rn[1], kmul(k, rn[0], rn[0])));
  const double rinv = rsqrt_ff(k, rn2);
  const double fd = kmul(k, kmul(k, -mu, G1), kmul(k, u, rinv)), gd = fma(-mG2, rinv, 1.0);
  const bool take = star ? FREE : ok;
#pragma unroll
  for (int c = 0; c < 3; c++) {
    const double vn = fma(fd, r[c], kmul(k, gd, v[c]));
    if (take && !star) v[c] = vn;
    if (take) r[c] = rn[c];
  }
  if (take) {
    rq = rinv;
    r2 = rn2;
  }
  return take;
}

}  // namespace swarm
