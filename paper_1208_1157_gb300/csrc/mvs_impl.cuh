// Mixed-variable symplectic integrator (Sec. 2.2.3, Sec. 4.3.4) on sm_103a, body per lane.
//
// Lane b of a group holds body b's canonical coordinates: b = 0 the centre of mass,
// b >= 1 a planet (democratic heliocentric Q_b = x_b - x_0, u_b = v_b - v_cm; or Jacobi
// r'_b, v'_b).  Each step runs the paper's sub-steps in order: Cartesian drift half step,
// kick half step, Kepler drift, kick half step, Cartesian drift half step (DH); kick,
// Kepler, kick (Jacobi).  The interaction accelerations computed after the Kepler drift
// are reused by the next step's first kick (Sec. 4.3.4): one force evaluation per step.
// Here: the coordinate maps, and the drift and the accelerations in FP64, for the parts of a step
// that mvs_ff.cuh's pairs do not carry and for 16..32 bodies.
#pragma once
#include "hermite.cuh"
#include "kernels.h"

namespace swarm {

// ---------------------------------------------------------------- acceleration ring
// Acceleration only (Eq. 1), over M members at lanes base+OFF .. base+OFF+M-1; member j.
// Lanes outside the members (the centre-of-mass lane in DH) mirror member 0 and their
// results are discarded.
template <int M>
struct ARing {
  static constexpr int RF = (M - 1) / 2;
  static constexpr bool HALF = (M % 2) == 0 && M > 0;
  static constexpr int RT = RF + (HALF ? 1 : 0);
  static constexpr int RTA = RT > 0 ? RT : 1;
};

template <int M, int OFF>
__device__ __forceinline__ void ring_acc(const F64k &k, const double (&x)[3], double m, int j, int base, double (&a)[3],
                                         double (&d2)[ARing<M>::RTA]) {
#pragma unroll
  for (int c = 0; c < 3; c++) a[c] = 0.0;
#pragma unroll
  for (int r = 1; r <= ARing<M>::RF; r++) {
    int p = j + r;
    if (p >= M) p -= M;
    int q = j - r;
    if (q < 0) q += M;
    double dx[3];
#pragma unroll
    for (int c = 0; c < 3; c++) dx[c] = ksub(k, shfl(x[c], base + OFF + p), x[c]);
    double mp = shfl(m, base + OFF + p);
    double r2 = kmul(k, dx[0], dx[0]);
    r2 = fma(dx[1], dx[1], r2);
    r2 = fma(dx[2], dx[2], r2);
    double rho = rsqrt(r2);
    double rho3 = kmul(k, kmul(k, rho, rho), rho);
    double sp = kmul(k, mp, rho3), si = kmul(k, m, rho3);
#pragma unroll
    for (int c = 0; c < 3; c++) a[c] = fma(sp, dx[c], a[c]);
    double rdx[3];
#pragma unroll
    for (int c = 0; c < 3; c++) rdx[c] = shfl(dx[c], base + OFF + q);
    double rs = shfl(si, base + OFF + q);
#pragma unroll
    for (int c = 0; c < 3; c++) a[c] = fma(-rs, rdx[c], a[c]);
    d2[r - 1] = r2;
  }
  if (ARing<M>::HALF) {
    constexpr int r = M / 2;
    int p = j + r;
    if (p >= M) p -= M;
    double dx[3];
#pragma unroll
    for (int c = 0; c < 3; c++) dx[c] = ksub(k, shfl(x[c], base + OFF + p), x[c]);
    double mp = shfl(m, base + OFF + p);
    double r2 = kmul(k, dx[0], dx[0]);
    r2 = fma(dx[1], dx[1], r2);
    r2 = fma(dx[2], dx[2], r2);
    double rho = rsqrt(r2);
    double sp = kmul(k, mp, kmul(k, kmul(k, rho, rho), rho));
#pragma unroll
    for (int c = 0; c < 3; c++) a[c] = fma(sp, dx[c], a[c]);
    d2[ARing<M>::RT - 1] = r2;
  }
}

// ---------------------------------------------------------------- Stumpff and Kepler
// c2(z), c3(z) by their power series (8 terms each; on |z| <= 0.25 within 2.3e-16
// relative of the closed forms), reaching larger |z| by quartering the argument and the
// doubling relations c0(4z) = 2 c0^2 - 1, c1(4z) = c0 c1, c2(4z) = c1^2 / 2,
// c3(4z) = (c2 + c0 c3) / 4 (Danby 1988, Sec. 6.9).  Steps of 1/20 of an orbit give
// z ~ 0.1, so the series alone usually serves.
__device__ __forceinline__ void stumpff23(double z, double &c2, double &c3) {
  int k = 0;
  while (!abs_below_pow2(z, -2) && k < 40) {  // |z| >= 0.25, tested on the exponent bits
    z *= 0.25;
    k++;
  }
  // Horner forms of sum (-z)^i/(2i+2)! (i <= 7) and sum (-z)^i/(2i+3)! (i <= 7)
  c2 = fma(z, 1.0 / 20922789888000.0, -1.0 / 87178291200.0);
  c2 = fma(z, c2, 1.0 / 479001600.0);
  c2 = fma(z, c2, -1.0 / 3628800.0);
  c2 = fma(z, c2, 1.0 / 40320.0);
  c2 = fma(z, c2, -1.0 / 720.0);
  c2 = fma(z, c2, 1.0 / 24.0);
  c2 = fma(z, c2, -0.5);
  c2 = -c2;
  c3 = fma(z, -1.0 / 355687428096000.0, 1.0 / 1307674368000.0);
  c3 = fma(z, c3, -1.0 / 6227020800.0);
  c3 = fma(z, c3, 1.0 / 39916800.0);
  c3 = fma(z, c3, -1.0 / 362880.0);
  c3 = fma(z, c3, 1.0 / 5040.0);
  c3 = fma(z, c3, -1.0 / 120.0);
  c3 = fma(z, c3, 1.0 / 6.0);
  if (k) {
    double c1 = fma(-z, c3, 1.0);
    double c0 = fma(-z, c2, 1.0);
    for (int i = 0; i < k; i++) {
      c3 = 0.25 * fma(c0, c3, c2);
      c2 = 0.5 * c1 * c1;
      c1 = c0 * c1;
      c0 = fma(2.0 * c0, c0, -1.0);
    }
  }
}

struct KepConst {
  double mu, smu, smuinv, muinv;
};
__device__ __forceinline__ KepConst kep_const(double mu) {
  KepConst k;
  k.mu = mu;
  k.smu = sqrt(mu);
  k.smuinv = 1.0 / k.smu;
  k.muinv = 1.0 / mu;
  return k;
}

// Starting guesses of Vallado, "Fundamentals of Astrodynamics and Applications",
// Algorithm 8 (elliptic, hyperbolic, parabolic): for drifts longer than about a radian of
// eccentric anomaly, where the Taylor start below does not hold.
static __device__ __noinline__ double chi_guess(const KepConst &K, const double (&r)[3], const double (&v)[3], double r0, double sig0,
                            double alpha, double h) {
  if (alpha > 1e-6) return K.smu * alpha * h;
  if (alpha < -1e-6) {
    double a = 1.0 / alpha;
    double sg = h >= 0 ? 1.0 : -1.0;
    double arg = (-2.0 * K.mu * alpha * h) / (sig0 + sg * sqrt(-K.mu * a) * (1.0 - r0 * alpha));
    return arg > 0 ? sg * sqrt(-a) * log(arg) : K.smu * h / r0;
  }
  double hx = r[1] * v[2] - r[2] * v[1], hy = r[2] * v[0] - r[0] * v[2], hz = r[0] * v[1] - r[1] * v[0];
  double p = (hx * hx + hy * hy + hz * hz) * K.muinv;
  double s = 0.5 * atan(1.0 / (3.0 * sqrt(K.mu / (p * p * p)) * h));
  double w = atan(cbrt(tan(s)));
  return sqrt(p) * 2.0 / tan(2.0 * w);
}

// Universal-variable Kepler drift of (r, v) by h.  The universal anomaly chi solves
//   F(chi) = s0 U2 + beta U3 + r0 chi - sqrt(mu) h = 0,   U_k = chi^k c_k(alpha chi^2),
// s0 = r0.v0/sqrt(mu), beta = 1 - alpha r0, with F' = |r(chi)|, F'' = s0 U0 + beta U1 and
// F''' = beta U0 - alpha s0 U1 (U3' = U2, U2' = U1, U1' = U0, U0' = -alpha U1).
//  - Start: the Taylor series of chi(t) about the current state to fourth order in h,
//    from d chi/dt = sqrt(mu)/r, dr/dt = sigma/r, d sigma/dt = v^2 - mu/r and
//    d v^2/dt = -2 mu sigma/r^3 (sigma = r.v, u = 1/r); the derivatives are
//      1st: sqrt(mu) u,  2nd: -sqrt(mu) sigma u^3,
//      3rd: -sqrt(mu) u^3 (v^2 - mu u - 3 sigma^2 u^2),
//      4th: sqrt(mu) sigma u^5 (9 v^2 - 8 mu u - 15 sigma^2 u^2).
//    Its error is of order e (n h)^5/120 of chi for eccentricity e and mean motion n
//    (~4e-7 relative for e = 0.1 and steps of 1/20 orbit).  Beyond about a radian of
//    eccentric anomaly (|alpha| (sqrt(mu) u h)^2 >= 1) Vallado's guesses are taken instead.
//  - First iteration: Halley's method, cubic convergence, its remaining error
//    |F'''/(6F') - (F''/(2F'))^2| dchi^3; later iterations (rare) Newton's, remaining
//    error |F''/(2F')| dchi^2.  Stop when that error is below 1e-16 |chi| (half an ulp: the
//    root to rounding) or |dchi| <= 1e-14 max(1, |chi|) (the oracle's test).  One Halley
//    step from the Taylor start meets the first test for moderate eccentricities.
//  - The universal functions at the root come from those of the last iterate by a
//    third-order Taylor step in its correction (exact to rounding for |dchi| <= 1e-5
//    max(1, |chi|), dropped terms ~ dchi^4/24; else recomputed at the root); then the
//    Lagrange f, g, fdot, gdot.
// Executed by every lane of the warp; lanes with `on` false do not change their state.
// Returns false on non-convergence in 50 iterations.  The corrections divide by
// rcp_newton, whose error (~1e-13 relative at most) only scales the small last correction.
// RQ: rq holds 1/|r| of the current r on entry (computed by the same expression); on exit
// the lanes that drifted hold 1/|r| of the new r there.
template <bool RQ>
__device__ __forceinline__ bool kepler_drift(const F64k k, bool on, const KepConst &K, double (&r)[3], double (&v)[3],
                                             double h, int &iters, double &rq) {
  const double r2 = fma(r[2], r[2], fma(r[1], r[1], kmul(k, r[0], r[0])));
  const double u = RQ ? rq : rsqrt(r2);  // 1/r0
  const double r0 = kmul(k, r2, u);
  const double sig0 = fma(r[2], v[2], fma(r[1], v[1], kmul(k, r[0], v[0])));
  const double v2 = fma(v[2], v[2], fma(v[1], v[1], kmul(k, v[0], v[0])));
  const double mu_u = kmul(k, K.mu, u);
  const double alpha = kmul(k, ksub(k, kmul(k, 2.0, mu_u), v2), K.muinv);  // (2 mu/r0 - v^2)/mu
  const double s0 = kmul(k, sig0, K.smuinv);
  const double beta = fma(-alpha, r0, 1.0);
  const double target = kmul(k, K.smu, h);
  const double ms0a = kmul(k, -alpha, s0);
  // fourth-order Taylor start: chi = h (T1 + h (T2 + h (T3 + h T4)))
  const double T1 = kmul(k, K.smu, u);  // sqrt(mu) u
  const double su = kmul(k, sig0, u);   // sigma u
  const double su2 = kmul(k, su, su);
  const double Pu = kmul(k, T1, u);     // sqrt(mu) u^2
  const double Q = kmul(k, Pu, u);      // sqrt(mu) u^3
  const double A = ksub(k, v2, mu_u);   // v^2 - mu u
  const double T2 = kmul(k, kmul(k, -0.5, Pu), su);
  const double T3 = kmul(k, kmul(k, Q, -1.0 / 6.0), fma(-3.0, su2, A));
  const double T4 = kmul(k, kmul(k, kmul(k, Q, su), 1.0 / 24.0), fma(-15.0, su2, fma(9.0, A, mu_u)));
  double x = kmul(k, h, fma(h, fma(h, fma(h, T4, T3), T2), T1));
  const double x1 = kmul(k, T1, h);
  if (on && !abs_below_pow2(kmul(k, alpha, kmul(k, x1, x1)), 0)) x = chi_guess(K, r, v, r0, sig0, alpha, h);
  bool done = !on;
  int it = 0;
  // universal functions U0..U3 at the last iterate and its correction dx
  double U0 = 1.0, U1 = 0.0, U2 = 0.0, U3 = 0.0, dx = 0.0;
  for (int i = 0; i < 50; i++) {
    if (__all_sync(0xffffffffu, done)) break;
    if (!done) {
      const double xx = kmul(k, x, x);
      const double z = kmul(k, alpha, xx);
      double c2, c3;
      stumpff23(z, c2, c3);
      U0 = fma(-z, c2, 1.0);
      U1 = kmul(k, x, fma(-z, c3, 1.0));
      U2 = kmul(k, xx, c2);
      U3 = kmul(k, kmul(k, xx, x), c3);
      const double F = fma(s0, U2, fma(beta, U3, fma(r0, x, -target)));
      const double dF = fma(s0, U1, fma(beta, U2, r0));  // |r(chi)|
      const double ddF = fma(s0, U0, kmul(k, beta, U1));
      double err;
      if (it == 0) {  // Halley
        const double D = fma(kmul(k, -0.5, F), ddF, kmul(k, dF, dF));
        const double rD = rcp_newton(k, D);
        const double idF = kmul(k, dF, rD);  // ~1/F' (D = F'^2 (1 + O(F)))
        dx = kmul(k, kmul(k, F, dF), rD);
        const double dddF = fma(ms0a, U1, kmul(k, beta, U0));
        const double g2 = kmul(k, kmul(k, 0.5, ddF), idF);
        const double C = fma(-g2, g2, kmul(k, kmul(k, dddF, idF), 1.0 / 6.0));
        err = kmul(k, kmul(k, fabs(C), fabs(dx)), kmul(k, dx, dx));
      } else {  // Newton
        const double idF = rcp_newton(k, dF);
        dx = kmul(k, F, idF);
        err = kmul(k, kmul(k, kmul(k, 0.5, fabs(ddF)), idF), kmul(k, dx, dx));
      }
      x = ksub(k, x, dx);
      it++;
      const double adx = fabs(dx), ax = fabs(x);
      if (nonneg_lt(err, kmul(k, 1e-16, ax)) || !nonneg_lt(1e-14, adx) || !nonneg_lt(kmul(k, 1e-14, ax), adx))
        done = true;
    }
  }
  iters = it;
  if (!on) return true;
  if (!done) return false;
  const double d = -dx;  // last iterate -> root
  if (nonneg_lt(fabs(d), 1e-5) || nonneg_lt(fabs(d), kmul(k, 1e-5, fabs(x)))) {
    const double d2 = kmul(k, kmul(k, 0.5, d), d);        // d^2/2
    const double d3 = kmul(k, kmul(k, d2, d), 1.0 / 3.0);  // d^3/6
    const double aU1 = kmul(k, alpha, U1), aU0 = kmul(k, alpha, U0);
    const double U3n = fma(U0, d3, fma(U1, d2, fma(U2, d, U3)));
    const double U2n = fma(-aU1, d3, fma(U0, d2, fma(U1, d, U2)));
    U1 = fma(-aU0, d3, fma(-aU1, d2, fma(U0, d, U1)));
    U2 = U2n;
    U3 = U3n;
  } else {  // a large last correction: evaluate at the root
    const double xx = x * x;
    const double z = alpha * xx;
    double c2, c3;
    stumpff23(z, c2, c3);
    U1 = x * fma(-z, c3, 1.0);
    U2 = xx * c2;
    U3 = xx * x * c3;
  }
  const double f = fma(-U2, u, 1.0);
  const double g = fma(-U3, K.smuinv, h);
  double rn[3];
#pragma unroll
  for (int c = 0; c < 3; c++) rn[c] = fma(f, r[c], kmul(k, g, v[c]));
  const double rinv = rsqrt(fma(rn[2], rn[2], fma(rn[1], rn[1], kmul(k, rn[0], rn[0]))));
  const double fd = kmul(k, kmul(k, -K.smu, U1), kmul(k, u, rinv));
  const double gd = fma(-U2, rinv, 1.0);
#pragma unroll
  for (int c = 0; c < 3; c++) {
    v[c] = fma(fd, r[c], kmul(k, gd, v[c]));
    r[c] = rn[c];
  }
  rq = rinv;
  return true;
}

// ---------------------------------------------------------------- drift shared by replicas
// mvs_ff.cuh: the lanes that a warp's groups leave over replicate its first group's lanes through
// the drift, so that its votes stay warp-wide.

// ---------------------------------------------------------------- coordinate maps
// inertial (x, v) of the lane's body -> DH (q, u); all lanes execute
template <int N>
__device__ __forceinline__ void to_dh(const double (&x)[3], const double (&v)[3], double m, double Minv, int b,
                                      int base, double (&q)[3], double (&u)[3]) {
#pragma unroll
  for (int c = 0; c < 3; c++) {
    double X = grp_sum<N>(m * x[c], b, base) * Minv;
    double V = grp_sum<N>(m * v[c], b, base) * Minv;
    double x0 = shfl(x[c], base);
    q[c] = b == 0 ? X : x[c] - x0;
    u[c] = b == 0 ? V : v[c] - V;
  }
}

template <int N>
__device__ __forceinline__ void from_dh(const double (&q)[3], const double (&u)[3], double m, double m0,
                                        double Minv, int b, int base, double (&x)[3], double (&v)[3]) {
#pragma unroll
  for (int c = 0; c < 3; c++) {
    double sq = grp_sum<N>(b == 0 ? 0.0 : m * q[c], b, base);
    double su = grp_sum<N>(b == 0 ? 0.0 : m * u[c], b, base);
    double X = shfl(q[c], base), V = shfl(u[c], base);
    double x0 = X - sq * Minv;
    double v0 = V - su / m0;
    x[c] = b == 0 ? x0 : q[c] + x0;
    v[c] = b == 0 ? v0 : u[c] + V;
  }
}

// Jacobi: r'_b = x_b - (sum_{k<b} m_k x_k)/eta_{b-1}; r'_0 = centre of mass
template <int N>
__device__ __forceinline__ void to_jacobi(const double (&x)[3], const double (&v)[3], double m, double Minv,
                                          double eta_prev_inv, int b, int base, double (&q)[3], double (&u)[3]) {
#pragma unroll
  for (int c = 0; c < 3; c++) {
    double px = grp_scan_excl<N>(m * x[c], b);
    double pv = grp_scan_excl<N>(m * v[c], b);
    double X = grp_sum<N>(m * x[c], b, base) * Minv;
    double V = grp_sum<N>(m * v[c], b, base) * Minv;
    q[c] = b == 0 ? X : x[c] - px * eta_prev_inv;
    u[c] = b == 0 ? V : v[c] - pv * eta_prev_inv;
  }
}

// x_b = r'_b + CoM - sum_{k>=b} w_k r'_k (b >= 1), x_0 = CoM - sum_{k>=1} w_k r'_k,
// w_k = m_k / eta_k
template <int N>
__device__ __forceinline__ void from_jacobi(const double (&q)[3], const double (&u)[3], double w, int b, int base,
                                            double (&x)[3], double (&v)[3]) {
#pragma unroll
  for (int c = 0; c < 3; c++) {
    double cq = b == 0 ? 0.0 : w * q[c];
    double cu = b == 0 ? 0.0 : w * u[c];
    double sq = grp_suffix_excl<N>(cq, b) + cq;  // inclusive suffix from b
    double su = grp_suffix_excl<N>(cu, b) + cu;
    double s1q = shfl(sq, base + 1), s1u = shfl(su, base + 1);
    double X = shfl(q[c], base), V = shfl(u[c], base);
    x[c] = b == 0 ? X - s1q : q[c] + X - sq;
    v[c] = b == 0 ? V - s1u : u[c] + V - su;
  }
}

// heliocentric positions from Jacobi ones: Q_b = r'_b + sum_{1<=k<b} w_k r'_k, Q_0 = 0
template <int N>
__device__ __forceinline__ void jacobi_helio(const F64k &k, const double (&q)[3], double w, int b, double (&Q)[3]) {
#pragma unroll
  for (int c = 0; c < 3; c++) {
    double pre = grp_scan_excl<N>(k, b == 0 ? 0.0 : kmul(k, w, q[c]), b);
    Q[c] = b == 0 ? 0.0 : kadd(k, q[c], pre);
  }
}

// Interaction acceleration in FP64.  DH: planet-planet terms (Sec. 2.2.3).  Jacobi: Jacobi
// components of all pair accelerations plus mu_b r'_b/|r'_b|^3.
template <int N, bool JAC>
__device__ __forceinline__ void mvs_acc(const F64k &fk, const double (&q)[3], double m, double w, double eta_prev_inv,
                                        double mu, int b, int base, double (&acc)[3]) {
  double d2[ARing<(JAC ? N : N - 1)>::RTA];
  if constexpr (!JAC) {
    ring_acc<N - 1, 1>(fk, q, m, b == 0 ? 0 : b - 1, base, acc, d2);
#pragma unroll
    for (int c = 0; c < 3; c++)
      if (b == 0) acc[c] = 0.0;
  } else {
    double Q[3], a[3];
    jacobi_helio<N>(fk, q, w, b, Q);
    ring_acc<N, 0>(fk, Q, m, b, base, a, d2);
    const double iq = rsqrt(fma(q[2], q[2], fma(q[1], q[1], kmul(fk, q[0], q[0]))));
    const double k = kmul(fk, kmul(fk, kmul(fk, mu, iq), iq), iq);
#pragma unroll
    for (int c = 0; c < 3; c++) {
      double pre = grp_scan_excl<N>(fk, kmul(fk, m, a[c]), b);
      acc[c] = b == 0 ? 0.0 : fma(-pre, eta_prev_inv, fma(k, q[c], a[c]));
    }
  }
}

}  // namespace swarm
