// Runge-Kutta Cash-Karp 4(5) (Sec. 2.2.2, Sec. 4.3.3) on sm_103a, body per lane.
//
// y = (x, v), dy/dt = (v, a(x)) with a from Eq. 1 (acceleration only, no jerk).  Six
// stages per step; the 5th-order solution is propagated and the difference to the
// embedded 4th-order solution is the error estimate of the adaptive version.  The
// acceleration at the accepted state is the next step's first stage and gives the
// monitor its pair distances, so a step costs six force evaluations.
//
// Lane b of a group holds body b: its stage velocities and accelerations stay in
// registers (11 vectors); pair terms are exchanged with warp shuffles (ring_acc).
#pragma once
#include "mvs_impl.cuh"

namespace swarm {

// The embedded pair of Cash & Karp, ACM TOMS 16 (1990) 201: stage coefficients A, the
// 5th-order weights B5 and the differences E = B5 - B4 to the 4th-order weights.
struct CK {
  static constexpr double A21 = 1.0 / 5.0;
  static constexpr double A31 = 3.0 / 40.0, A32 = 9.0 / 40.0;
  static constexpr double A41 = 3.0 / 10.0, A42 = -9.0 / 10.0, A43 = 6.0 / 5.0;
  static constexpr double A51 = -11.0 / 54.0, A52 = 5.0 / 2.0, A53 = -70.0 / 27.0, A54 = 35.0 / 27.0;
  static constexpr double A61 = 1631.0 / 55296.0, A62 = 175.0 / 512.0, A63 = 575.0 / 13824.0,
                          A64 = 44275.0 / 110592.0, A65 = 253.0 / 4096.0;
  static constexpr double B1 = 37.0 / 378.0, B3 = 250.0 / 621.0, B4 = 125.0 / 594.0, B6 = 512.0 / 1771.0;
  static constexpr double E1 = 37.0 / 378.0 - 2825.0 / 27648.0, E3 = 250.0 / 621.0 - 18575.0 / 48384.0,
                          E4 = 125.0 / 594.0 - 13525.0 / 55296.0, E5 = -277.0 / 14336.0,
                          E6 = 512.0 / 1771.0 - 1.0 / 4.0;
};

constexpr int kRkckTrialCap = 1 << 24;

// group maximum of non-negative values, broadcast to every lane of the group
template <int N>
__device__ __forceinline__ double grp_max(double val, int b, int base) {
#pragma unroll
  for (int off = 1; off < N; off <<= 1) {
    double o = __shfl_down_sync(0xffffffffu, val, off);
    if (b + off < N) val = fmax(val, o);
  }
  return shfl(val, base);
}

// e^(-1/10) (the step-control factor err^(-1/5) from the squared error e = err^2): a
// single-precision estimate, relative error d ~ 1e-7, refined by one Newton step on
// y^-10 = e (y <- y (11 - e y^10) / 10), which leaves 5.5 d^2 ~ 1e-12; e in [1e-30, 1e30].
__device__ __forceinline__ double inv_tenth_root(double e) {
  const float yf = exp2f(-0.1f * log2f((float)e));
  const double y = (double)yf;
  const double y2 = y * y;
  const double y4 = y2 * y2;
  const double y10 = y4 * y4 * y2;
  return y * fma(-e, y10, 11.0) * 0.1;
}

// Squared scaled error of a trial, (err / eps)^2 with err = max_b max(|ex_b| / X, |ev_b| / V):
// from the squared norms, one division and no square root.
__device__ __forceinline__ double rk_err2(double px, double pv, double X2, double V2, double inv_eps2) {
  const double inv = 1.0 / (X2 * V2);
  return fmax(px * (V2 * inv), pv * (X2 * inv)) * inv_eps2;
}

// The same stages in Nystrom form.  For y' = (v, a(x)) the stage positions need no stage
// velocities: with v_j = v + h sum_l A_jl a_l,
//   x_i = x + c_i h v + h^2 sum_l Abar_il a_l,     Abar = A A,  c_i = sum_j A_ij,
//   x5  = x + h v + h^2 sum_l Bbar_l a_l,          Bbar = B5 A,
//   ex  = h^2 sum_l Ebar_l a_l,                    Ebar = (B5 - B4) A  (sum_j E_j = 0),
//   v5  = v + h sum_j B5_j a_j,   ev = h sum_j E_j a_j.
// Exact rational products of the tableau above (Abar_32, Bbar_2, Bbar_6, Ebar_2 vanish).
struct CKN {
  static constexpr double C2 = 1.0 / 5.0, C3 = 3.0 / 10.0, C4 = 3.0 / 5.0, C6 = 7.0 / 8.0;
  static constexpr double A31 = 9.0 / 200.0;
  static constexpr double A41 = -9.0 / 100.0, A42 = 27.0 / 100.0;
  static constexpr double A51 = 25.0 / 36.0, A52 = -7.0 / 4.0, A53 = 14.0 / 9.0;
  static constexpr double A61 = 4949.0 / 27648.0, A62 = -805.0 / 4096.0, A63 = 8855.0 / 27648.0,
                          A64 = 8855.0 / 110592.0;
  static constexpr double B1 = 11.0 / 108.0, B3 = 50.0 / 189.0, B4 = 25.0 / 216.0, B5 = 1.0 / 56.0;
  static constexpr double E1 = -277.0 / 73728.0, E3 = 1385.0 / 129024.0, E4 = -1385.0 / 147456.0,
                          E5 = 277.0 / 114688.0;
};

// One Cash-Karp step of length h from (x, v) with first-stage acceleration a1: writes
// the 5th-order solution and, when E is true, the error vector (5th minus 4th order).
// acc(xs, a) evaluates the accelerations at the stage positions xs.
template <bool E, class Acc>
__device__ __forceinline__ void rkck_step(const F64k &k, const double (&x)[3], const double (&v)[3],
                                          const double (&a1)[3], double h, Acc &&acc, double (&x5)[3],
                                          double (&v5)[3], double (&ex)[3], double (&ev)[3]) {
  double a2[3], a3[3], a4[3], a5[3], a6[3], xs[3];
  const double h2 = kmul(k, h, h);
  const double hc2 = kmul(k, CKN::C2, h), hc3 = kmul(k, CKN::C3, h), hc4 = kmul(k, CKN::C4, h),
               hc6 = kmul(k, CKN::C6, h);
#pragma unroll
  for (int c = 0; c < 3; c++) xs[c] = fma(hc2, v[c], x[c]);
  acc(xs, a2);
#pragma unroll
  for (int c = 0; c < 3; c++) xs[c] = fma(hc3, v[c], fma(h2, kmul(k, CKN::A31, a1[c]), x[c]));
  acc(xs, a3);
#pragma unroll
  for (int c = 0; c < 3; c++) xs[c] = fma(hc4, v[c], fma(h2, fma(CKN::A42, a2[c], kmul(k, CKN::A41, a1[c])), x[c]));
  acc(xs, a4);
#pragma unroll
  for (int c = 0; c < 3; c++)
    xs[c] = fma(h, v[c], fma(h2, fma(CKN::A53, a3[c], fma(CKN::A52, a2[c], kmul(k, CKN::A51, a1[c]))), x[c]));
  acc(xs, a5);
#pragma unroll
  for (int c = 0; c < 3; c++)
    xs[c] = fma(hc6, v[c],
                fma(h2, fma(CKN::A64, a4[c], fma(CKN::A63, a3[c], fma(CKN::A62, a2[c], kmul(k, CKN::A61, a1[c])))),
                    x[c]));
  acc(xs, a6);
#pragma unroll
  for (int c = 0; c < 3; c++) {
    x5[c] = fma(h, v[c],
                fma(h2, fma(CKN::B5, a5[c], fma(CKN::B4, a4[c], fma(CKN::B3, a3[c], kmul(k, CKN::B1, a1[c])))), x[c]));
    v5[c] = fma(h, fma(CK::B6, a6[c], fma(CK::B4, a4[c], fma(CK::B3, a3[c], kmul(k, CK::B1, a1[c])))), v[c]);
    if (E) {
      ex[c] = kmul(k, h2, fma(CKN::E5, a5[c], fma(CKN::E4, a4[c], fma(CKN::E3, a3[c], kmul(k, CKN::E1, a1[c])))));
      ev[c] = kmul(k, h, fma(CK::E6, a6[c], fma(CK::E5, a5[c], fma(CK::E4, a4[c], fma(CK::E3, a3[c], kmul(k, CK::E1, a1[c]))))));
    }
  }
}

template <int N, bool E>
__device__ __forceinline__ void rkck_stages(const F64k &k, const double (&x)[3], const double (&v)[3], const double (&a1)[3],
                                            double m, int b, int base, double h, double (&x5)[3], double (&v5)[3],
                                            double (&ex)[3], double (&ev)[3]) {
  double d2[ARing<N>::RTA];
  rkck_step<E>(k, x, v, a1, h, [&](const double (&xs)[3], double (&a)[3]) { ring_acc<N, 0>(k, xs, m, b, base, a, d2); },
               x5, v5, ex, ev);
}

// ---------------------------------------------------------------- system per lane
// Accelerations (Eq. 1) of bodies k = 1..N-1 relative to body 0 from X_k = x_k - x_0:
//   A_k = -m_0 s_k X_k - a_0 + sum_{i >= 1, i != k} m_i s_ik (X_i - X_k),
//   a_0 = sum_{j >= 1} m_j s_j X_j  (stored in A[0]),  s = 1/r^3;
// monitor distances q2[k] = |X_k|^2, d2[i][k] = |X_k - X_i|^2.
template <int N>
__device__ __forceinline__ void spl_acc_rel(const F64k &kk, const double (&X)[N][3], const double (&m)[N],
                                            double (&A)[N][3], double (&q2)[N], double (&d2)[N][N]) {
  double m0s[N];
#pragma unroll
  for (int k = 1; k < N; k++) {
    double r2 = kmul(kk, X[k][0], X[k][0]);
    r2 = fma(X[k][1], X[k][1], r2);
    r2 = fma(X[k][2], X[k][2], r2);
    const double rho = rsqrt(r2);
    const double s3 = kmul(kk, kmul(kk, rho, rho), rho);
    const double ms = kmul(kk, m[k], s3);
    m0s[k] = kmul(kk, m[0], s3);
    q2[k] = r2;
#pragma unroll
    for (int c = 0; c < 3; c++) A[0][c] = k == 1 ? kmul(kk, ms, X[k][c]) : fma(ms, X[k][c], A[0][c]);
  }
#pragma unroll
  for (int k = 1; k < N; k++)
#pragma unroll
    for (int c = 0; c < 3; c++) A[k][c] = fma(-m0s[k], X[k][c], -A[0][c]);
#pragma unroll
  for (int i = 1; i < N; i++)
#pragma unroll
    for (int k = i + 1; k < N; k++) {
      double dx[3];
#pragma unroll
      for (int c = 0; c < 3; c++) dx[c] = ksub(kk, X[k][c], X[i][c]);
      double r2 = kmul(kk, dx[0], dx[0]);
      r2 = fma(dx[1], dx[1], r2);
      r2 = fma(dx[2], dx[2], r2);
      const double rho = rsqrt(r2);
      const double s3 = kmul(kk, kmul(kk, rho, rho), rho);
      const double sk = kmul(kk, m[k], s3), si = kmul(kk, m[i], s3);
#pragma unroll
      for (int c = 0; c < 3; c++) {
        A[i][c] = fma(sk, dx[c], A[i][c]);
        A[k][c] = fma(-si, dx[c], A[k][c]);
      }
      d2[i][k] = r2;
    }
}

// One Cash-Karp step (Nystrom form, see rkck_step) of every relative body of a lane's
// system; with E also the error vectors, body 0's included (index 0: its velocity error
// from its stage accelerations a_0, its position error -sum_k m_k ex_k / M from the
// barycentre's fixed velocity, since sum_s (b5 - b4)_s = 0).  The monitor distances of
// the last stage are discarded; the caller evaluates the accepted state.
template <int N, bool E>
__device__ __forceinline__ void spl_rkck_step(const F64k &k, const double (&x)[N][3], const double (&v)[N][3],
                                              const double (&a1)[N][3], const double (&m)[N], double Minv,
                                              double h, double (&x5)[N][3], double (&v5)[N][3],
                                              double (&ex)[N][3], double (&ev)[N][3]) {
  double a2[N][3], a3[N][3], a4[N][3], a5[N][3], a6[N][3], xs[N][3], q2[N], d2[N][N];
  const double h2 = kmul(k, h, h);
  const double hc2 = kmul(k, CKN::C2, h), hc3 = kmul(k, CKN::C3, h), hc4 = kmul(k, CKN::C4, h),
               hc6 = kmul(k, CKN::C6, h);
#pragma unroll
  for (int i = 1; i < N; i++)
#pragma unroll
    for (int c = 0; c < 3; c++) xs[i][c] = fma(hc2, v[i][c], x[i][c]);
  spl_acc_rel<N>(k, xs, m, a2, q2, d2);
#pragma unroll
  for (int i = 1; i < N; i++)
#pragma unroll
    for (int c = 0; c < 3; c++) xs[i][c] = fma(hc3, v[i][c], fma(h2, kmul(k, CKN::A31, a1[i][c]), x[i][c]));
  spl_acc_rel<N>(k, xs, m, a3, q2, d2);
#pragma unroll
  for (int i = 1; i < N; i++)
#pragma unroll
    for (int c = 0; c < 3; c++)
      xs[i][c] = fma(hc4, v[i][c], fma(h2, fma(CKN::A42, a2[i][c], kmul(k, CKN::A41, a1[i][c])), x[i][c]));
  spl_acc_rel<N>(k, xs, m, a4, q2, d2);
#pragma unroll
  for (int i = 1; i < N; i++)
#pragma unroll
    for (int c = 0; c < 3; c++)
      xs[i][c] = fma(h, v[i][c],
                     fma(h2, fma(CKN::A53, a3[i][c], fma(CKN::A52, a2[i][c], kmul(k, CKN::A51, a1[i][c]))), x[i][c]));
  spl_acc_rel<N>(k, xs, m, a5, q2, d2);
#pragma unroll
  for (int i = 1; i < N; i++)
#pragma unroll
    for (int c = 0; c < 3; c++)
      xs[i][c] = fma(hc6, v[i][c],
                     fma(h2,
                         fma(CKN::A64, a4[i][c],
                             fma(CKN::A63, a3[i][c], fma(CKN::A62, a2[i][c], kmul(k, CKN::A61, a1[i][c])))),
                         x[i][c]));
  spl_acc_rel<N>(k, xs, m, a6, q2, d2);
#pragma unroll
  for (int i = 1; i < N; i++)
#pragma unroll
    for (int c = 0; c < 3; c++) {
      x5[i][c] = fma(h, v[i][c],
                     fma(h2, fma(CKN::B5, a5[i][c], fma(CKN::B4, a4[i][c], fma(CKN::B3, a3[i][c], kmul(k, CKN::B1, a1[i][c])))),
                         x[i][c]));
      v5[i][c] = fma(h, fma(CK::B6, a6[i][c], fma(CK::B4, a4[i][c], fma(CK::B3, a3[i][c], kmul(k, CK::B1, a1[i][c])))),
                     v[i][c]);
    }
  if (E) {
#pragma unroll
    for (int i = 0; i < N; i++)
#pragma unroll
      for (int c = 0; c < 3; c++) {
        if (i > 0)
          ex[i][c] = kmul(k, h2, fma(CKN::E5, a5[i][c], fma(CKN::E4, a4[i][c], fma(CKN::E3, a3[i][c], kmul(k, CKN::E1, a1[i][c])))));
        ev[i][c] = kmul(k, h, fma(CK::E6, a6[i][c], fma(CK::E5, a5[i][c], fma(CK::E4, a4[i][c], fma(CK::E3, a3[i][c], kmul(k, CK::E1, a1[i][c]))))));
      }
#pragma unroll
    for (int c = 0; c < 3; c++) {
      double sx = 0.0;
#pragma unroll
      for (int i = 1; i < N; i++) sx = fma(m[i], ex[i][c], sx);
      ex[0][c] = kmul(k, -sx, Minv);
    }
  }
}

}  // namespace swarm
