// Runge-Kutta Cash-Karp steps (Sec. 2.2.2) with the FP64 pipe kept for what needs it, as in
// hermite_ff.cuh: the state's sums, h v, h a_1 and body 0's pull are FP64, the rest float pairs.
//
// With D_j = a_j - a_1 (~ c_j eta a for eta = h omega) and the tableau's row sums (sum B5 = 1,
// sum_l Abar_il = c_i^2/2, sum Bbar = 1/2, sum E = sum Ebar = 0) the step reads
//   x_i = x + c_i h v + h^2 (c_i^2/2 a_1 + sum_{l>=2} Abar_il D_l),
//   x5  = x + h v + h^2 (a_1/2 + sum Bbar_l D_l),   v5 = v + h a_1 + h sum B5_j D_j,
//   ex  = h^2 sum Ebar_l D_l,                       ev = h sum E_j D_j.
// The star's part of D_j is one DFMA, -M_j X_j + M_1 X_1, so a pair holds it to 2^-48 eta of a:
// the level of the FP64 stages' own rounding, also for the error vectors, in which the a_1
// cancel.  Stages whose weight in v5 (and E, where it is formed) is zero enter with h^2 only and
// are pairs altogether.  Checked at every state (`rk_guard`): eta <= 1/8, perturbations
// h a_pert/v <= 2^-8 of their rounding; else the step is FP64.
//
// n = 3: 190 FP64 instructions per adaptive step instead of 640.
#pragma once
#include "hermite_bpl_ff.cuh"
#include "rkck_impl.cuh"

namespace swarm {

// sum of constants times pairs
__device__ __forceinline__ ff ff_lin(double c, const ff &a) { return ff_mul_raw(ff_const(c), a); }
__device__ __forceinline__ ff ff_lin(double c, const ff &a, const ff &s) { return ff_fma_raw(ff_const(c), a, s); }

struct RkStep {
  double h, hc3, hc4, hc6;
  ff f, h2;
  float fl;  // what f leaves of h
};
__device__ __forceinline__ RkStep rk_step(const F64k &k, double h) {
  RkStep R;
  R.h = h;
  R.hc3 = kmul(k, CKN::C3, h);
  R.hc4 = kmul(k, CKN::C4, h);
  R.hc6 = kmul(k, CKN::C6, h);
  const ff3 h3 = ff3_from(h);
  R.f = ff_norm(ff_make(h3.h, h3.l));
  R.fl = h3.t;
  R.h2 = ff_mul(R.f, R.f);
  return R;
}
// h times a pair.  The third part of h (up to 2^-48 of it) is the same at every fixed step, and left
// out it adds up like a change of the step's length: at 60 steps an orbit, where h is such a number,
// 200 steps of two bodies ended 6.2e-14 from quadruple precision instead of FP64's 3.2e-14.
__device__ __forceinline__ ff rk_hmul(const RkStep &R, const ff &a) {
  const ff p = ff_mul_raw(R.f, a);
  return ff_norm(ff_make(p.h, __fmaf_rn(R.fl, a.h, p.l)));
}
// Per component, from a = a_1 and the D_j: what a stage adds to v in x_i = x + c_i h (v + w_i)
// and the result in x5 = x + h (v + w): one rounding of x, and v + w's is taken by c_i h.
__device__ __forceinline__ ff rk_w3(const RkStep &R, const ff &a) { return rk_hmul(R, ff_lin(0.5 * CKN::C3, a)); }
__device__ __forceinline__ ff rk_w4(const RkStep &R, const ff &a, const ff &d2) {
  return rk_hmul(R, ff_lin(CKN::A42 / CKN::C4, d2, ff_lin(0.5 * CKN::C4, a)));
}
__device__ __forceinline__ ff rk_w5(const RkStep &R, const ff &a, const ff &d2, const ff &d3) {
  return rk_hmul(R, ff_lin(CKN::A53, d3, ff_lin(CKN::A52, d2, ff_lin(0.5, a))));
}
__device__ __forceinline__ ff rk_w6(const RkStep &R, const ff &a, const ff &d2, const ff &d3, const ff &d4) {
  return rk_hmul(R, ff_lin(CKN::A64 / CKN::C6, d4, ff_lin(CKN::A63 / CKN::C6, d3, ff_lin(CKN::A62 / CKN::C6, d2, ff_lin(0.5 * CKN::C6, a)))));
}
__device__ __forceinline__ ff rk_wx(const RkStep &R, const ff &a, const ff &d3, const ff &d4, const ff &d5) {
  return rk_hmul(R, ff_lin(CKN::B5, d5, ff_lin(CKN::B4, d4, ff_lin(CKN::B3, d3, ff_lin(0.5, a)))));
}
// and v5 = v + h (S1 + this)
__device__ __forceinline__ ff rk_av(const ff &p1, const ff &d3, const ff &d4, const ff &d6) {
  return ff_norm(ff_lin(CK::B6, d6, ff_lin(CK::B4, d4, ff_lin(CK::B3, d3, p1))));
}
__device__ __forceinline__ ff rk_ex(const RkStep &R, const ff &d3, const ff &d4, const ff &d5) {
  return ff_norm(ff_mul_raw(R.h2, ff_lin(CKN::E5, d5, ff_lin(CKN::E4, d4, ff_lin(CKN::E3, d3)))));
}
__device__ __forceinline__ ff rk_ev(const RkStep &R, const ff &d3, const ff &d4, const ff &d5, const ff &d6) {
  return ff_norm(ff_mul_raw(R.f, ff_lin(CK::E6, d6, ff_lin(CK::E5, d5, ff_lin(CK::E4, d4, ff_lin(CK::E3, d3))))));
}

// e1 = mu/r^3 and sv = (S/v)^2 (see fguard) of a state, largest over its planets; h the step
__device__ __forceinline__ bool rk_guard(double h, float e1, float sv) {
  const float hf = f_from(h), h2 = hf * hf;
  return h2 * e1 <= 0x1p-6f && h2 * sv <= 0x1p-16f && fscale(h, -40, 60);
}
// max of two non-negative pairs
__device__ __forceinline__ ff ff_max(const ff &a, const ff &b) {
  return ff_sel(a.h > b.h || (a.h == b.h && a.l > b.l), a, b);
}
// 0.9 e^(-1/10) (step control from the squared scaled error e): see inv_tenth_root
__device__ __forceinline__ ff rk_factor(const ff &e) {
  const float y = exp2f(-0.1f * log2f(e.h));
  const ff y2 = two_prod(y, y);
  const ff y4 = ff_mul(y2, y2);
  const ff r = ff_mul(e, ff_mul(ff_mul(y4, y4), y2));
  const float d = __fsub_rn(__fsub_rn(1.0f, r.h), r.l);
  return ff_mul(ff_const(0.9), fast_two_sum(y, __fmul_rn(__fmul_rn(0.1f, y), d)));
}
// the length after a trial of |hs| whose squared scaled error is e (0.2 <= ratio <= 5)
__device__ __forceinline__ double rk_next_h(double hs, const ff &e, bool accept) {
  if (e.h <= 1e-18f) return 5.0 * hs;  // (0.9 e^(-1/10) > 5)
  const ff f = rk_factor(e);
  if (f.h <= 0.2f) return 0.2 * hs;
  if (accept && f.h >= 5.0f) return 5.0 * hs;
  return ff_double(f) * hs;
}

// ---------------------------------------------------------------- system per lane
template <int N>
struct SplAcc {
  double M[N];
  ff P[N][3], I[3];  // I: body 0's acceleration
  float q2[N], d2[N][N], e1, sv;
  bool range;
};
// V: velocities, for the guard (STATE)
template <int N, bool STATE>
__device__ __forceinline__ void spl_acc_full(const F64k &kk, const FMass<N> &F, const double (&X)[N][3],
                                             const double (&v)[N][3], SplAcc<N> &R) {
  ff Xf[N][3], T[N][3], Q[N][3];
  SplGeo<N> g;
  float r0[N];
#pragma unroll
  for (int k = 1; k < N; k++) {
    ff rho3, rho2;
    float rho;
    double q2;
    star_pull(kk, X[k], F.mu[k], R.M[k], q2, rho3, rho2, rho);
    R.q2[k] = f_from(q2);
    r0[k] = R.q2[k] * rho;
    g.s[0][k] = rho3.h;
    g.p[0][k] = rho2.h;
#pragma unroll
    for (int c = 0; c < 3; c++) {
      Xf[k][c] = ff_from(X[k][c]);
      T[k][c] = ff_mul_raw(rho3, Xf[k][c]);
    }
  }
  spl_pert<N, 0>(F, Xf, Xf, T, T, R.P, Q, R.d2, g);
#pragma unroll
  for (int c = 0; c < 3; c++) {
    R.I[c] = ff_mul_raw(F.m[1], T[1][c]);
#pragma unroll
    for (int k = 2; k < N; k++) R.I[c] = ff_fma_raw(F.m[k], T[k][c], R.I[c]);
#pragma unroll
    for (int k = 1; k < N; k++) R.P[k][c] = ff_norm(R.P[k][c]);
  }
  if (STATE) {
    R.range = F.ok;
    R.e1 = R.sv = 0.0f;
#pragma unroll
    for (int k = 1; k < N; k++) {
      float S = 0.0f;
#pragma unroll
      for (int j = 1; j < N; j++)
        if (j != k) {
          R.range = R.range && frange(j < k ? R.d2[j][k] : R.d2[k][j]);
          S = __fmaf_rn(F.m[j].h, __fmaf_rn(j < k ? g.s[j][k] : g.s[k][j], r0[k] + r0[j], g.p[0][j]), S);
        }
      const float a = f_from(v[k][0]), b = f_from(v[k][1]), c = f_from(v[k][2]);
      const float V2 = __fmaf_rn(c, c, __fmaf_rn(b, b, __fmul_rn(a, a)));
      R.range = R.range && ff_tame(X[k], v[k]) && frange(R.q2[k]) && V2 < 0x1p80f && V2 > 0x1p-80f;
      R.e1 = fmaxf(R.e1, F.muf[k].h * g.s[0][k]);
      R.sv = fmaxf(R.sv, S * S / V2);
    }
  }
}
template <int N>
__device__ __forceinline__ void spl_acc_ff(const FMass<N> &F, const ff (&X)[N][3], ff (&A)[N][3]) {
  ff T[N][3], Q[N][3];
  SplGeo<N> g;
  float d2[N][N];
#pragma unroll
  for (int k = 1; k < N; k++) {
    ff rho3, rho2;
    ff_rho3(ff_norm2(X[k]), rho3, rho2);
#pragma unroll
    for (int c = 0; c < 3; c++) T[k][c] = ff_mul_raw(rho3, X[k][c]);
  }
  spl_pert<N, 0>(F, X, X, T, T, A, Q, d2, g);
#pragma unroll
  for (int k = 1; k < N; k++)
#pragma unroll
    for (int c = 0; c < 3; c++) A[k][c] = ff_fma(ff_neg(F.muf[k]), T[k][c], A[k][c]);
}

// One step of length h from (x, v) with the first stage's S1 = -M X (FP64), P1 (perturbations)
// and I1 (body 0's acceleration): the new x, v and (E) the relative error vectors, index 0 body
// 0's velocity error.
template <int N, bool E>
__device__ __forceinline__ void spl_rkck_ff_step(const F64k &kk, const FMass<N> &F, double h, const double (&x)[N][3],
                                                 const double (&v)[N][3], const double (&S1)[N][3],
                                                 const ff (&P1)[N][3], const ff (&I1)[3], double (&x5)[N][3],
                                                 double (&v5)[N][3], ff (&ex)[N][3], ff (&ev)[N][3]) {
  const RkStep R = rk_step(kk, h);
  ff a[N][3], D2[N][3], D3[N][3], D4[N][3], D5[N][3], D6[N][3], Xf[N][3];
  double xs[N][3];
  SplAcc<N> A;
  auto diff = [&](ff (&D)[N][3]) {  // evaluation at xs
    spl_acc_full<N, false>(kk, F, xs, v, A);
#pragma unroll
    for (int k = 1; k < N; k++)
#pragma unroll
      for (int c = 0; c < 3; c++)
        D[k][c] = ff_norm(ff_add_raw(ff_from(fma(-A.M[k], xs[k][c], -S1[k][c])), ff_sub_raw(A.P[k][c], P1[k][c])));
    if (E)
#pragma unroll
      for (int c = 0; c < 3; c++) D[0][c] = ff_norm(ff_sub_raw(A.I[c], I1[c]));
  };
#pragma unroll
  for (int k = 1; k < N; k++)
#pragma unroll
    for (int c = 0; c < 3; c++) {
      a[k][c] = ff_norm(ff_add_raw(ff_from(S1[k][c]), P1[k][c]));
      Xf[k][c] = ff_norm(ff_fma_raw(ff_lin(CKN::C2, R.f), ff_from(v[k][c]), ff_from(x[k][c])));
    }
  spl_acc_ff<N>(F, Xf, D2);
#pragma unroll
  for (int k = 1; k < N; k++)
#pragma unroll
    for (int c = 0; c < 3; c++) D2[k][c] = ff_sub(D2[k][c], a[k][c]);
  // The stages 3..6.  Adaptive trials: as a loop with one copy of the evaluation, since a trial with
  // the step control around it is 120 KB of instructions unrolled and waits for them half its
  // time (20000 x 3 systems: 11.7 -> 9.8 ms).  Fixed steps fit the cache better and are faster
  // unrolled (20000 x 3, 100 steps: 1.28 ms, as a loop 1.70).
  auto stage = [&](int st) {
    ff w[N][3];
    auto each = [&](auto f) {
#pragma unroll
      for (int k = 1; k < N; k++)
#pragma unroll
        for (int c = 0; c < 3; c++) w[k][c] = f(k, c);
    };
    double hc = R.h;
    if (st == 3) {
      hc = R.hc3;
      each([&](int k, int c) { return rk_w3(R, a[k][c]); });
    } else if (st == 4) {
      hc = R.hc4;
      each([&](int k, int c) { return rk_w4(R, a[k][c], D2[k][c]); });
    } else if (st == 5) {
      each([&](int k, int c) { return rk_w5(R, a[k][c], D2[k][c], D3[k][c]); });
    } else {
      hc = R.hc6;
      each([&](int k, int c) { return rk_w6(R, a[k][c], D2[k][c], D3[k][c], D4[k][c]); });
    }
#pragma unroll
    for (int k = 1; k < N; k++)
#pragma unroll
      for (int c = 0; c < 3; c++) {
        xs[k][c] = fma(hc, ff_addto(v[k][c], w[k][c]), x[k][c]);
        if (!E) Xf[k][c] = ff_norm(ff_fma_raw(R.f, ff_add(ff_from(v[k][c]), w[k][c]), ff_from(x[k][c])));
      }
    if (E || st != 5) {
      diff(w);
    } else {
      spl_acc_ff<N>(F, Xf, w);
#pragma unroll
      for (int k = 1; k < N; k++)
#pragma unroll
        for (int c = 0; c < 3; c++) w[k][c] = ff_sub(w[k][c], a[k][c]);
    }
#pragma unroll
    for (int k = E ? 0 : 1; k < N; k++)
#pragma unroll
      for (int c = 0; c < 3; c++) {
        if (st == 3) D3[k][c] = w[k][c];
        else if (st == 4) D4[k][c] = w[k][c];
        else if (st == 5) D5[k][c] = w[k][c];
        else D6[k][c] = w[k][c];
      }
  };
  if (E) {
#pragma unroll 1
    for (int st = 3; st <= 6; st++) stage(st);
  } else {
    stage(3);
    stage(4);
    stage(5);
    stage(6);
  }
#pragma unroll
  for (int k = 1; k < N; k++)
#pragma unroll
    for (int c = 0; c < 3; c++)
      x5[k][c] = fma(R.h, ff_addto(v[k][c], rk_wx(R, a[k][c], D3[k][c], D4[k][c], D5[k][c])), x[k][c]);
#pragma unroll
  for (int k = 1; k < N; k++)
#pragma unroll
    for (int c = 0; c < 3; c++)
      v5[k][c] = fma(R.h, ff_addto(S1[k][c], rk_av(P1[k][c], D3[k][c], D4[k][c], D6[k][c])), v[k][c]);
  if (E)
#pragma unroll
    for (int k = 0; k < N; k++)
#pragma unroll
      for (int c = 0; c < 3; c++) {
        if (k > 0) ex[k][c] = rk_ex(R, D3[k][c], D4[k][c], D5[k][c]);
        ev[k][c] = rk_ev(R, D3[k][c], D4[k][c], D5[k][c], D6[k][c]);
      }
}

// squared scaled error of a trial (over eps): max over bodies of the inertial error vectors, with
// the largest inertial position and speed at the step's start
template <int N>
__device__ __forceinline__ ff spl_rk_error(const FMass<N> &F, const ff &Minv, const ff &inv_eps, const double (&x)[N][3],
                                           const double (&v)[N][3], const ff (&Xc)[3], const ff (&Vc)[3],
                                           const ff (&ex)[N][3], const ff (&ev)[N][3]) {
  ff x0[3], v0[3], e0[3];
#pragma unroll
  for (int c = 0; c < 3; c++) {
    ff sx = ff_make(0.0f, 0.0f), sv = sx, se = sx;
#pragma unroll
    for (int k = 1; k < N; k++) {
      sx = ff_fma_raw(F.m[k], ff_from(x[k][c]), sx);
      sv = ff_fma_raw(F.m[k], ff_from(v[k][c]), sv);
      se = ff_fma_raw(F.m[k], ex[k][c], se);
    }
    x0[c] = ff_sub(Xc[c], ff_mul(sx, Minv));
    v0[c] = ff_sub(Vc[c], ff_mul(sv, Minv));
    e0[c] = ff_neg(ff_mul(se, Minv));
  }
  ff X2 = ff_norm2(x0), V2 = ff_norm2(v0), pe = ff_make(0.0f, 0.0f), pf = pe;
#pragma unroll
  for (int k = 0; k < N; k++) {
    ff p[3], q[3], e[3], f[3];
#pragma unroll
    for (int c = 0; c < 3; c++) {
      if (k > 0) {
        p[c] = ff_add(ff_from(x[k][c]), x0[c]);
        q[c] = ff_add(ff_from(v[k][c]), v0[c]);
      }
      e[c] = ff_mul(inv_eps, k > 0 ? ff_add(ex[k][c], e0[c]) : e0[c]);
      f[c] = ff_mul(inv_eps, k > 0 ? ff_add(ev[k][c], ev[0][c]) : ev[0][c]);
    }
    if (k > 0) {
      X2 = ff_max(X2, ff_norm2(p));
      V2 = ff_max(V2, ff_norm2(q));
    }
    pe = ff_max(pe, ff_norm2(e));
    pf = ff_max(pf, ff_norm2(f));
  }
  return ff_max(ff_div(pe, X2), ff_div(pf, V2));
}

// A trial wholly in FP64 (guard not met), out of line: the new state and, ADAPT, the squared
// scaled error.
template <int N, bool ADAPT>
static __device__ __noinline__ double spl_rkck_fp64_trial(const F64k &kk, const double (&m)[N], double Minv, double hs,
                                                          double inv_eps2, const double (&x)[N][3],
                                                          const double (&v)[N][3], const double (&Xc)[3],
                                                          const double (&Vc)[3], double (&x5)[N][3],
                                                          double (&v5)[N][3]) {
  double a1[N][3], q2[N], d2[N][N], ex[N][3], ev[N][3], xn[N][3], vn[N][3], err = 0.0;
  spl_acc_rel<N>(kk, x, m, a1, q2, d2);
  spl_rkck_step<N, ADAPT>(kk, x, v, a1, m, Minv, hs, xn, vn, ex, ev);
  if (ADAPT) {
    double xi[N][3], vi[N][3];
    spl_from_rel<N>(m, x, v, Minv, Xc, Vc, xi, vi);
    double X2 = 0.0, V2 = 0.0;
#pragma unroll
    for (int i = 0; i < N; i++) {
      X2 = fmax(X2, fma(xi[i][2], xi[i][2], fma(xi[i][1], xi[i][1], kmul(kk, xi[i][0], xi[i][0]))));
      V2 = fmax(V2, fma(vi[i][2], vi[i][2], fma(vi[i][1], vi[i][1], kmul(kk, vi[i][0], vi[i][0]))));
    }
#pragma unroll
    for (int i = 0; i < N; i++) {
      double e[3], f[3];
#pragma unroll
      for (int c = 0; c < 3; c++) {
        e[c] = i == 0 ? ex[0][c] : kadd(kk, ex[i][c], ex[0][c]);
        f[c] = i == 0 ? ev[0][c] : kadd(kk, ev[i][c], ev[0][c]);
      }
      const double px = fma(e[2], e[2], fma(e[1], e[1], kmul(kk, e[0], e[0])));
      const double pv = fma(f[2], f[2], fma(f[1], f[1], kmul(kk, f[0], f[0])));
      err = fmax(err, rk_err2(px, pv, X2, V2, inv_eps2));
    }
  }
#pragma unroll
  for (int i = 1; i < N; i++)
#pragma unroll
    for (int c = 0; c < 3; c++) {
      x5[i][c] = xn[i][c];
      v5[i][c] = vn[i][c];
    }
  return err;
}

// System per lane (n <= 3), coordinates relative to body 0 plus the barycentre (the
// same method in exact arithmetic: every stage is linear in the state and the stage
// accelerations, and A_k = a_k - a_0), work handed out per lane: a lane whose system
// reached its end time or stopped takes the bin's next one.  Step rules, error norm
// (in inertial coordinates, rebuilt from the relative ones) and step control are those
// of bpl_rkck_stream.
template <int N, bool ADAPT>
__device__ __forceinline__ void spl_rkck_stream(const BinView &B, const StepParams &P) {
  constexpr unsigned long long NP = (unsigned long long)N * (N - 1) / 2;
  const unsigned FULL = 0xffffffffu;
  const int SP = B.S_pad;
  const double dir = P.dt > 0 ? 1.0 : -1.0;
  const int nmax = ADAPT ? (P.max_steps > 0 ? P.max_steps : kRkckTrialCap) : 0;
  const double inv_eps2 = 1.0 / (P.rk_eps * P.rk_eps);
  const bool eps_ok = P.rk_eps > 0x1p-60;
  const ff inv_eps = ff_from(1.0 / P.rk_eps);
  double x[N][3], v[N][3], m[N], S1[N][3];
  ff P1[N][3], I1[3];
  FMass<N> F;
  FLimits<N> L;
  float e1 = 0.0f, sv = 0.0f;
  bool range = false;  // of the state, for rk_guard
  double Minv = 1.0, Xc[3] = {0.0, 0.0, 0.0}, Vc[3] = {0.0, 0.0, 0.0};
  LaunchPlan plan;
  plan.N = 0;
  plan.full = 1;
  plan.exact = 1;
  plan.h_last = P.dt;
  plan.t_end = P.t_end;
  double t = 0.0, t0 = 0.0, te = 0.0, h = fabs(P.dt);
  int s = 0, steps = 0, trials = 0;
  bool has = false, exhausted = false;
  bool fresh = false, at_end = false;  // a state without its evaluation; its time is the end time
  for (;;) {
    if (!has && !exhausted) {
      s = stream_system(B, atomicAdd(P.work_next, 1));
      if (s < 0) {
        exhausted = true;
      } else {
        const bool runnable = B.status[s] <= SWARM_SYS_DONE;
        t0 = B.t[s];
        bool go;
        if (!ADAPT) {
          plan = launch_plan(B, P, s, t0, runnable);
          te = plan.t_end;
          go = runnable && plan.N > 0;
        } else {
          te = adaptive_end(B, P, s);
          go = runnable && ((te - t0) * dir > 1e-12 * fmax(1.0, fabs(te)));
        }
        if (runnable && !go) B.status[s] = SWARM_SYS_DONE;
        if (go) {
#pragma unroll
          for (int i = 0; i < N; i++) {
            m[i] = B.m[(size_t)i * SP + s];
#pragma unroll
            for (int c = 0; c < 3; c++) {
              x[i][c] = B.x[(size_t)(c * N + i) * SP + s];
              v[i][c] = B.v[(size_t)(c * N + i) * SP + s];
            }
          }
          L = flimits<N>(m, P.ce_factor, P.eject2);
          F = fmass<N>(m);
          spl_to_rel<N>(m, x, v, Minv, Xc, Vc);
          t = t0;
          steps = 0;
          trials = 0;
          h = fabs(P.dt);
          has = fresh = true;
          at_end = false;
        }
      }
    }
    bool more = __any_sync(FULL, has || !exhausted);
    if (ADAPT) more = __syncthreads_or(more);  // see spl_hermite_adaptive_run
    if (!more) break;
    // the new states' evaluation (also a refill's: one copy)
    float q2[N], d2[N][N];
    if (fresh) {
      SplAcc<N> A;
      spl_acc_full<N, true>(P.fk, F, x, v, A);
#pragma unroll
      for (int k = 1; k < N; k++) {
        q2[k] = A.q2[k];
#pragma unroll
        for (int c = 0; c < 3; c++) {
          S1[k][c] = kmul(P.fk, -A.M[k], x[k][c]);
          P1[k][c] = A.P[k][c];
          I1[c] = A.I[c];
        }
#pragma unroll
        for (int j = k + 1; j < N; j++) d2[k][j] = A.d2[k][j];
      }
      e1 = A.e1;
      sv = A.sv;
      range = A.range;
    }
    if (!has) continue;
    int code = 0;
    bool reached = false;
    if (fresh && steps > 0) {  // the monitor of the step that led here
      code = spl_ff_monitor<N>(P.fk, range ? 1 : 0, L, q2, d2, x, v, P.eject2);
      reached = !code && at_end;
      if (!ADAPT && (code || reached || (P.log_interval > 0 && (steps % P.log_interval) == 0)))
        t = step_time(plan, steps, t0, P.dt);  // fixed steps: time formed when it is used
      if (P.log_interval > 0 && !code && (steps % P.log_interval) == 0)
        spl_write<N>(B, s, m, x, v, Minv, Xc, Vc, t - t0, &P, t);
    }
    fresh = false;
    bool capped = ADAPT && !code && !reached && trials >= nmax;
    if (!code && !reached && !capped) {
      // ---- one step (or trial)
      double hs;
      bool last;
      if (!ADAPT) {
        last = steps + 1 == plan.N;
        hs = (last && !plan.exact) ? plan.h_last : P.dt;
      } else {
        const double rem = kmul(P.fk, ksub(P.fk, te, t), dir);
        last = __double2hiint(h) >= __double2hiint(rem) && h >= rem;  // (FP64 compares are slow)
        hs = kmul(P.fk, last ? rem : h, dir);
      }
      double x5[N][3], v5[N][3];
      bool accept = true, pairs = range && rk_guard(hs, e1, sv) && (!ADAPT || eps_ok);
      ff err = ff_make(0.0f, 0.0f);  // squared scaled error of the trial
      double err64 = 0.0;
      if (pairs) {
        ff ex[N][3], ev[N][3];
        spl_rkck_ff_step<N, ADAPT>(P.fk, F, hs, x, v, S1, P1, I1, x5, v5, ex, ev);
        if (ADAPT) {
          ff X[3], V[3];
          const ff el = ff_from(t - t0);
#pragma unroll
          for (int c = 0; c < 3; c++) {
            V[c] = ff_norm(ff_from(Vc[c]));
            X[c] = ff_fma(el, V[c], ff_from(Xc[c]));
          }
          err = spl_rk_error<N>(F, ff_from(Minv), inv_eps, x, v, X, V, ex, ev);
          if (!(err.h < 0x1p100f)) pairs = false;  // out of FP32's range: in FP64
        }
      }
      if (!pairs) {
        double X[3];
#pragma unroll
        for (int c = 0; c < 3; c++) X[c] = fma(t - t0, Vc[c], Xc[c]);
        err64 = spl_rkck_fp64_trial<N, ADAPT>(P.fk, m, Minv, hs, inv_eps2, x, v, X, Vc, x5, v5);
      }
      if (ADAPT) {
        bool bad = false;
        if (pairs) {
          accept = err.h < 1.0f || (err.h == 1.0f && err.l <= 0.0f);
        } else {
          bad = nonfinite(err64);
          accept = !bad && err64 <= 1.0;
        }
        trials++;
        if (bad) code = SWARM_SYS_NONFINITE;
        if (accept) t = last ? te : kadd(P.fk, t, hs);
        if (!code && !(accept && last)) {
          if (pairs) {
            h = rk_next_h(fabs(hs), err, accept);
          } else {
            double f;  // 0.9 err^(-1/5), from the squared error
            if (err64 <= 1e-30) f = 5.0;
            else if (err64 >= 1e30) f = 0.2;
            else f = 0.9 * inv_tenth_root(err64);
            h = fabs(hs) * (accept ? fmin(5.0, fmax(0.2, f)) : fmax(0.2, f));
          }
          if (!(h > 0.0) || nonfinite(h) || t + dir * h == t) code = SWARM_SYS_NONFINITE;  // step-size underflow
        }
      }
      if (accept) {
#pragma unroll
        for (int i = 1; i < N; i++)
#pragma unroll
          for (int c = 0; c < 3; c++) {
            x[i][c] = x5[i][c];
            v[i][c] = v5[i][c];
          }
        steps++;
        fresh = true;
        at_end = last;
      } else {
        capped = ADAPT && trials >= nmax;
      }
      if (!code && !capped) continue;
      fresh = false;
    }
    // ---- the system is done with
    spl_write<N>(B, s, m, x, v, Minv, Xc, Vc, t - t0, nullptr, t);
    B.t[s] = t;
    if (code) B.status[s] = code;
    else if (ADAPT) B.status[s] = reached ? SWARM_SYS_DONE : SWARM_SYS_ACTIVE;
    else B.status[s] = plan.full ? SWARM_SYS_DONE : SWARM_SYS_ACTIVE;
    if (P.counters) {
      const unsigned long long tr = ADAPT ? (unsigned long long)trials : (unsigned long long)steps;
      if (steps > 0) atomicAdd(&P.counters[0], (unsigned long long)steps);
      atomicAdd(&P.counters[1], NP * (1ull + 6ull * tr));
    }
    has = false;
  }
}

// ---------------------------------------------------------------- body per lane
struct BplAcc {
  double M, dX[3];
  ff P[3];
  float q2, e1, sv;
  bool tame, range, near;  // tame: this lane's x and v (body 0's too)
};
// Acceleration -M dX + P of the lane's body (bpl_eval_ff without the jerks).  FULL: body 0's pull
// in FP64 from x; else everything from the pairs xf, the acceleration in P.
template <int N, bool FULL, bool STATE>
__device__ __forceinline__ void bpl_acc_ff(const F64k &k, const BplBody<N> &g, const double (&x)[3], const ff (&xf)[3],
                                           const double (&v)[3], const float *kcf, BplAcc &R) {
  ff X[3], rho3, rho2, T[3];
  const bool star = g.b == 0;
  if (FULL) {
    float rho;
    double q2;
#pragma unroll
    for (int c = 0; c < 3; c++) R.dX[c] = ksub(k, x[c], shfl(x[c], g.base));
    if (star) R.dX[0] = 1.0;  // any distance: body 0's lane drops its own terms
    star_pull(k, R.dX, g.m0, R.M, q2, rho3, rho2, rho);
    R.q2 = f_from(q2);
#pragma unroll
    for (int c = 0; c < 3; c++) X[c] = ff_from(R.dX[c]);
    if (star) R.M = 0.0;
  } else {
#pragma unroll
    for (int c = 0; c < 3; c++) X[c] = ff_sub(xf[c], shfl_ff(xf[c], g.base));
    if (star) X[0].h = 1.0f;
    ff_rho3(ff_norm2(X), rho3, rho2);
  }
#pragma unroll
  for (int c = 0; c < 3; c++) {
    T[c] = ff_mul_raw(rho3, X[c]);
    R.P[c] = ff_make(0.0f, 0.0f);
  }
  // S begins with body 0's answer to this body, which is in pairs as well (its lane's sum, 2^-46
  // of it): allowed 1/160 of the relative velocity in a step.  Masses (1e-3, 1), 60 to 130 steps
  // an orbit, without it: 1.5 to 2.9 times the FP64 steps' error; (1, 1), 470 steps: 0.83.
  float S = STATE ? 0.625f * g.mf.h * rho2.h : 0.0f;
  if (STATE) {
    R.near = false;
    R.tame = ff_tame(x, v);
    R.range = frange(R.q2);
  }
#pragma unroll kRingUnroll<N>
  for (int r = 1; r <= g.RT(); r++) {
    const int p = g.next(r), q = g.prev(r);
    ff dx[3], u[3], s3, s2;
#pragma unroll
    for (int c = 0; c < 3; c++) dx[c] = ff_sub_raw(shfl_ff(X[c], p), X[c]);
    const ff r2 = ff_norm2(dx);
    ff_rho3(r2, s3, s2);
    const ff mp = shfl_ff(g.mf, p);
#pragma unroll
    for (int c = 0; c < 3; c++) {
      u[c] = ff_mul_raw(s3, dx[c]);
      R.P[c] = ff_fma_raw(mp, u[c], R.P[c]);
    }
    float sg = 0.0f;
    if (STATE) {  // |X_b| + |X_p| <= sqrt(2 (q2_b + q2_p))
      const float t = R.q2 + __shfl_sync(0xffffffffu, R.q2, p);
      sg = s3.h * (1.41422f * t) * rsqrtf(t);
      S = __fmaf_rn(mp.h, sg, S);
      R.near |= !(r2.h >= kcf[r - 1] * t);
      R.range = R.range && frange(r2.h);
    }
    if (r <= g.RF()) {  // the pair that lane q evaluated with this one
      const ff mq = ff_neg(shfl_ff(g.mf, q));
#pragma unroll
      for (int c = 0; c < 3; c++) R.P[c] = ff_fma_raw(mq, shfl_ff(u[c], q), R.P[c]);
      if (STATE) S = __fmaf_rn(-mq.h, __shfl_sync(0xffffffffu, sg, q), S);
    }
  }
#pragma unroll
  for (int c = 0; c < 3; c++) {
    const ff Tn = ff_norm(T[c]);  // (raw lower parts are of one sign, and so is then their rounding)
    ff w = ff_mul_raw(g.mf, Tn);
    w = fast_two_sum(w.h, __fmaf_rn(g.mf.l, Tn.l, __fmaf_rn(g.mt, Tn.h, w.l)));
    const ff sa = grp_planets_ff<N>(g, w);
    R.P[c] = ff_sel(star, sa, FULL ? ff_norm(R.P[c]) : ff_fma(ff_neg(g.m0f), T[c], R.P[c]));
  }
  if (STATE) {
    float V[3];
#pragma unroll
    for (int c = 0; c < 3; c++) {
      V[c] = f_from(v[c]);
      V[c] -= __shfl_sync(0xffffffffu, V[c], g.base);
    }
    const float V2 = __fmaf_rn(V[2], V[2], __fmaf_rn(V[1], V[1], __fmul_rn(V[0], V[0])));
    R.range = R.range && V2 < 0x1p80f && V2 > 0x1p-80f;
    R.e1 = (g.m0f.h + g.mf.h) * rho3.h;  // of the relative orbit: body 0 need not be the heavy one
    R.sv = __fmul_rn(S, S) / V2;
  }
}

template <int N, bool E>
__device__ __forceinline__ void bpl_rkck_ff_step(const F64k &kk, const BplBody<N> &g, double h, const double (&x)[3],
                                                 const double (&v)[3], const double (&S1)[3], const ff (&P1)[3],
                                                 double (&x5)[3], double (&v5)[3], ff (&ex)[3], ff (&ev)[3]) {
  const RkStep R = rk_step(kk, h);
  ff a[3], D2[3], D3[3], D4[3], D5[3], D6[3], w6[3], Xf[3];
  double xs[3];
  BplAcc A;
#pragma unroll
  for (int c = 0; c < 3; c++) {
    a[c] = ff_norm(ff_add_raw(ff_from(S1[c]), P1[c]));
    Xf[c] = ff_norm(ff_fma_raw(ff_lin(CKN::C2, R.f), ff_from(v[c]), ff_from(x[c])));
    D2[c] = D3[c] = D4[c] = D5[c] = D6[c] = w6[c] = ff_make(0.0f, 0.0f);
  }
  bpl_acc_ff<N, false, false>(kk, g, x, Xf, v, nullptr, A);
#pragma unroll
  for (int c = 0; c < 3; c++) D2[c] = ff_sub(A.P[c], a[c]);
  // stages 3..6 (5 in pairs unless the error is wanted), one copy of the evaluation
#pragma unroll 1
  for (int st = 3; st <= 6; st++) {
    if (st == 3) {
#pragma unroll
      for (int c = 0; c < 3; c++) xs[c] = fma(R.hc3, ff_addto(v[c], rk_w3(R, a[c])), x[c]);
    } else if (st == 4) {
#pragma unroll
      for (int c = 0; c < 3; c++) xs[c] = fma(R.hc4, ff_addto(v[c], rk_w4(R, a[c], D2[c])), x[c]);
    } else if (st == 5) {
#pragma unroll
      for (int c = 0; c < 3; c++) {
        w6[c] = rk_w6(R, a[c], D2[c], D3[c], D4[c]);
        xs[c] = fma(R.h, ff_addto(v[c], rk_w5(R, a[c], D2[c], D3[c])), x[c]);
      }
    } else {
#pragma unroll
      for (int c = 0; c < 3; c++) {
        xs[c] = fma(R.hc6, ff_addto(v[c], w6[c]), x[c]);
        x5[c] = fma(R.h, ff_addto(v[c], rk_wx(R, a[c], D3[c], D4[c], D5[c])), x[c]);
      }
    }
    bpl_acc_ff<N, true, false>(kk, g, xs, Xf, v, nullptr, A);
#pragma unroll
    for (int c = 0; c < 3; c++) {
      const ff D = ff_norm(ff_add_raw(ff_from(fma(-A.M, A.dX[c], -S1[c])), ff_sub_raw(A.P[c], P1[c])));
      if (st == 3) D3[c] = D;
      else if (st == 4) D4[c] = D;
      else if (st == 5) D5[c] = D;
      else D6[c] = D;
    }
  }
#pragma unroll
  for (int c = 0; c < 3; c++) {
    v5[c] = fma(R.h, ff_addto(S1[c], rk_av(P1[c], D3[c], D4[c], D6[c])), v[c]);
    if (E) {
      ex[c] = rk_ex(R, D3[c], D4[c], D5[c]);
      ev[c] = rk_ev(R, D3[c], D4[c], D5[c], D6[c]);
    }
  }
}

// the largest of a group's non-negative pairs, in every lane
template <int N>
__device__ __forceinline__ ff grp_max_ff(const BplBody<N> &g, ff t) {
#pragma unroll
  for (int off = 1; off < N; off <<= 1) {
    const ff o = ff_make(__shfl_down_sync(0xffffffffu, t.h, off), __shfl_down_sync(0xffffffffu, t.l, off));
    if (g.b + off < g.n()) t = ff_max(t, o);
  }
  return shfl_ff(t, g.base);
}

// a trial wholly in FP64, out of line (every lane takes part)
template <int N, bool ADAPT>
static __device__ __noinline__ double bpl_rkck_fp64_trial(const F64k &k, const BplBody<N> &g, double m, double hs,
                                                          double inv_eps2, const double (&x)[3], const double (&v)[3],
                                                          double (&x5)[3], double (&v5)[3]) {
  double a1[3], d2[ARing<N>::RTA], ex[3], ev[3], xn[3], vn[3], err = 0.0;
  ring_acc<N, 0>(k, x, m, g.b, g.base, a1, d2);
  rkck_stages<N, ADAPT>(k, x, v, a1, m, g.b, g.base, hs, xn, vn, ex, ev);
  if (ADAPT) {
    const double X2 = grp_max<N>(x[0] * x[0] + x[1] * x[1] + x[2] * x[2], g.b, g.base);
    const double V2 = grp_max<N>(v[0] * v[0] + v[1] * v[1] + v[2] * v[2], g.b, g.base);
    const double px = ex[0] * ex[0] + ex[1] * ex[1] + ex[2] * ex[2];
    const double pv = ev[0] * ev[0] + ev[1] * ev[1] + ev[2] * ev[2];
    err = grp_max<N>(rk_err2(px, pv, X2, V2, inv_eps2), g.b, g.base);  // squared
  }
#pragma unroll
  for (int c = 0; c < 3; c++) {
    x5[c] = xn[c];
    v5[c] = vn[c];
  }
  return err;
}
// the monitor in FP64 (kc: close-encounter coefficients of the ring over all n bodies)
template <int N>
static __device__ __noinline__ int bpl_acc_monitor_fp64(const F64k &k, const BplBody<N> &g, const double (&x)[3],
                                                        const double (&v)[3], const double (&kc)[ARing<N>::RTA],
                                                        double eject2) {
  const double dq0 = x[0] - shfl(x[0], g.base), dq1 = x[1] - shfl(x[1], g.base), dq2 = x[2] - shfl(x[2], g.base);
  const double q2 = dq0 * dq0 + dq1 * dq1 + dq2 * dq2;
  const bool nf = nonfinite(x[0]) | nonfinite(x[1]) | nonfinite(x[2]) | nonfinite(v[0]) | nonfinite(v[1]) |
                  nonfinite(v[2]);
  const bool ej = g.b != 0 && eject2 > 0.0 && q2 > eject2;
  bool ce = false;
  for (int r = 1; r <= ARing<N>::RT; r++) {
    int p = g.b + r;
    if (p >= N) p -= N;
    const double q2p = shfl(q2, g.base + p);
    double d2 = 0.0;
#pragma unroll
    for (int c = 0; c < 3; c++) {
      const double d = ksub(k, shfl(x[c], g.base + p), x[c]);
      d2 = fma(d, d, d2);
    }
    if (kc[r - 1] > 0.0 && close_encounter(k, d2, kc[r - 1], q2, q2p)) ce = true;
  }
  return (nf ? 1 : 0) | (ej ? 2 : 0) | (ce ? 4 : 0);
}

// Body per lane: G = 32/N systems per warp, lane b of a group holds body b.  Work is
// handed out per system: each group takes the bin's next system (a per-bin counter) as
// soon as its own one has reached its end time or stopped, so groups whose systems need
// fewer (adaptive) steps or stop early do not idle until the warp's last system is done.
// A refill round loads the new systems and evaluates their first stage (the other groups
// re-evaluate their unchanged state, which gives the same values).
// ADAPT = false: fixed steps with the step-count rule of the fixed-step integrators.
// ADAPT = true: the caller's dt is the first trial step; a trial is accepted when the
// scaled error max_b max(|ex_b|/X, |ev_b|/V) (X, V the largest body position and speed
// at the step's start) is at most P.rk_eps; the next trial is h * clamp(0.9 err^(-1/5)).
template <int N, bool ADAPT>
__device__ __forceinline__ void bpl_rkck_stream(const BinView &B, const StepParams &P) {
  constexpr int G = 32 / N;
  constexpr int RT = ARing<N>::RTA;
  constexpr unsigned long long NP = (unsigned long long)N * (N - 1) / 2;
  const unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  BplBody<N> g;
  g.nn = N;
  int grp = lane / N;
  g.b = lane - grp * N;
  const bool lane_ok = grp < G;
  if (!lane_ok) {  // spare lanes mirror group 0 (same broadcasts, same state)
    grp = 0;
    g.b = lane - G * N;
  }
  g.base = grp * N;
  const int b = g.b;
  const int SP = B.S_pad;
  const unsigned gm = g.mask();
  const double dir = P.dt > 0 ? 1.0 : -1.0;
  const int nmax = ADAPT ? (P.max_steps > 0 ? P.max_steps : kRkckTrialCap) : 0;
  const double inv_eps2 = 1.0 / (P.rk_eps * P.rk_eps);
  const bool eps_ok = P.rk_eps > 0x1p-60;
  const ff inv_eps = ff_from(1.0 / P.rk_eps);
  const float ejf = P.eject2 > 0.0 ? 0.998f * (float)P.eject2 : __int_as_float(0x7f800000);

  int s = 0;
  bool has = false, exhausted = false, scaled = false;
  double x[3] = {0.0, 0.0, 0.0}, v[3] = {0.0, 0.0, 0.0}, m = 1.0, S1[3] = {0.0, 0.0, 0.0};
  ff P1[3];
  double kc[RT];
  float kcf[kRoundsA<N>], e1 = 0.0f, sv = 0.0f;
  bool range = false, near = false;
  LaunchPlan plan;
  plan.N = 0;
  plan.full = 1;
  plan.exact = 1;
  plan.h_last = P.dt;
  plan.t_end = P.t_end;
  double t = 0.0, t0 = 0.0, te = 0.0, h = fabs(P.dt);
  int steps = 0, trials = 0;
  bool fresh = false, at_end = false;  // a state without its evaluation; its time is the end time
  g.m0 = 1.0;
  g.m0f = g.mf = ff_make(1.0f, 0.0f);
  g.mt = 0.0f;
#pragma unroll
  for (int c = 0; c < 3; c++) P1[c] = ff_make(0.0f, 0.0f);
  for (int r = 0; r < RT; r++) kc[r] = 0.0;
  for (int r = 0; r < kRoundsA<N>; r++) kcf[r] = 0.0f;

  for (;;) {
    // ---- refill: groups without a system take the bin's next one
    const bool need = !has && !exhausted;
    if (__any_sync(FULL, need)) {
      int sn = 0;
      if (need && lane_ok && b == 0) sn = atomicAdd(P.work_next, 1);
      sn = __shfl_sync(FULL, sn, g.base);
      const int ss = stream_system(B, sn);
      const bool take = need && ss >= 0;
      if (need && ss < 0) exhausted = true;
      if (take) {
        s = ss;
#pragma unroll
        for (int c = 0; c < 3; c++) {
          x[c] = B.x[(size_t)(c * N + b) * SP + s];
          v[c] = B.v[(size_t)(c * N + b) * SP + s];
        }
        m = B.m[(size_t)b * SP + s];
      }
      const double m0 = shfl(m, g.base);
      const bool sc = (__ballot_sync(FULL, !fmass_ok(m, b == 0)) & gm) == 0;
      for (int r = 1; r <= ARing<N>::RT; r++) {
        int p = b + r;
        if (p >= N) p -= N;
        const double mp = shfl(m, g.base + p);
        const double kk = (b != 0 && p != 0) ? hill_kc(P.ce_factor, m, mp, m0) : 0.0;
        if (take) kc[r - 1] = kk;
      }
      for (int r = 1; r <= g.RT(); r++) {
        const double mp = shfl(m, g.next(r));
        const float kk = 2.004f * (float)hill_kc(P.ce_factor, m, mp, m0);
        if (take) kcf[r - 1] = kk;
      }
      if (take) {
        scaled = sc;
        g.m0 = m0;
        g.m0f = ff_from(m0);
        g.mf = ff_norm(ff_from(m));
        g.mt = (float)((m - (double)g.mf.h) - (double)g.mf.l);
        t0 = t = B.t[s];
        steps = 0;
        trials = 0;
        h = fabs(P.dt);
        const bool runnable = B.status[s] <= SWARM_SYS_DONE;
        bool go;
        if (!ADAPT) {
          plan = launch_plan(B, P, s, t0, runnable);
          te = plan.t_end;
          go = runnable && plan.N > 0;
        } else {
          te = adaptive_end(B, P, s);
          go = runnable && ((te - t0) * dir > 1e-12 * fmax(1.0, fabs(te)));
        }
        has = fresh = go;
        at_end = false;
        if (runnable && !go && lane_ok && b == 0) B.status[s] = SWARM_SYS_DONE;
      }
      if (__any_sync(FULL, !has && !exhausted)) continue;
    }
    if (!__any_sync(FULL, has)) break;

    // ---- the new states' evaluation (refills' too: one copy), and the monitor
    if (__any_sync(FULL, fresh)) {
      BplAcc A;
      bpl_acc_ff<N, true, true>(P.fk, g, x, P1, v, kcf, A);
      if (fresh) {
#pragma unroll
        for (int c = 0; c < 3; c++) {
          S1[c] = kmul(P.fk, -A.M, A.dX[c]);
          P1[c] = A.P[c];
        }
        e1 = A.e1;
        sv = A.sv;
        range = scaled && A.tame && (b == 0 || A.range);
        near = !A.tame || (b != 0 && (!A.range || A.near || !(A.q2 < ejf)));
      }
    }
    const bool moved = has && fresh && steps > 0;  // a step led here
    int code = 0;
    if (__any_sync(FULL, moved && near)) {
      const int fl = bpl_acc_monitor_fp64<N>(P.fk, g, x, v, kc, P.eject2);
      const unsigned bnf = __ballot_sync(FULL, moved && (fl & 1)) & gm;
      const unsigned bej = __ballot_sync(FULL, moved && (fl & 2)) & gm;
      const unsigned bce = __ballot_sync(FULL, moved && (fl & 4)) & gm;
      code = bnf ? SWARM_SYS_NONFINITE : bej ? SWARM_SYS_EJECTED : bce ? SWARM_SYS_CLOSE_ENCOUNTER : 0;
      if (!moved) code = 0;
    }
    bool reached = moved && !code && at_end;
    if (!ADAPT && moved && (code || reached || (P.log_interval > 0 && (steps % P.log_interval) == 0)))
      t = step_time(plan, steps, t0, P.dt);  // fixed steps: time formed when it is used
    if (P.log_interval > 0) {
      const bool need_log = moved && !code && (steps % P.log_interval) == 0;
      if (__any_sync(FULL, need_log)) {
        double e4[4];
        ring_energy<N>(x, v, m, b, g.base, e4);
        if (need_log && lane_ok && b == 0) write_log(P, B.gidx[s], t, e4);
      }
    }
    fresh = false;
    bool capped = ADAPT && has && !code && !reached && trials >= nmax;
    const bool alive = has && !code && !reached && !capped;
    if (__any_sync(FULL, alive)) {
      // ---- one step (or trial) for every group whose system goes on
      double hs;
      bool last;
      if (!ADAPT) {
        last = steps + 1 == plan.N;
        hs = (last && !plan.exact) ? plan.h_last : P.dt;
      } else {
        const double rem = kmul(P.fk, ksub(P.fk, te, t), dir);
        last = __double2hiint(h) >= __double2hiint(rem) && h >= rem;  // (FP64 compares are slow)
        hs = kmul(P.fk, last ? rem : h, dir);
      }
      const bool mine = b == 0 ? range : (range && rk_guard(hs, e1, sv));
      bool pairs = (__ballot_sync(FULL, !mine) & gm) == 0 && (!ADAPT || eps_ok);
      double x5[3], v5[3];
      ff err = ff_make(0.0f, 0.0f);  // squared scaled error of the trial
      if (__any_sync(FULL, alive && pairs)) {
        ff ex[3], ev[3];
        bpl_rkck_ff_step<N, ADAPT>(P.fk, g, hs, x, v, S1, P1, x5, v5, ex, ev);
        if (ADAPT) {
          ff X[3], V[3];
#pragma unroll
          for (int c = 0; c < 3; c++) {
            X[c] = ff_norm(ff_from(x[c]));
            V[c] = ff_norm(ff_from(v[c]));
            ex[c] = ff_mul(inv_eps, ex[c]);
            ev[c] = ff_mul(inv_eps, ev[c]);
          }
          const ff X2 = grp_max_ff<N>(g, ff_norm2(X)), V2 = grp_max_ff<N>(g, ff_norm2(V));
          const ff pe = grp_max_ff<N>(g, ff_norm2(ex)), pf = grp_max_ff<N>(g, ff_norm2(ev));
          err = ff_max(ff_div(pe, X2), ff_div(pf, V2));
          const bool out = !(err.h < 0x1p100f);  // out of FP32's range: in FP64
          if ((__ballot_sync(FULL, out) & gm) != 0) pairs = false;
        }
      }
      double err64 = 0.0;
      if (__any_sync(FULL, alive && !pairs)) {
        double x6[3], v6[3];
        err64 = bpl_rkck_fp64_trial<N, ADAPT>(P.fk, g, m, hs, inv_eps2, x, v, x6, v6);
        if (!pairs)
#pragma unroll
          for (int c = 0; c < 3; c++) {
            x5[c] = x6[c];
            v5[c] = v6[c];
          }
      }
      bool accept = alive;
      if (ADAPT && alive) {
        bool bad = false;
        if (pairs) {
          accept = err.h < 1.0f || (err.h == 1.0f && err.l <= 0.0f);
        } else {
          bad = nonfinite(err64);
          accept = !bad && err64 <= 1.0;
        }
        trials++;
        if (bad) code = SWARM_SYS_NONFINITE;
        if (accept) t = last ? te : kadd(P.fk, t, hs);
        if (!code && !(accept && last)) {
          if (pairs) {
            h = rk_next_h(fabs(hs), err, accept);
          } else {
            double f;  // 0.9 err^(-1/5), from the squared error
            if (err64 <= 1e-30) f = 5.0;
            else if (err64 >= 1e30) f = 0.2;
            else f = 0.9 * inv_tenth_root(err64);
            h = fabs(hs) * (accept ? fmin(5.0, fmax(0.2, f)) : fmax(0.2, f));
          }
          if (!(h > 0.0) || nonfinite(h) || t + dir * h == t) code = SWARM_SYS_NONFINITE;  // step-size underflow
        }
      }
      if (accept) {
#pragma unroll
        for (int c = 0; c < 3; c++) {
          x[c] = x5[c];
          v[c] = v5[c];
        }
        steps++;
        fresh = true;
        at_end = last;
      } else if (alive) {
        capped = ADAPT && trials >= nmax;
      }
    }
    // ---- systems that are done with
    const bool finish = has && (code != 0 || reached || capped);
    if (finish && lane_ok) {
#pragma unroll
      for (int c = 0; c < 3; c++) {
        B.x[(size_t)(c * N + b) * SP + s] = x[c];
        B.v[(size_t)(c * N + b) * SP + s] = v[c];
      }
      if (b == 0) {
        B.t[s] = t;
        if (code) B.status[s] = code;
        else if (ADAPT) B.status[s] = reached ? SWARM_SYS_DONE : SWARM_SYS_ACTIVE;
        else B.status[s] = plan.full ? SWARM_SYS_DONE : SWARM_SYS_ACTIVE;
        if (P.counters) {
          const unsigned long long tr = ADAPT ? (unsigned long long)trials : (unsigned long long)steps;
          if (steps > 0) atomicAdd(&P.counters[0], (unsigned long long)steps);
          atomicAdd(&P.counters[1], NP * (1ull + 6ull * tr));
        }
      }
    }
    if (finish) has = fresh = false;
  }
}

// Persistent kernel for one bin: every warp streams systems through its groups until the
// bin's counter runs out (work unit = system).
template <int N, bool ADAPT>
__global__ void __launch_bounds__(128, N <= 3 ? 2 : 3) rkck_uniform_kernel(BinView B, int nunits, StepParams P) {
  (void)nunits;
  if constexpr (N <= 3) spl_rkck_stream<N, ADAPT>(B, P);  // system per lane
  else bpl_rkck_stream<N, ADAPT>(B, P);
}

template <int N, bool ADAPT>
cudaError_t launch_rkck_uniform_n(const BinView &B, int nunits, const StepParams &P, int grid, cudaStream_t st,
                                  int *blocks) {
  if (blocks) cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks, rkck_uniform_kernel<N, ADAPT>, 128, 0);
  if (grid <= 0) return cudaSuccess;
  rkck_uniform_kernel<N, ADAPT><<<grid, 128, 0, st>>>(B, nunits, P);
  return cudaGetLastError();
}

}  // namespace swarm
