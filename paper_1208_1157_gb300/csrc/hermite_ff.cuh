// Hermite-4 steps with the FP64 pipe kept for what needs it (Sec. 2.2.1, Eqs. 3-4).
//
// Per step and coordinate the state moves by x -> x + dx, v -> v + dv, dx ~ eta x and
// dv ~ eta v for a step of 1/1000 orbit (eta = h omega = 6e-3).  Relative to x and v,
//   - dx and dv are formed as float pairs (ff.cuh): 2^-48 eta, below the rounding of the one
//     FP64 sum that adds them;
//   - body 0's pull, which carries the orbit, is FP64; the jerk enters with h^2/12 j ~ eta^2/12
//     and the other planets' accelerations with h a_pert / v (2^-10 and below for planetary
//     masses): pairs;
//   - all but the last corrector pass only move the next evaluation's position, by eta^2/6
//     of their own error, and its acceleration enters with eta: pairs throughout, the
//     perturbers' jerks FP32.
// Each weight is checked at every state (`fguard`); a state where one of them is too large
// for the pairs (large steps, deep encounters, three comparable masses close together) takes
// its step wholly in FP64.
#pragma once
#include "ff.cuh"
#include "hermite.cuh"

namespace swarm {

// coefficients of a step h chosen on the device (adaptive steps)
__device__ __forceinline__ FCoef fcoef(double h) {
  FCoef C;
  C.h = h;
  C.f = ff_from(h);
  C.fl = 0.0f;  // steps of changing length: their roundings do not add up
  C.hh = ff_make(0.5f * C.f.h, 0.5f * C.f.l);
  const ff h2 = ff_mul(C.f, C.f);
  C.h2_2 = ff_make(0.5f * h2.h, 0.5f * h2.l);
  const ff third = ff_make(0x1.555556p-2f, -0x1.555556p-27f);  // 1/3 to 2^-50
  C.h3_6 = ff_mul(ff_mul(C.h2_2, C.f), third);
  const ff h2_4 = ff_make(0.25f * h2.h, 0.25f * h2.l);
  C.h2_12 = ff_mul(h2_4, third);
  C.hf = fabsf(C.f.h);
  return C;
}
// h times a pair, with the product of the lower parts (of one sign for a truncated pair) and,
// for fixed steps, a third part of h: left out, they add up over the steps like a change of
// their length.
__device__ __forceinline__ ff fstep(const FCoef &C, const ff &a) {
  const ff p = ff_mul_raw(C.f, a);
  return ff_make(p.h, __fmaf_rn(C.f.l, a.l, __fmaf_rn(C.fl, a.h, p.l)));
}
// Prediction of Eq. 3: x + h v + G, v + W.
__device__ __forceinline__ void fpredict(const FCoef &C, const ff &a, const ff &j, ff &G, ff &W) {
  G = ff_fma_raw(C.h3_6, j, ff_mul_raw(C.h2_2, a));
  W = ff_norm(ff_fma_raw(C.h2_2, j, fstep(C, a)));
}
// The corrector (time-symmetric form) from the differences D = a_k - a_0 and E = j_0 - j_k:
//   v_k = v + h a_0 + U, U = hh D + h^2/12 E,  x_k = x + h v + G, G = hh (h a_0 + U) - h^2/12 D.
__device__ __forceinline__ void fcorrect(const FCoef &C, const ff &a0, const ff &D, const ff &E, ff &G, ff &W, ff &U) {
  U = ff_norm(ff_fma_raw(C.h2_12, E, ff_mul_raw(C.hh, D)));
  W = ff_add(fstep(C, a0), U);
  G = ff_norm(ff_fma_raw(C.h2_12, ff_neg(D), ff_mul_raw(C.hh, W)));
}

// The correction to a prediction (x + G, v + W) from D = a_k - a_0 - h j_0 and E = j_k - j_0:
// u = hh D - h^2/12 E in v, y = hh u - h^2/12 D in x.
__device__ __forceinline__ void fcorrect_delta(const FCoef &C, const ff &D, const ff &E, ff &y, ff &u) {
  u = ff_fma_raw(ff_neg(C.h2_12), E, ff_mul_raw(C.hh, D));
  y = ff_fma_raw(ff_neg(C.h2_12), D, ff_mul_raw(C.hh, u));
}
__device__ __forceinline__ void fcorrect_delta32(const FCoef &C, float D, float E, float &y, float &u) {
  u = __fmaf_rn(C.hh.h, D, -C.h2_12.h * E);
  y = __fmaf_rn(C.hh.h, u, -C.h2_12.h * D);
}

// Smallness conditions of a state: E = h^2 mu/r^3 (eta^2), S = bound on the perturbing
// accelerations' rounding over 2^-45, V2 = |v|^2 of the body.  Level 0: FP64 steps; 1: pairs
// carry the weights listed above; 2: eta < 0.0134 too, where the FP32 parts of
// `spl_hermite_delta_step` (relative error 2^-22, weight eta^5/8 in v) stay
// below 2^-55.
constexpr float kFFEta2 = 0x1p-8f, kFFEta2Delta = 1.8e-4f;
__device__ __forceinline__ int fguard(float hf, float E, float S, float V2) {
  const float w = hf * S;
  const float w2 = w * w;
  if (!(E <= kFFEta2 && w2 <= 0x1p-18f * V2 && w2 * E * E * E <= 0x1p-55f * V2)) return 0;
  return E <= kFFEta2Delta ? 2 : 1;
}
// squared distances whose powers stay well inside FP32
__device__ __forceinline__ bool frange(float r2) { return r2 > 0x1p-40f && r2 < 0x1p40f; }
// masses, velocities and steps likewise
__device__ __forceinline__ bool fscale(double v, int lo, int hi) {
  const int e = (__double2hiint(v) & 0x7ff00000) >> 20;
  return e > 1023 + lo && e < 1023 + hi;
}

// a body's mass (test particles have tiny ones: what underflows of a planet's pull is below any
// rounding of body 0's)
__device__ __forceinline__ bool fmass_ok(double m, bool star) { return fscale(m, star ? -60 : -100, 40); }

// ---------------------------------------------------------------- adaptive step (Eq. 5)
// The Hermite propagator with the step of Sec. 4.3.2: dt = tau (sum_i |j_i|^2/|a_i|^2)^(-1/2)
// from the values at the start of the step, clamped so that the last step lands on the
// system's end time.  P.dt carries tau (its sign gives the direction).  A launch takes at
// most P.max_steps (or 2^24) steps per system; a system that has not reached its end time
// then stays ACTIVE.  The system-per-lane versions run on coordinates relative to body 0
// like spl_hermite_body; Eq. 5 takes the inertial a and jerk rebuilt from them.
constexpr int kAdaptiveStepCap = 1 << 24;

__device__ __forceinline__ double adaptive_end(const BinView &B, const StepParams &P, int s) {
  return B.t_end ? B.t_end[s] : (P.t_end_dev ? *P.t_end_dev : P.t_end);
}

// FP64 part of one planet's pull towards body 0: M = mu / |X|^3 and q2 = |X|^2; rho^3 and
// rho^2 as pairs.  The root's seed y (hardware rsqrt of the double's upper word, 21 bits, so
// y^2 is exact) is refined by the series of (1 - t)^(-3/2), t = 1 - |X|^2 y^2 formed in FP64
// (one DFMA) and the series in pairs: 8 FP64 instructions, against 14 with rsqrt(double).
__device__ __forceinline__ double rsqrt_seed(double a) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(a));
  return __hiloint2double(__double2hiint(y), 0);
}
__device__ __forceinline__ void star_pull(const F64k &k, const double (&X)[3], double mu, double &M, double &q2,
                                          ff &rho3, ff &rho2, float &rho) {
  q2 = kmul(k, X[0], X[0]);
  q2 = fma(X[1], X[1], q2);
  q2 = fma(X[2], X[2], q2);
  const double y = rsqrt_seed(q2);
  const double y2 = kmul(k, y, y);
  const ff t = ff_from(fma(-q2, y2, k.one));
  // q = (1 - t)^(-3/2) - 1 = t (3/2 + t (15/8 + 35/16 t)), |t| < 2^-19
  const ff w = fast_two_sum(1.5f, __fmul_rn(t.h, __fmaf_rn(2.1875f, t.h, 1.875f)));
  const ff q = ff_mul(t, w);
  const double m3 = kmul(k, kmul(k, y2, y), mu);
  M = fma(ff_double(q), m3, m3);
  const float yf = f_from(y);  // exact
  rho = yf;
  const ff y2f = two_prod(yf, yf);
  const ff y3f = ff_mulf(y2f, yf);
  // y^3 + y^3 q with q's lower part: q is up to 2^-18, and body 0's own acceleration, in which
  // rho^3 is no small weight, wants 2^-46
  const ff c3 = ff_mul_raw(y3f, q), s3 = fast_two_sum(y3f.h, c3.h);
  rho3 = fast_two_sum(s3.h, __fadd_rn(s3.l, __fadd_rn(y3f.l, c3.l)));
  const float p2 = __fmaf_rn(t.h, t.h, t.h);
  rho2 = fast_two_sum(y2f.h, __fmaf_rn(y2f.h, p2, y2f.l));
}

// w = v + c x, c = -3 (x.v) rho^2  (the jerk's direction, Eq. 1's derivative); returns c
__device__ __forceinline__ float fjerk_dir(const ff (&x)[3], const ff (&v)[3], const ff &rho2, ff (&w)[3]) {
  const ff c = ff_mul(ff_mulf(ff_dot(x, v), -3.0f), rho2);
#pragma unroll
  for (int i = 0; i < 3; i++) w[i] = ff_fma_raw(c, x[i], v[i]);
  return c.h;
}
// the same in FP32
__device__ __forceinline__ void fjerk_dir32(const ff (&x)[3], const ff (&v)[3], float rho2, float (&w)[3]) {
  const float rv = __fmaf_rn(x[2].h, v[2].h, __fmaf_rn(x[1].h, v[1].h, __fmul_rn(x[0].h, v[0].h)));
  const float c = -3.0f * rv * rho2;
#pragma unroll
  for (int i = 0; i < 3; i++) w[i] = __fmaf_rn(c, x[i].h, v[i].h);
}

// Change of a pair's terms T = s x, Z = s (u + c x) (x, u its difference vectors, s = 1/|x|^3,
// p = 1/|x|^2, c = -3 (x.u) p) when x, u move by d, e, in FP32: the algebraic difference, not a
// linearisation, so its error is 2^-22 of the change itself.
__device__ __forceinline__ void fpair_delta(const float (&x)[3], const float (&u)[3], const float (&d)[3],
                                            const float (&e)[3], float s, float p, float c, float (&DT)[3],
                                            float (&DZ)[3]) {
  float xn[3], e2 = 0.0f, rv = 0.0f;
#pragma unroll
  for (int q = 0; q < 3; q++) {
    e2 = __fmaf_rn(d[q], __fmaf_rn(2.0f, x[q], d[q]), e2);
    xn[q] = x[q] + d[q];
    rv = __fmaf_rn(d[q], u[q], __fmaf_rn(xn[q], e[q], rv));
  }
  e2 *= p;                                               // |x + d|^2 / |x|^2 - 1
  const float f = __fmaf_rn(e2, e2, -e2);                // 1/(1 + e2) - 1
  const float t = e2 * __fmaf_rn(1.875f, e2, -1.5f);     // (1 + e2)^(-3/2) - 1
  const float dc = __fmaf_rn(c, f, __fmaf_rn(f, -3.0f * rv * p, -3.0f * rv * p));
#pragma unroll
  for (int q = 0; q < 3; q++) {
    DT[q] = s * __fmaf_rn(t, xn[q], d[q]);
    const float w = __fmaf_rn(c, x[q], u[q]);
    const float dw = __fmaf_rn(c, d[q], __fmaf_rn(dc, xn[q], e[q]));
    DZ[q] = s * __fmaf_rn(t, w + dw, dw);
  }
}

// ---------------------------------------------------------------- system per lane
// masses of a system per lane as pairs
template <int N>
struct FMass {
  double mu[N];  // m_0 + m_k
  ff m[N], muf[N];
  bool ok;       // representable
};
template <int N>
__device__ __forceinline__ FMass<N> fmass(const double (&m)[N]) {
  FMass<N> f;
  f.ok = true;
#pragma unroll
  for (int i = 0; i < N; i++) {
    f.mu[i] = m[0] + m[i];
    f.m[i] = ff_from(m[i]);
    f.muf[i] = ff_from(f.mu[i]);
    f.ok = f.ok && fmass_ok(m[i], i == 0);
  }
  return f;
}

// An evaluation of a system per lane: A_k = -M_k X_k + P_k with M_k (and X_k) FP64, the
// perturbations P_k and the jerks J_k pairs; index 0: body 0's own (kStar).
enum { kGuard = 1, kGeo = 2, kStar = 4 };
template <int N>
struct SplEval {
  double M[N];
  ff P[N][3], J[N][3];
  float q2[N], d2[N][N];
};
template <int N>
struct SplGeo {
  float X[N][3], V[N][3], s[N][N], p[N][N], c[N][N];
};

// Perturbations of the relative accelerations, P_k = sum_{j != k} m_j (s_kj (X_j - X_k) - s_j X_j),
// and of the jerks, from the positions, velocities, T_k = s_k X_k and Z_k = s_k w_k.
// JERK 0: none, 1: FP32, 2: pairs.  S_k: see fguard.
template <int N, int JERK>
__device__ __forceinline__ void spl_pert(const FMass<N> &F, const ff (&X)[N][3], const ff (&V)[N][3], const ff (&T)[N][3],
                                         const ff (&Z)[N][3], ff (&P)[N][3], ff (&Q)[N][3], float (&d2)[N][N],
                                         SplGeo<N> &g) {
#pragma unroll
  for (int k = 1; k < N; k++)
#pragma unroll
    for (int c = 0; c < 3; c++) P[k][c] = Q[k][c] = ff_make(0.0f, 0.0f);
#pragma unroll
  for (int i = 1; i < N; i++)
#pragma unroll
    for (int k = i + 1; k < N; k++) {
      ff dx[3], u[3], rho3, rho2;
#pragma unroll
      for (int c = 0; c < 3; c++) dx[c] = ff_sub_raw(X[k][c], X[i][c]);
      const ff r2 = ff_norm2(dx);
      ff_rho3(r2, rho3, rho2);
      d2[i][k] = r2.h;
      g.s[i][k] = rho3.h;
      g.p[i][k] = rho2.h;
#pragma unroll
      for (int c = 0; c < 3; c++) {
        u[c] = ff_mul_raw(rho3, dx[c]);
        // planet i: + m_k (u - T_k); planet k: - m_i (u + T_i)
        const ff ui = ff_sub_raw(u[c], T[k][c]), uk = ff_neg(ff_add_raw(u[c], T[i][c]));
        P[i][c] = i == 1 && k == 2 ? ff_mul_raw(F.m[k], ui) : ff_fma_raw(F.m[k], ui, P[i][c]);
        P[k][c] = i == 1 ? ff_mul_raw(F.m[i], uk) : ff_fma_raw(F.m[i], uk, P[k][c]);
      }
      if (JERK == 2) {
        ff dv[3], w[3];
#pragma unroll
        for (int c = 0; c < 3; c++) dv[c] = ff_sub_raw(V[k][c], V[i][c]);
        g.c[i][k] = fjerk_dir(dx, dv, rho2, w);
#pragma unroll
        for (int c = 0; c < 3; c++) {
          const ff z = ff_mul_raw(rho3, w[c]);
          const ff zi = ff_sub_raw(z, Z[k][c]), zk = ff_neg(ff_add_raw(z, Z[i][c]));
          Q[i][c] = i == 1 && k == 2 ? ff_mul_raw(F.m[k], zi) : ff_fma_raw(F.m[k], zi, Q[i][c]);
          Q[k][c] = i == 1 ? ff_mul_raw(F.m[i], zk) : ff_fma_raw(F.m[i], zk, Q[k][c]);
        }
      } else if (JERK == 1) {
        ff dv[3];
        float w[3];
#pragma unroll
        for (int c = 0; c < 3; c++) dv[c] = ff_make(__fsub_rn(V[k][c].h, V[i][c].h), 0.0f);
        fjerk_dir32(dx, dv, rho2.h, w);
#pragma unroll
        for (int c = 0; c < 3; c++) {
          const float z = __fmul_rn(rho3.h, w[c]);
          Q[i][c].h = __fmaf_rn(F.m[k].h, __fsub_rn(z, Z[k][c].h), Q[i][c].h);
          Q[k][c].h = __fmaf_rn(-F.m[i].h, __fadd_rn(z, Z[i][c].h), Q[k][c].h);
        }
      }
    }
}

// Evaluation at a state given in FP64 (X) and pairs (V).  kGuard: returns the level (`fguard`)
// of this state for steps of length hf.  kGeo: the geometry in FP32 for `spl_delta`, whose
// pairs are indexed [i][k] (i = 0: body 0): 1/d^3, 1/d^2 and -3 (d.u)/d^2.  kStar: body 0's own
// acceleration and jerk too (Eq. 5 wants the inertial ones, a_k = A_k + a_0).
template <int N, int FLAGS>
__device__ __forceinline__ int spl_eval_full(const F64k &kk, const FMass<N> &F, float hf, const double (&X)[N][3],
                                             const ff (&V)[N][3], SplEval<N> &R, SplGeo<N> &g) {
  ff Xf[N][3], T[N][3], Z[N][3], Q[N][3];
  float r0[N];
#pragma unroll
  for (int k = 1; k < N; k++) {
    ff rho3, rho2, w[3];
    float rho;
    double q2;
    star_pull(kk, X[k], F.mu[k], R.M[k], q2, rho3, rho2, rho);
    R.q2[k] = f_from(q2);
#pragma unroll
    for (int c = 0; c < 3; c++) Xf[k][c] = ff_from(X[k][c]);
    g.c[0][k] = fjerk_dir(Xf[k], V[k], rho2, w);
#pragma unroll
    for (int c = 0; c < 3; c++) {
      T[k][c] = ff_mul_raw(rho3, Xf[k][c]);
      Z[k][c] = ff_mul_raw(rho3, w[c]);
    }
    g.s[0][k] = rho3.h;
    g.p[0][k] = rho2.h;
    if (FLAGS & kGeo)
#pragma unroll
      for (int c = 0; c < 3; c++) {
        g.X[k][c] = Xf[k][c].h;
        g.V[k][c] = V[k][c].h;
      }
    if (FLAGS & kGuard) r0[k] = R.q2[k] * rho;
  }
  spl_pert<N, 2>(F, Xf, V, T, Z, R.P, Q, R.d2, g);
  if (FLAGS & kStar)
#pragma unroll
    for (int c = 0; c < 3; c++) {
      R.P[0][c] = ff_mul_raw(F.m[1], T[1][c]);
      R.J[0][c] = ff_mul_raw(F.m[1], Z[1][c]);
#pragma unroll
      for (int k = 2; k < N; k++) {
        R.P[0][c] = ff_fma_raw(F.m[k], T[k][c], R.P[0][c]);
        R.J[0][c] = ff_fma_raw(F.m[k], Z[k][c], R.J[0][c]);
      }
    }
  bool ok = F.ok;
  int level = 2;
#pragma unroll
  for (int k = 1; k < N; k++) {
#pragma unroll
    for (int c = 0; c < 3; c++) R.J[k][c] = ff_fma(ff_neg(F.muf[k]), Z[k][c], Q[k][c]);
    if (FLAGS & kGuard) {
      // the pairs' differences lose (|X_k| + |X_j|)/d of their bits: s d (|X_k| + |X_j|)/d
      float S = 0.0f;
#pragma unroll
      for (int j = 1; j < N; j++)
        if (j != k) {
          ok = ok && frange(j < k ? R.d2[j][k] : R.d2[k][j]);
          S = __fmaf_rn(F.m[j].h, __fmaf_rn(j < k ? g.s[j][k] : g.s[k][j], r0[k] + r0[j], g.p[0][j]), S);
        }
      const float V2 = __fmaf_rn(V[k][2].h, V[k][2].h, __fmaf_rn(V[k][1].h, V[k][1].h, __fmul_rn(V[k][0].h, V[k][0].h)));
      ok = ok && frange(R.q2[k]) && V2 < 0x1p80f;
      level = min(level, fguard(hf, hf * hf * F.muf[k].h * g.s[0][k], S, V2));
    }
  }
  return ok ? level : 0;
}
// Evaluation wholly in pairs (perturbers' jerks FP32).
template <int N>
__device__ __forceinline__ void spl_eval_ff(const FMass<N> &F, const ff (&X)[N][3], const ff (&V)[N][3], ff (&A)[N][3],
                                            ff (&J)[N][3]) {
  ff T[N][3], Z[N][3];
  SplGeo<N> g;
  float d2[N][N];
#pragma unroll
  for (int k = 1; k < N; k++) {
    ff rho3, rho2, w[3];
    ff_rho3(ff_norm2(X[k]), rho3, rho2);
    fjerk_dir(X[k], V[k], rho2, w);
#pragma unroll
    for (int c = 0; c < 3; c++) {
      T[k][c] = ff_mul_raw(rho3, X[k][c]);
      Z[k][c] = ff_mul_raw(rho3, w[c]);
    }
  }
  spl_pert<N, 1>(F, X, V, T, Z, A, J, d2, g);
#pragma unroll
  for (int k = 1; k < N; k++)
#pragma unroll
    for (int c = 0; c < 3; c++) {
      A[k][c] = ff_fma(ff_neg(F.muf[k]), T[k][c], A[k][c]);
      J[k][c] = ff_fma(ff_neg(F.muf[k]), Z[k][c], J[k][c]);
    }
}

// Change of the evaluation (accelerations DA, jerks DJ) when the positions and velocities
// move by dX, dV from those of the geometry g, in FP32: the algebraic differences of Eq. 1's
// terms, not a linearisation, so their error is 2^-22 of the change itself.
template <int N>
__device__ __forceinline__ void spl_delta(const FMass<N> &F, const SplGeo<N> &g, const float (&dX)[N][3],
                                          const float (&dV)[N][3], float (&DA)[N][3], float (&DJ)[N][3]) {
  float T[N][3], Z[N][3];
#pragma unroll
  for (int k = 1; k < N; k++) {
    fpair_delta(g.X[k], g.V[k], dX[k], dV[k], g.s[0][k], g.p[0][k], g.c[0][k], T[k], Z[k]);
#pragma unroll
    for (int q = 0; q < 3; q++) {
      DA[k][q] = -F.muf[k].h * T[k][q];
      DJ[k][q] = -F.muf[k].h * Z[k][q];
      // index 0: body 0's own (dropped where it is not used)
      DA[0][q] = k == 1 ? F.m[k].h * T[k][q] : __fmaf_rn(F.m[k].h, T[k][q], DA[0][q]);
      DJ[0][q] = k == 1 ? F.m[k].h * Z[k][q] : __fmaf_rn(F.m[k].h, Z[k][q], DJ[0][q]);
    }
  }
#pragma unroll
  for (int i = 1; i < N; i++)
#pragma unroll
    for (int k = i + 1; k < N; k++) {
      float x[3], u[3], d[3], e[3], t[3], z[3];
#pragma unroll
      for (int q = 0; q < 3; q++) {
        x[q] = g.X[k][q] - g.X[i][q];
        u[q] = g.V[k][q] - g.V[i][q];
        d[q] = dX[k][q] - dX[i][q];
        e[q] = dV[k][q] - dV[i][q];
      }
      fpair_delta(x, u, d, e, g.s[i][k], g.p[i][k], g.c[i][k], t, z);
#pragma unroll
      for (int q = 0; q < 3; q++) {
        DA[i][q] = __fmaf_rn(F.m[k].h, t[q] - T[k][q], DA[i][q]);
        DJ[i][q] = __fmaf_rn(F.m[k].h, z[q] - Z[k][q], DJ[i][q]);
        DA[k][q] = __fmaf_rn(-F.m[i].h, t[q] + T[i][q], DA[k][q]);
        DJ[k][q] = __fmaf_rn(-F.m[i].h, z[q] + Z[i][q], DJ[k][q]);
      }
    }
}

// A step from a state of level 2: one evaluation, at the predicted state, in FP64 and pairs;
// the corrector moves the positions by eta^4/24 only, and the evaluations after it are that
// one plus FP32 differences.  The accelerations are a0 (FP64) plus da (their FP32
// difference).  x, v, a0, da, j0 become those of the new state, q2 and d2 its FP32 distances;
// returns the next step's level, for a length of at most hf.  STAR: sa, sj get body 0's acceleration and jerk.
template <int N, bool STAR>
__device__ __forceinline__ int spl_hermite_delta_step(const F64k &kk, const FMass<N> &F, const FCoef &C, float hf, int n_corr,
                                                      double (&x)[N][3], double (&v)[N][3], double (&a0)[N][3],
                                                      float (&da)[N][3], ff (&j0)[N][3], float (&q2)[N],
                                                      float (&d2)[N][N], ff (&sa)[3], ff (&sj)[3]) {
  SplEval<N> R;
  SplGeo<N> g;
  ff G[N][3], W[N][3], D[N][3], E[N][3];
  int level;
  {
    ff V[N][3];
    double xp[N][3];
#pragma unroll
    for (int k = 1; k < N; k++)
#pragma unroll
      for (int c = 0; c < 3; c++) {
        // rounded pairs: the truncated ones' lower parts have one sign, a bias in h v and h a
        const ff a = ff_from(a0[k][c]), w = ff_norm(ff_from(v[k][c]));
        fpredict(C, ff_norm(ff_make(a.h, a.l + da[k][c])), j0[k][c], G[k][c], W[k][c]);
        G[k][c] = ff_norm(ff_add_raw(fstep(C, w), G[k][c]));
        V[k][c] = ff_add(w, W[k][c]);
        xp[k][c] = ff_addto(x[k][c], G[k][c]);
      }
    level = spl_eval_full<N, kGuard | kGeo | (STAR ? kStar : 0)>(kk, F, hf, xp, V, R, g);
#pragma unroll
    for (int k = 1; k < N; k++)
#pragma unroll
      for (int c = 0; c < 3; c++) {
        // D = a_1 - a_0 - h j_0, E = j_1 - j_0; body 0's pull on the new state from xp
        const ff P = ff_norm(R.P[k][c]);
        ff d = ff_from(fma(-R.M[k], xp[k][c], -a0[k][c]));
        d = ff_add_raw(ff_make(d.h, d.l - da[k][c]), P);
        D[k][c] = ff_norm(ff_fma_raw(ff_neg(C.f), j0[k][c], d));
        E[k][c] = ff_norm(ff_sub_raw(R.J[k][c], j0[k][c]));
        a0[k][c] = fma(-R.M[k], xp[k][c], ff_double(P));
      }
  }
  float DJ[N][3], dX[N][3], dV[N][3];
#pragma unroll
  for (int k = 1; k < N; k++)
#pragma unroll
    for (int c = 0; c < 3; c++) da[k][c] = DJ[k][c] = 0.0f;
  for (int ic = 1; ic < n_corr; ic++) {
#pragma unroll
    for (int k = 1; k < N; k++)
#pragma unroll
      for (int c = 0; c < 3; c++) {
        fcorrect_delta32(C, D[k][c].h + da[k][c], E[k][c].h + DJ[k][c], dX[k][c], dV[k][c]);
      }
    spl_delta<N>(F, g, dX, dV, da, DJ);
  }
#pragma unroll
  for (int k = 1; k < N; k++)
#pragma unroll
    for (int c = 0; c < 3; c++) {
      ff y, u;
      fcorrect_delta(C, ff_make(D[k][c].h, D[k][c].l + da[k][c]), ff_make(E[k][c].h, E[k][c].l + DJ[k][c]), y, u);
      dV[k][c] = u.h + u.l;
      dX[k][c] = y.h + y.l;
      x[k][c] = ff_addto(x[k][c], ff_add(G[k][c], y));
      v[k][c] = ff_addto(v[k][c], ff_add(W[k][c], u));
    }
  spl_delta<N>(F, g, dX, dV, da, DJ);
#pragma unroll
  for (int k = 1; k < N; k++) {
    q2[k] = R.q2[k];
#pragma unroll
    for (int j = k + 1; j < N; j++) d2[k][j] = R.d2[k][j];
#pragma unroll
    for (int c = 0; c < 3; c++) j0[k][c] = ff_norm(ff_make(R.J[k][c].h, R.J[k][c].l + DJ[k][c]));
  }
  if (STAR)
#pragma unroll
    for (int c = 0; c < 3; c++) {
      sa[c] = ff_make(R.P[0][c].h, R.P[0][c].l + da[0][c]);
      sj[c] = ff_make(R.J[0][c].h, R.J[0][c].l + DJ[0][c]);
    }
  return level;
}

// The new (x, v) of a step from a state of level 1 (or 2), accelerations a0 + da.  At these
// step lengths h v and h a_0 are FP64 too.
template <int N>
__device__ __forceinline__ void spl_hermite_ff_advance(const F64k &kk, const FMass<N> &F, const FCoef &C, int n_corr,
                                                       double (&x)[N][3], double (&v)[N][3], const double (&a0)[N][3],
                                                       const float (&da)[N][3], const ff (&j0)[N][3]) {
  ff V[N][3], G[N][3], W[N][3], af[N][3], U[N][3];
#pragma unroll
  for (int k = 1; k < N; k++)
#pragma unroll
    for (int c = 0; c < 3; c++) {
      V[k][c] = ff_from(v[k][c]);
      af[k][c] = ff_from(a0[k][c]);
      af[k][c] = ff_norm(ff_make(af[k][c].h, af[k][c].l + da[k][c]));
      x[k][c] = fma(C.h, v[k][c], x[k][c]);
      fpredict(C, af[k][c], j0[k][c], G[k][c], W[k][c]);
    }
  // every corrector pass but the last
  for (int ic = 1; ic < n_corr; ic++) {
    ff X[N][3], A[N][3], J[N][3];
#pragma unroll
    for (int k = 1; k < N; k++)
#pragma unroll
      for (int c = 0; c < 3; c++) {
        X[k][c] = ff_add(ff_from(x[k][c]), G[k][c]);
        U[k][c] = ff_add(V[k][c], W[k][c]);
      }
    spl_eval_ff<N>(F, X, U, A, J);
#pragma unroll
    for (int k = 1; k < N; k++)
#pragma unroll
      for (int c = 0; c < 3; c++)
        fcorrect(C, af[k][c], ff_sub(A[k][c], af[k][c]), ff_sub(j0[k][c], J[k][c]), G[k][c], W[k][c], U[k][c]);
  }
  SplEval<N> R;
  SplGeo<N> g;
  double xp[N][3];
#pragma unroll
  for (int k = 1; k < N; k++)
#pragma unroll
    for (int c = 0; c < 3; c++) {
      xp[k][c] = ff_addto(x[k][c], ff_norm(G[k][c]));
      U[k][c] = ff_add(V[k][c], W[k][c]);
    }
  spl_eval_full<N, 0>(kk, F, C.hf, xp, U, R, g);
#pragma unroll
  for (int k = 1; k < N; k++)
#pragma unroll
    for (int c = 0; c < 3; c++) {
      // a_k - a_0: body 0's pull in one DFMA
      ff D = ff_from(fma(-R.M[k], xp[k][c], -a0[k][c]));
      D = ff_add(ff_make(D.h, D.l - da[k][c]), R.P[k][c]);
      fcorrect(C, af[k][c], D, ff_sub(j0[k][c], R.J[k][c]), G[k][c], W[k][c], U[k][c]);
      x[k][c] = ff_addto(x[k][c], G[k][c]);
      U[k][c].l = __fmaf_rn(C.f.h, da[k][c], U[k][c].l);
      v[k][c] = ff_addto(fma(C.h, a0[k][c], v[k][c]), ff_norm(U[k][c]));
    }
}

// Eq. 5 sum over the bodies of a system held by one lane, sum_i |j_i|^2 / |a_i|^2, with
// one division: the running fraction num/den takes body i as (num A_i + J_i den)/(den A_i)
// (A = |a|^2, J = |j|^2; den stays within range for the n <= 4 of this mapping).
template <int N>
__device__ __forceinline__ double spl_eq5_sum(const F64k &k, const double (&a)[N][3], const double (&j)[N][3]) {
  double num = 0.0, den = 1.0;
#pragma unroll
  for (int i = 0; i < N; i++) {
    const double A = fma(a[i][2], a[i][2], fma(a[i][1], a[i][1], kmul(k, a[i][0], a[i][0])));
    const double J = fma(j[i][2], j[i][2], fma(j[i][1], j[i][1], kmul(k, j[i][0], j[i][0])));
    num = fma(num, A, kmul(k, J, den));
    den = kmul(k, den, A);
  }
  return num / den;
}

// The same sum from the relative-coordinate values of spl_accjerk_rel: a_0 = A[0],
// a_k = A[k] + A[0] (likewise the jerks).
template <int N>
__device__ __forceinline__ double spl_eq5_sum_rel(const F64k &kk, const double (&A)[N][3], const double (&J)[N][3]) {
  double a[N][3], j[N][3];
#pragma unroll
  for (int c = 0; c < 3; c++) {
    a[0][c] = A[0][c];
    j[0][c] = J[0][c];
#pragma unroll
    for (int k = 1; k < N; k++) {
      a[k][c] = kadd(kk, A[k][c], A[0][c]);
      j[k][c] = kadd(kk, J[k][c], J[0][c]);
    }
  }
  return spl_eq5_sum<N>(kk, a, j);
}

// The monitor in FP64 (kc: `hill_kc` of the planet pairs).
template <int N>
__device__ __forceinline__ int spl_monitor(const F64k &kk, const double (&x)[N][3], const double (&v)[N][3],
                                           const double (&q2)[N], const double (&d2)[N][N], const double (&kc)[N][N],
                                           double eject2) {
  bool nf = false, ej = false, ce = false;
#pragma unroll
  for (int i = 1; i < N; i++) {
    ej |= eject2 > 0.0 && nonneg_lt(eject2, q2[i]);
#pragma unroll
    for (int c = 0; c < 3; c++) nf |= nonfinite(x[i][c]) | nonfinite(v[i][c]);
#pragma unroll
    for (int j = i + 1; j < N; j++)
      if (kc[i][j] > 0.0 && close_encounter(kk, d2[i][j], kc[i][j], q2[i], q2[j])) ce = true;
  }
  return nf ? SWARM_SYS_NONFINITE : ej ? SWARM_SYS_EJECTED : ce ? SWARM_SYS_CLOSE_ENCOUNTER : 0;
}

// Up to `count` steps wholly in FP64, for states of level 0 (and a shortened last step): fixed
// steps of h, or (ADAPT) Eq. 5 steps of tau = h toward te.  a0 and j0 (`jb`: FP64 bits in the
// pairs' registers) are those of the state, or formed first.  Stops with the monitor's code;
// `done` counts the steps taken, `reached` tells that te was.  Out of line, with the
// evaluations carried from step to step, so that a system that stays at level 0 costs what an
// FP64 kernel's does.
template <int N, bool ADAPT, bool PRINTED>
static __device__ __noinline__ int spl_hermite_fp64_run(const F64k &kk, const double (&m)[N], const double (&kc)[N][N],
                                                 double eject2, double hh, int n_corr, int count, bool first,
                                                 double (&xs)[N][3], double (&vs)[N][3], double (&as)[N][3],
                                                 ff (&jb)[N][3], int &done, double &ts, double te, bool &reached) {
  constexpr bool kCache = N <= 3;
  const double tau = fabs(hh), dir = hh > 0 ? 1.0 : -1.0;
  HCoef C = hcoef(hh);
  RhoCache<N> rc;
  double x[N][3], v[N][3], a0[N][3], j0[N][3], q2[N], d2[N][N], xk[N][3], vk[N][3], Xb[N][3], Vb[N][3], t = ts;
#pragma unroll
  for (int i = 0; i < N; i++)
#pragma unroll
    for (int c = 0; c < 3; c++) {
      x[i][c] = xs[i][c];
      v[i][c] = vs[i][c];
      a0[i][c] = as[i][c];
      j0[i][c] = __hiloint2double(__float_as_int(jb[i][c].h), __float_as_int(jb[i][c].l));
    }
  if (first) spl_accjerk_rel<N>(kk, x, v, m, a0, j0, q2, d2);
  int code = 0;
  for (int s = 0; s < count; s++) {
    bool last = false;
    double h = hh;
    if (ADAPT) {
      h = kmul(kk, tau, rsqrt(spl_eq5_sum_rel<N>(kk, a0, j0)));
      if (!(h > 0.0) || nonfinite(h)) {
        code = SWARM_SYS_NONFINITE;
        break;
      }
      const double rem = kmul(kk, ksub(kk, te, t), dir);
      last = h >= rem;
      h = kmul(kk, last ? rem : h, dir);
      C = hcoef(kk, h);
    }
    const PCoef PC = pcoef(h);
#pragma unroll
    for (int i = 1; i < N; i++)
#pragma unroll
      for (int c = 0; c < 3; c++) {
        xk[i][c] = fma(j0[i][c], C.h3_6, fma(a0[i][c], C.h2_2, fma(v[i][c], C.h, x[i][c])));
        vk[i][c] = fma(j0[i][c], C.h2_2, fma(a0[i][c], C.h, v[i][c]));
        Vb[i][c] = fma(j0[i][c], C.h2_12, fma(a0[i][c], C.hh, v[i][c]));
        Xb[i][c] = PRINTED ? fma(j0[i][c], PC.pj, fma(a0[i][c], PC.pa, xk[i][c]))
                           : fma(a0[i][c], C.h2_12, fma(v[i][c], C.hh, x[i][c]));
      }
    for (int ic = 0; ic < n_corr; ic++) {
      double ak[N][3], jk[N][3];
      if (!kCache) spl_accjerk_rel<N>(kk, xk, vk, m, ak, jk, q2, d2);
      else if (ic == 0) spl_accjerk_rel_cached<N, true>(kk, xk, vk, m, ak, jk, q2, d2, rc);
      else spl_accjerk_rel_cached<N, false>(kk, xk, vk, m, ak, jk, q2, d2, rc);
#pragma unroll
      for (int i = 1; i < N; i++)
#pragma unroll
        for (int c = 0; c < 3; c++) {
          vk[i][c] = fma(-C.h2_12, jk[i][c], fma(C.hh, ak[i][c], Vb[i][c]));
          xk[i][c] = PRINTED ? fma(PC.cj, jk[i][c], fma(PC.ca, ak[i][c], Xb[i][c]))
                             : fma(-C.h2_12, ak[i][c], fma(C.hh, vk[i][c], Xb[i][c]));
        }
    }
    if (!kCache) spl_accjerk_rel<N>(kk, xk, vk, m, a0, j0, q2, d2);
    else spl_accjerk_rel_cached<N, false>(kk, xk, vk, m, a0, j0, q2, d2, rc);
#pragma unroll
    for (int i = 1; i < N; i++)
#pragma unroll
      for (int c = 0; c < 3; c++) {
        x[i][c] = xk[i][c];
        v[i][c] = vk[i][c];
      }
    done++;
    if (ADAPT) t = last ? te : kadd(kk, t, h);
    code = spl_monitor<N>(kk, x, v, q2, d2, kc, eject2);
    reached = ADAPT && last && !code;
    if (code || reached) break;
  }
  ts = t;
#pragma unroll
  for (int i = 0; i < N; i++)
#pragma unroll
    for (int c = 0; c < 3; c++) {
      xs[i][c] = x[i][c];
      vs[i][c] = v[i][c];
      as[i][c] = a0[i][c];
      jb[i][c] = ff_make(__int_as_float(__double2hiint(j0[i][c])), __int_as_float(__double2loint(j0[i][c])));
    }
  return code;
}
constexpr int kStepRun = 16;  // FP64 steps between two looks at the level (a look costs 1/8 of one)

// Evaluation at a state (x, v): a0, j0, the monitor's distances; returns the level, 0 for a state
// that is not finite or that the pairs cannot hold.  Every state that comes from outside or from
// an FP64 step is looked at here.  A step from a state of level 1 or 2 cannot leave that range
// without the level's own tests seeing it: |x| < 2^20, |v| < 2^40 and h < 2^60 (h^2 mu/r^3 <=
// 2^-8, mu > 2^-60), so the new |x| is below 2^101 and |x|^2, which `f_from` would take for one
// within `frange` from 2^216 on, below 2^202.
template <int N, bool STAR>
__device__ __forceinline__ int spl_ff_state(const F64k &kk, const FMass<N> &F, float hf, const double (&x)[N][3],
                                            const double (&v)[N][3], double (&a0)[N][3], float (&da)[N][3],
                                            ff (&j0)[N][3], float (&q2)[N], float (&d2)[N][N],
                                            ff (&sa)[3], ff (&sj)[3]) {
  SplEval<N> R;
  SplGeo<N> g;
  ff V[N][3];
#pragma unroll
  for (int k = 1; k < N; k++)
#pragma unroll
    for (int c = 0; c < 3; c++) V[k][c] = ff_from(v[k][c]);
  int level = spl_eval_full<N, kGuard | (STAR ? kStar : 0)>(kk, F, hf, x, V, R, g);
#pragma unroll
  for (int k = 1; k < N; k++)
    if (!ff_tame(x[k], v[k])) level = 0;
#pragma unroll
  for (int k = 1; k < N; k++) {
    q2[k] = R.q2[k];
#pragma unroll
    for (int c = 0; c < 3; c++) {
      a0[k][c] = fma(-R.M[k], x[k][c], ff_double(ff_norm(R.P[k][c])));
      da[k][c] = 0.0f;
      j0[k][c] = R.J[k][c];
    }
#pragma unroll
    for (int j = k + 1; j < N; j++) d2[k][j] = R.d2[k][j];
  }
  if (STAR)
#pragma unroll
    for (int c = 0; c < 3; c++) {
      sa[c] = R.P[0][c];
      sj[c] = R.J[0][c];
    }
  return level;
}

// Both out of line, for what is not on the hot path (a step is some 3300 instructions, 53 KB:
// the loops have to stay within the instruction cache).
template <int N, bool STAR>
static __device__ __noinline__ int spl_ff_state_call(const F64k &kk, const FMass<N> &F, float hf, const double (&x)[N][3],
                                              const double (&v)[N][3], double (&a0)[N][3], float (&da)[N][3],
                                              ff (&j0)[N][3], float (&q2)[N], float (&d2)[N][N], ff (&sa)[3],
                                              ff (&sj)[3]) {
  return spl_ff_state<N, STAR>(kk, F, hf, x, v, a0, da, j0, q2, d2, sa, sj);
}
template <int N, bool STAR>
static __device__ __noinline__ int spl_hermite_ff_step_call(const F64k &kk, const FMass<N> &F, const FCoef &C, float hf,
                                                     int n_corr, double (&x)[N][3], double (&v)[N][3],
                                                     double (&a0)[N][3], float (&da)[N][3], ff (&j0)[N][3],
                                                     float (&q2)[N], float (&d2)[N][N], ff (&sa)[3], ff (&sj)[3]) {
  spl_hermite_ff_advance<N>(kk, F, C, n_corr, x, v, a0, da, j0);
  return spl_ff_state<N, STAR>(kk, F, hf, x, v, a0, da, j0, q2, d2, sa, sj);
}

template <int N>
static __device__ __noinline__ int spl_hermite_delta_step_call(const F64k &kk, const FMass<N> &F, const FCoef &C, float hf,
                                                        int n_corr, double (&x)[N][3], double (&v)[N][3],
                                                        double (&a0)[N][3], float (&da)[N][3], ff (&j0)[N][3],
                                                        float (&q2)[N], float (&d2)[N][N], ff (&sa)[3], ff (&sj)[3]) {
  return spl_hermite_delta_step<N, false>(kk, F, C, hf, n_corr, x, v, a0, da, j0, q2, d2, sa, sj);
}

// The monitor (Algorithm 1) after a step in pairs to a state of the given level.  A state of
// level 1 or 2 is finite (`spl_ff_state`), and its tests start from the FP32 distances (kcf = 2 kc, ejf = the
// squared ejection radius, both moved 2^-9 to the safe side); what comes near a limit, and
// any state of level 0, is tested in FP64.
template <int N>
struct FLimits {
  double kc[N][N];
  float kcf[N][N], ejf;
};
template <int N>
__device__ __forceinline__ FLimits<N> flimits(const double (&m)[N], double ce_factor, double eject2) {
  FLimits<N> L;
  L.ejf = eject2 > 0.0 ? 0.998f * (float)eject2 : __int_as_float(0x7f800000);
#pragma unroll
  for (int i = 1; i < N; i++)
#pragma unroll
    for (int k = i + 1; k < N; k++) {
      L.kc[i][k] = hill_kc(ce_factor, m[i], m[k], m[0]);
      L.kcf[i][k] = 2.004f * (float)L.kc[i][k];
    }
  return L;
}
template <int N>
static __device__ __noinline__ int spl_ff_monitor_fp64(const F64k &kk, const double (&x)[N][3], const double (&v)[N][3],
                                                const double (&kc)[N][N], double eject2) {
  double q2[N], d2[N][N];
#pragma unroll
  for (int i = 1; i < N; i++) {
    q2[i] = fma(x[i][2], x[i][2], fma(x[i][1], x[i][1], kmul(kk, x[i][0], x[i][0])));
#pragma unroll
    for (int j = i + 1; j < N; j++) {
      double d[3];
#pragma unroll
      for (int c = 0; c < 3; c++) d[c] = ksub(kk, x[j][c], x[i][c]);
      d2[i][j] = fma(d[2], d[2], fma(d[1], d[1], kmul(kk, d[0], d[0])));
    }
  }
  return spl_monitor<N>(kk, x, v, q2, d2, kc, eject2);
}
template <int N>
__device__ __forceinline__ int spl_ff_monitor(const F64k &kk, int level, const FLimits<N> &L, const float (&q2)[N],
                                              const float (&d2)[N][N], const double (&x)[N][3], const double (&v)[N][3],
                                              double eject2) {
  bool near = level == 0;
#pragma unroll
  for (int i = 1; i < N; i++) {
    near |= !(q2[i] < L.ejf);
#pragma unroll
    for (int j = i + 1; j < N; j++) near |= !(d2[i][j] >= L.kcf[i][j] * (q2[i] + q2[j]));
  }
  return near ? spl_ff_monitor_fp64<N>(kk, x, v, L.kc, eject2) : 0;
}

// The inertial state (barycentre moved by its velocity times `elapsed`) into the bin, or its
// energy record into the log.
template <int N>
__device__ __forceinline__ void spl_write(const BinView &B, int s, const double (&m)[N], const double (&x)[N][3],
                                          const double (&v)[N][3], double Minv, const double (&Xc)[3],
                                          const double (&Vc)[3], double elapsed, const StepParams *log, double t) {
  const int SP = B.S_pad;
  double xo[N][3], vo[N][3], Xe[3];
#pragma unroll
  for (int c = 0; c < 3; c++) Xe[c] = fma(elapsed, Vc[c], Xc[c]);
  spl_from_rel<N>(m, x, v, Minv, Xe, Vc, xo, vo);
  if (log) {
    double e[4];
    spl_energy<N>(xo, vo, m, e);
    write_log(*log, B.gidx[s], t, e);
    return;
  }
#pragma unroll
  for (int i = 0; i < N; i++)
#pragma unroll
    for (int c = 0; c < 3; c++) {
      B.x[(size_t)(c * N + i) * SP + s] = xo[i][c];
      B.v[(size_t)(c * N + i) * SP + s] = vo[i][c];
    }
}

// 1/a, and 1/sqrt(a), as pairs
__device__ __forceinline__ ff ff_div(const ff &a, const ff &b) {
  const float r = __frcp_rn(b.h);
  const float q = __fmul_rn(a.h, r);
  const ff d = ff_sub(a, ff_mulf(b, q));
  return fast_two_sum(q, __fmul_rn(d.h, r));
}
__device__ __forceinline__ ff ff_rsqrt(const ff &a) {
  const float y = rsqrtf(a.h);
  const ff p = ff_mul(a, two_prod(y, y));
  const float t = __fsub_rn(__fsub_rn(1.0f, p.h), p.l);
  return fast_two_sum(y, __fmul_rn(__fmul_rn(0.5f, y), __fmaf_rn(0.75f, __fmul_rn(t, t), t)));
}
// |j|^2/|a|^2 of a body.  Body 0's vectors have the planets' masses, whose squares (and their lower
// words first) leave FP32's range: both vectors are taken times the power of two that brings a to
// 1, which is exact.  NaN, which sends the step to FP64, for a body whose own components are so
// small that they have lost bits.
__device__ __forceinline__ ff ff_eq5_term(const ff (&a)[3], const ff (&j)[3]) {
  const float A = fmaxf(fmaxf(fabsf(a[0].h), fabsf(a[1].h)), fabsf(a[2].h));
  const float J = fmaxf(fmaxf(fabsf(j[0].h), fabsf(j[1].h)), fabsf(j[2].h));
  const float s = __int_as_float(0x7f000000 - (__float_as_int(A) & 0x7f800000));
  ff as[3], js[3];
#pragma unroll
  for (int c = 0; c < 3; c++) {
    as[c] = ff_make(s * a[c].h, s * a[c].l);
    js[c] = ff_make(s * j[c].h, s * j[c].l);
  }
  const ff r = ff_div(ff_norm2(js), ff_norm2(as));
  return A > 0x1p-100f && J > 0x1p-100f ? r : ff_make(__int_as_float(0x7fffffff), 0.0f);
}
// Eq. 5's step tau (sum_i |j_i|^2/|a_i|^2)^(-1/2) over the inertial accelerations and jerks, in
// pairs (relative error 2^-44: the step's length, not the state, takes it).
template <int N>
__device__ __forceinline__ ff spl_ff_eq5(const ff &tau, const double (&a0)[N][3], const float (&da)[N][3],
                                         const ff (&j0)[N][3], const ff (&sa)[3], const ff (&sj)[3]) {
  ff a[3], j[3];
#pragma unroll
  for (int c = 0; c < 3; c++) {
    a[c] = ff_norm(sa[c]);
    j[c] = ff_norm(sj[c]);
  }
  ff sum = ff_eq5_term(a, j);
#pragma unroll
  for (int k = 1; k < N; k++) {
#pragma unroll
    for (int c = 0; c < 3; c++) {
      const ff A = ff_from(a0[k][c]);
      a[c] = ff_add(ff_make(A.h, A.l + da[k][c]), sa[c]);
      j[c] = ff_add(j0[k][c], sj[c]);
    }
    sum = ff_add(sum, ff_eq5_term(a, j));
  }
  return ff_mul(tau, ff_rsqrt(sum));
}

}  // namespace swarm
