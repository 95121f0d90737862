// Mixed-variable steps (mvs_impl.cuh) with the FP64 pipe kept for the state and the drift's root.
//
// Per step and planet the FP64 pipe gets the drift's 54 instructions (kepler_ff.cuh), the two
// kicks (6) and, in democratic heliocentric coordinates, the two Cartesian drifts (6) and the
// new distance (6).  The interaction's accelerations and the star's reflex sum carry the
// planets' masses over the star's, so they are formed as float pairs:
//   - the ring runs over the n - 1 planets, whose positions keep all 53 bits (`ff3`), so that a
//     difference vector is good to 2^-48 of itself however close the pair is;
//   - Jacobi: with g = Q/|Q|^3 of the heliocentric position Q = r' + D, D = sum_{k<b} w_k r'_k,
//     and A the planets' pulls, the acceleration (mu r'/|r'|^3 and the Jacobi component of all
//     the pulls, which cancel to first order) is
//       (eta_b/eta_{b-1}) [m0 (r'/|r'|^3 - g) + A] - sum_{j>b} m_j (m0 g_j - A_j) / eta_{b-1};
//     the difference is taken algebraically: with s = |Q|^2/|r'|^2 - 1 = (2 r' + D).D/|r'|^2 and
//     e = 1 - (1+s)^(-3/2) it is (Q e - D)/|r'|^3.  No term of the star's full pull is left, so
//     a pair's 2^-44 is relative to the planets' masses.
// Checked at every evaluation: h |terms| <= 2^-8 |u| (the kick's error is then 2^-53 u), the
// reflex drift likewise against |r|, and the range of FP32; a system for which one fails takes
// that part in FP64 (mvs_acc, grp_sum).  All these choices follow from the system's own state,
// so that a system alone and in an ensemble moves bit for bit alike.  The monitor's tests run
// in FP32 with a margin and, where one of them is met, again in FP64.
//
// Bound: the FP64 pipe (79 instructions per warp and step at n = 8 Jacobi, 68 % busy with three
// CTAs per SM) and the latency of the drift's chain of 3200 instructions (a step of one system
// alone: 6.6 us), so 168 registers for three warps per sub-partition (two: 1.31 ms for 40 steps of
// 16384 systems, three: 1.18).  Before, wholly in FP64, -> now: 16384 Jacobi systems of 8 bodies
// over 500 steps 24.8 -> 8.5 ms, 3001 DH systems of 3..15 bodies over 300 steps 12.2 -> 3.1 ms,
// one system alone 9.9 -> 6.6 us per step (the former spread over a warp's idle groups).
// A FP64 form of a part costs its warp as much as before: the drift 5 us, the accelerations 3 us.
#pragma once
#include "hermite_bpl_ff.cuh"
#include "kepler_ff.cuh"
#include "mvs_impl.cuh"

namespace swarm {

__device__ __forceinline__ ff3 ff3_add(const ff3 &a, const ff &b) {
  const ff s = two_sum(a.h, b.h), n = two_sum(a.l, b.l), m = two_sum(n.h, s.l);
  ff3 r;
  r.h = s.h;
  r.l = m.h;
  r.t = __fadd_rn(__fadd_rn(m.l, n.l), a.t);
  return r;
}
__device__ __forceinline__ ff ff3_sub(const ff3 &a, const ff3 &b) {
  const ff s = two_sum(a.h, -b.h), m = two_sum(a.l, -b.l), v = two_sum(s.h, m.h);
  return ff_make(v.h, __fadd_rn(v.l, __fadd_rn(s.l, __fadd_rn(m.l, __fsub_rn(a.t, b.t)))));
}
__device__ __forceinline__ ff3 shfl_ff3(const ff3 &a, int src) {
  ff3 r;
  r.h = __shfl_sync(0xffffffffu, a.h, src);
  r.l = __shfl_sync(0xffffffffu, a.l, src);
  r.t = __shfl_sync(0xffffffffu, a.t, src);
  return r;
}

// sums over the group's lanes before (after) this one; every lane of the warp takes part
template <int N, bool AFTER>
__device__ __forceinline__ ff grp_scan_ff(const BplBody<N> &g, ff v) {
  const unsigned FULL = 0xffffffffu;
  auto from = [&](float f, int off) { return AFTER ? __shfl_down_sync(FULL, f, off) : __shfl_up_sync(FULL, f, off); };
  auto in = [&](int off) { return AFTER ? g.b + off < g.n() : g.b >= off; };
#pragma unroll
  for (int off = 1; off < (N ? N : 32); off <<= 1) {
    const ff o = ff_make(from(v.h, off), from(v.l, off));
    if (in(off)) v = ff_add_raw(v, o);
  }
  const ff o = ff_make(from(v.h, 1), from(v.l, 1));
  return in(1) ? ff_norm(o) : ff_make(0.0f, 0.0f);
}
template <int N>
__device__ __forceinline__ float grp_after32(const BplBody<N> &g, float v) {
  const unsigned FULL = 0xffffffffu;
#pragma unroll
  for (int off = 1; off < (N ? N : 32); off <<= 1) {
    const float o = __shfl_down_sync(FULL, v, off);
    if (g.b + off < g.n()) v += o;
  }
  const float o = __shfl_down_sync(FULL, v, 1);
  return g.b + 1 < g.n() ? o : 0.0f;
}

// ---------------------------------------------------------------- FP64 forms (cold)
struct MvsMass {
  double m0, Minv, eta_prev_inv, w, mu;
};
template <int N, bool JAC>
__device__ __forceinline__ MvsMass mvs_mass(double m, int b, int base) {
  MvsMass M;
  M.m0 = shfl(m, base);
  M.Minv = 1.0 / grp_sum<N>(m, b, base);
  const double eta = grp_scan_excl<N>(m, b) + m;
  const double eta_prev = eta - m;
  M.eta_prev_inv = b == 0 ? 0.0 : 1.0 / eta_prev;
  M.w = m / eta;
  M.mu = JAC ? (b == 0 ? M.m0 : M.m0 * eta * M.eta_prev_inv) : M.m0;
  return M;
}
template <int N, bool JAC>
static __device__ __noinline__ void mvs_acc_fp64(const F64k &k, const double (&q)[3], double m, int b, int base,
                                                 double (&acc)[3]) {
  const MvsMass M = mvs_mass<N, JAC>(m, b, base);
  mvs_acc<N, JAC>(k, q, m, M.w, M.eta_prev_inv, M.mu, b, base, acc);
}
template <int N>
static __device__ __noinline__ void mvs_reflex_fp64(const F64k &k, const double (&u)[3], double m, int b, int base,
                                                    double (&p)[3]) {
  const double m0inv = 1.0 / shfl(m, base);
#pragma unroll
  for (int c = 0; c < 3; c++) {
    const double s = grp_sum<N>(k, b == 0 ? 0.0 : kmul(k, m, u[c]), b, base);
    p[c] = b == 0 ? u[c] : s * m0inv;
  }
}
static __device__ __noinline__ bool mvs_drift_fp64(const F64k &k, bool on, double mu, double (&r)[3], double (&v)[3],
                                                   double h, int &its, double &rq, double &r2) {
  const KepConst K = kep_const(mu);
  const bool ok = kepler_drift<false>(k, on, K, r, v, h, its, rq);
  r2 = fma(r[2], r[2], fma(r[1], r[1], kmul(k, r[0], r[0])));
  return ok;
}
// the status code of the group's state (0: none); w: Jacobi's m_b/eta_b; kc: the planets' ring's
// close-encounter coefficients; ok: the drift converged
template <int N, bool JAC>
static __device__ __noinline__ int mvs_code_fp64(const StepParams &P, const BplBody<N> &g, const double (&q)[3],
                                                 const double (&u)[3], double w, const double *kc, bool ok) {
  const unsigned FULL = 0xffffffffu, gm = g.mask();
  double Q[3] = {q[0], q[1], q[2]};
  if (JAC) jacobi_helio<N>(P.fk, q, w, g.b, Q);
  const double q2 = fma(Q[2], Q[2], fma(Q[1], Q[1], kmul(P.fk, Q[0], Q[0])));
  const bool nf = nonfinite(q[0]) | nonfinite(q[1]) | nonfinite(q[2]) | nonfinite(u[0]) | nonfinite(u[1]) | nonfinite(u[2]);
  const bool ej = g.b != 0 && P.eject2 > 0.0 && q2 > P.eject2;
  bool ce = false;
#pragma unroll 1
  for (int r = 1; r <= g.RT(); r++) {
    const int p = g.next(r);
    double d2 = 0.0;
#pragma unroll
    for (int c = 0; c < 3; c++) {
      const double d = ksub(P.fk, shfl(Q[c], p), Q[c]);
      d2 = fma(d, d, d2);
    }
    const double q2p = shfl(q2, p);
    if (g.b != 0 && kc[r - 1] > 0.0 && close_encounter(P.fk, d2, kc[r - 1], q2, q2p)) ce = true;
  }
  const unsigned bnf = __ballot_sync(FULL, nf) & gm, bkn = __ballot_sync(FULL, !ok) & gm;
  const unsigned bej = __ballot_sync(FULL, ej) & gm, bce = __ballot_sync(FULL, ce) & gm;
  return bkn ? SWARM_SYS_KEPLER_NOCONV
             : bnf ? SWARM_SYS_NONFINITE : bej ? SWARM_SYS_EJECTED : bce ? SWARM_SYS_CLOSE_ENCOUNTER : 0;
}

// ---------------------------------------------------------------- one system's lane
template <int N, bool JAC>
struct MvsLane {
  int s = 0, kg = 0;
  bool has = false, scaled = false;
  double m = 1.0, mu = 1.0, t0 = 0.0;
  // Jacobi: w = m_b/eta_b, gr = eta_b/eta_{b-1}, ei = 1/eta_{b-1}; DH: md = m_b/m_0
  ff w, gr, ei;
  LaunchPlan plan;
  double q[3] = {0.0, 0.0, 0.0}, u[3] = {0.0, 0.0, 0.0}, acc[3] = {0.0, 0.0, 0.0};
  double p[3] = {0.0, 0.0, 0.0};  // DH: the star's reflex sum m_j u_j / m_0 (lane 0: its velocity)
  double rq = 1.0, r2 = 1.0;      // Jacobi: 1/|q|, |q|^2
};

// Close-encounter coefficients of the lane's ring pairs, and in FP32 with a margin: 2^-17 for
// the arithmetic's rounding, in DH 2^-7 for the Cartesian drift that follows the test (below
// 2^-9 |q|, see mvs_reflex; the sum of two distances squared then moves by 2^-8 at most).
template <int N>
struct MvsKc {
  double kc[kRoundsA<N>];
  float kcf[kRoundsA<N>];
};

// Accelerations at q (has: the lane's system counts for the choices; hf = |h|).  Also |Q|^2 of the
// heliocentric position, and whether a pair is near the close-encounter limit.
template <int N, bool JAC>
__device__ __forceinline__ void mvs_force(const F64k &k, const BplBody<N> &g, const MvsLane<N, JAC> &L, bool has,
                                          float hf, const double (&q)[3], const double (&u)[3], double rq,
                                          const float *kcf, double (&acc)[3], float &q2, bool &near) {
  const bool star = g.b == 0;
  ff3 X[3];
  ff E[3], gp[3];  // Jacobi: r'/|r'|^3 - g, and g
  float W = 0.0f, gf = 0.0f;
#pragma unroll
  for (int c = 0; c < 3; c++) X[c] = ff3_from(q[c]);
  if (JAC) {
    ff D[3], t[3];
#pragma unroll
    for (int c = 0; c < 3; c++) {
      const ff qf = ff_make(X[c].h, X[c].l);
      D[c] = grp_scan_ff<N, false>(g, star ? ff_make(0.0f, 0.0f) : ff_mul_raw(L.w, qf));
      t[c] = ff_add_raw(ff_make(2.0f * qf.h, 2.0f * qf.l), D[c]);
      X[c] = ff3_add(X[c], D[c]);
    }
    const ff y = ff_norm(ff_from(rq)), y2 = ff_mul(y, y), y3 = ff_mul(y2, y);
    const ff s = ff_mul(ff_dot(t, D), y2);
    ff R, R1;
    ff_rho3(ff_add(ff_make(1.0f, 0.0f), s), R, R1);
    // e = s (3 + 3 s + s^2) R^2 / (1 + R), R = (1 + s)^(-3/2)
    const ff three = ff_make(3.0f, 0.0f);
    const ff e = ff_div(ff_mul(ff_mul(R, R), ff_mul(s, ff_fma(s, ff_add(three, s), three))), ff_add(ff_make(1.0f, 0.0f), R));
    const ff s3 = ff_mul(R, y3);
#pragma unroll
    for (int c = 0; c < 3; c++) {
      const ff Q = ff_make(X[c].h, X[c].l);
      E[c] = ff_mul(y3, ff_sub(ff_mul(e, Q), D[c]));
      gp[c] = ff_mul_raw(s3, Q);
      W += fabsf(E[c].h) + fabsf(y3.h * e.h * Q.h);
    }
    W *= g.m0f.h;
  }
  q2 = __fmaf_rn(X[2].h, X[2].h, __fmaf_rn(X[1].h, X[1].h, __fmul_rn(X[0].h, X[0].h)));
  const float qi = rsqrtf(q2), qa = q2 * qi;
  gf = qi * qi;
  bool range = L.scaled && frange(q2);
#pragma unroll
  for (int c = 0; c < 3; c++) range = range && abs_below_pow2(q[c], 40) && abs_below_pow2(u[c], 40);
  near = false;
  ff A[3];
  float S = 0.0f;
#pragma unroll
  for (int c = 0; c < 3; c++) A[c] = ff_make(0.0f, 0.0f);
#pragma unroll kRingUnroll<N>
  for (int r = 1; r <= g.RT(); r++) {
    const int p = g.next(r), o = g.prev(r);
    ff dx[3], s3, s2;
#pragma unroll
    for (int c = 0; c < 3; c++) dx[c] = ff3_sub(shfl_ff3(X[c], p), X[c]);
    const ff r2 = ff_norm2(dx);
    ff_rho3(r2, s3, s2);
    const ff mp = shfl_ff(g.mf, p);
#pragma unroll
    for (int c = 0; c < 3; c++) {
      dx[c] = ff_mul_raw(s3, dx[c]);
      A[c] = ff_fma_raw(mp, dx[c], A[c]);
    }
    S = __fmaf_rn(mp.h, s2.h, S);
    range = range && frange(r2.h);
    const float qs = qa + __shfl_sync(0xffffffffu, qa, p);
    near |= !(r2.h >= kcf[r - 1] * (qs * qs));
    if (r <= g.RF()) {  // the pair that lane o evaluated with this one
      const ff mo = ff_neg(shfl_ff(g.mf, o));
#pragma unroll
      for (int c = 0; c < 3; c++) A[c] = ff_fma_raw(mo, shfl_ff(dx[c], o), A[c]);
      S = __fmaf_rn(-mo.h, __shfl_sync(0xffffffffu, s2.h, o), S);
    }
  }
  W += S;
  if (JAC) {
    const ff mm = star ? ff_make(0.0f, 0.0f) : g.mf;
    const float ss = grp_after32<N>(g, mm.h * __fmaf_rn(g.m0f.h, gf, S));
    W = __fmaf_rn(ss, L.ei.h, W);
#pragma unroll
    for (int c = 0; c < 3; c++) {
      const ff t = grp_scan_ff<N, true>(g, ff_mul(mm, ff_sub(ff_mul(g.m0f, gp[c]), A[c])));
      const ff d = ff_fma(g.m0f, E[c], A[c]);
      A[c] = ff_sub(ff_mul(L.gr, d), ff_mul(L.ei, t));
    }
  }
#pragma unroll
  for (int c = 0; c < 3; c++) acc[c] = star ? 0.0 : ff_double(ff_norm(A[c]));
  const float uf[3] = {f_from(u[0]), f_from(u[1]), f_from(u[2])};
  const float V2 = __fmaf_rn(uf[2], uf[2], __fmaf_rn(uf[1], uf[1], __fmul_rn(uf[0], uf[0])));
  const float w = hf * W;
  const bool bad = has && !star && !(range && w * w <= 0x1p-16f * V2);
  if (__any_sync(0xffffffffu, bad)) {
    const unsigned bm = __ballot_sync(0xffffffffu, bad) & g.mask();
    double qc[3] = {q[0], q[1], q[2]}, a[3];
    mvs_acc_fp64<N, JAC>(k, qc, L.m, g.b, g.base, a);
    if (bm) {
#pragma unroll
      for (int c = 0; c < 3; c++) acc[c] = a[c];
      near = true;  // the monitor in FP64
    }
  }
}

// DH: p = sum_j m_j u_j / m_0 (Eq. of the Cartesian drift)
template <int N>
__device__ __forceinline__ void mvs_reflex(const F64k &k, const BplBody<N> &g, const MvsLane<N, false> &L, bool has,
                                           float hf, float q2, const double (&u)[3], double (&p)[3]) {
  const bool star = g.b == 0;
  float V2 = 0.0f;
  bool range = L.scaled && frange(q2);
#pragma unroll
  for (int c = 0; c < 3; c++) {
    range = range && abs_below_pow2(u[c], 40);
    const ff uf = ff_norm(ff_from(u[c]));
    V2 = __fmaf_rn(uf.h, uf.h, V2);
    const ff s = shfl_ff(grp_planets_ff<N>(g, ff_mul_raw(L.w, uf)), g.base);
    p[c] = star ? u[c] : ff_double(s);
  }
  const float w = hf * __shfl_sync(0xffffffffu, grp_planets32<N>(g, L.w.h * __fsqrt_rn(V2)), g.base);
  const bool bad = has && !star && !(range && w * w <= 0x1p-16f * q2);
  if (__any_sync(0xffffffffu, bad)) {
    const unsigned bm = __ballot_sync(0xffffffffu, bad) & g.mask();
    double uc[3] = {u[0], u[1], u[2]}, a[3];
    mvs_reflex_fp64<N>(k, uc, L.m, g.b, g.base, a);
    if (bm)
#pragma unroll
      for (int c = 0; c < 3; c++) p[c] = a[c];
  }
}

// the group's system, from the stored state; take: the lanes that take one (every lane of the
// warp executes this)
template <int N, bool JAC>
__device__ __forceinline__ void mvs_load(const BinView &B, const StepParams &P, const BplBody<N> &g0, BplBody<N> &g,
                                         MvsLane<N, JAC> &L, bool take, int ss, bool lane_ok, MvsKc<N> &kc) {
  const int SP = B.S_pad, b = g0.b, base = g0.base;
  const int sl = take ? ss : L.s;  // a valid row for every lane's loads
  MvsLane<N, JAC> M;
  BplBody<N> gn = g0;
  double x[3], v[3];
#pragma unroll
  for (int c = 0; c < 3; c++) {
    x[c] = B.x[(size_t)(c * N + b) * SP + sl];
    v[c] = B.v[(size_t)(c * N + b) * SP + sl];
  }
  M.m = B.m[(size_t)b * SP + sl];
  const MvsMass W = mvs_mass<N, JAC>(M.m, b, base);
  M.mu = W.mu;
  gn.m0 = W.m0;
  gn.m0f = ff_norm(ff_from(W.m0));
  gn.mf = ff_norm(ff_from(M.m));
  if (JAC) {
    M.w = ff_norm(ff_from(W.w));
    M.gr = ff_norm(ff_from(1.0 + M.m * W.eta_prev_inv));
    M.ei = ff_norm(ff_from(W.eta_prev_inv));
  } else {
    M.w = ff_norm(ff_from(M.m / W.m0));
    M.gr = M.ei = ff_make(0.0f, 0.0f);
  }
  M.scaled = (__ballot_sync(0xffffffffu, !fmass_ok(M.m, b == 0)) & g0.mask()) == 0 && fscale(P.dt, -60, 40);
  MvsKc<N> kk;
#pragma unroll 1
  for (int r = 1; r <= kRoundsA<N>; r++) {
    const double mp = shfl(M.m, g0.next(r));
    kk.kc[r - 1] = r <= g0.RT() ? hill_kc(P.ce_factor, M.m, mp, W.m0) : 0.0;
    kk.kcf[r - 1] = (JAC ? 1.00001f : 1.008f) * (float)kk.kc[r - 1];
  }
  if (JAC) to_jacobi<N>(x, v, M.m, W.Minv, W.eta_prev_inv, b, base, M.q, M.u);
  else to_dh<N>(x, v, M.m, W.Minv, b, base, M.q, M.u);
  M.r2 = fma(M.q[2], M.q[2], fma(M.q[1], M.q[1], kmul(P.fk, M.q[0], M.q[0])));
  M.rq = rsqrt(M.r2);
  const double tn = B.t[sl];
  const bool runnable = take && B.status[sl] <= SWARM_SYS_DONE;
  M.plan = launch_plan(B, P, sl, tn, runnable);
  M.t0 = tn;
  M.s = sl;
  M.kg = 0;
  M.has = runnable && M.plan.N > 0;
  if (runnable && M.plan.N == 0 && lane_ok && b == 0) B.status[sl] = SWARM_SYS_DONE;
  float q2;
  bool near;
  mvs_force<N, JAC>(P.fk, gn, M, M.has, P.fc.hf, M.q, M.u, M.rq, kk.kcf, M.acc, q2, near);
  if constexpr (!JAC) mvs_reflex<N>(P.fk, gn, M, M.has, P.fc.hf, q2, M.u, M.p);
  if (take) {
    L = M;
    g = gn;
    kc = kk;
  }
}

// One step of every group holding a system; on a finish or log point the results are written.
// Returns whether the lane's system finished.
template <int N, bool JAC>
__device__ __forceinline__ bool mvs_step(const BinView &B, const StepParams &P, const BplBody<N> &g, MvsLane<N, JAC> &L,
                                         bool lane_ok, const MvsKc<N> &kc, float ejf, unsigned long long &kep_iters) {
  constexpr unsigned long long NP = JAC ? (unsigned long long)N * (N - 1) / 2 : (unsigned long long)(N - 1) * (N - 2) / 2;
  const unsigned FULL = 0xffffffffu;
  const int b = g.b, base = g.base, SP = B.S_pad;
  const bool active = L.has, star = b == 0;
  if (active) L.kg++;
  const double h = (active && L.kg == L.plan.N && !L.plan.exact) ? L.plan.h_last : P.dt;
  const double hh = 0.5 * h;
  if (!JAC) {
#pragma unroll
    for (int c = 0; c < 3; c++) L.q[c] = fma(hh, L.p[c], L.q[c]);
    L.r2 = fma(L.q[2], L.q[2], fma(L.q[1], L.q[1], kmul(P.fk, L.q[0], L.q[0])));
    L.rq = rsqrt_ff(P.fk, L.r2);
  }
#pragma unroll
  for (int c = 0; c < 3; c++) L.u[c] = fma(hh, L.acc[c], L.u[c]);
  bool ok = true;
  int its = star ? 0 : 1;
  {
    double r[3] = {L.q[0], L.q[1], L.q[2]}, v[3] = {L.u[0], L.u[1], L.u[2]}, rq = L.rq, r2 = L.r2;
    bool took = kepler_drift_ff<JAC>(P.fk, star, L.mu, r, v, h, rq, r2);
    took = star || (took && L.scaled);
    if (took) {
#pragma unroll
      for (int c = 0; c < 3; c++) {
        L.q[c] = r[c];
        L.u[c] = v[c];
      }
      L.rq = rq;
      L.r2 = r2;
    }
    const bool slow = active && !took;
    if (__any_sync(FULL, slow)) {
      double rc[3] = {L.q[0], L.q[1], L.q[2]}, vc[3] = {L.u[0], L.u[1], L.u[2]}, rqc = L.rq, r2c = L.r2;
      int ic = 0;
      const bool okc = mvs_drift_fp64(P.fk, slow, L.mu, rc, vc, h, ic, rqc, r2c);
      if (slow) {
        ok = okc;
        its = ic;
#pragma unroll
        for (int c = 0; c < 3; c++) {
          L.q[c] = rc[c];
          L.u[c] = vc[c];
        }
        L.rq = rqc;
        L.r2 = r2c;
      }
    }
  }
  if (active && lane_ok) kep_iters += its;
  float q2;
  bool look;
  mvs_force<N, JAC>(P.fk, g, L, active, P.fc.hf, L.q, L.u, L.rq, kc.kcf, L.acc, q2, look);
#pragma unroll
  for (int c = 0; c < 3; c++) L.u[c] = fma(hh, L.acc[c], L.u[c]);
  if constexpr (!JAC) {
    mvs_reflex<N>(P.fk, g, L, active, P.fc.hf, q2, L.u, L.p);
#pragma unroll
    for (int c = 0; c < 3; c++) L.q[c] = fma(hh, L.p[c], L.q[c]);
    const float x = f_from(L.q[0]), y = f_from(L.q[1]), z = f_from(L.q[2]);
    q2 = __fmaf_rn(z, z, __fmaf_rn(y, y, __fmul_rn(x, x)));
  }
  // monitor at the end of the step: FP32 tests with a margin, then FP64 ones
  look = !star && (look || !(q2 < ejf));
  {
    int e = 0;
#pragma unroll
    for (int c = 0; c < 3; c++) e = max(e, max(__double2hiint(L.q[c]) & 0x7fffffff, __double2hiint(L.u[c]) & 0x7fffffff));
    look = active && (look || !ok || e >= (1023 + 40) << 20);
  }
  int code = 0;
  if (__any_sync(FULL, look)) {
    double qc[3] = {L.q[0], L.q[1], L.q[2]}, uc[3] = {L.u[0], L.u[1], L.u[2]};
    code = mvs_code_fp64<N, JAC>(P, g, qc, uc, ff_double(L.w), kc.kc, ok);
  }
  const bool finish = active && (code != 0 || L.kg == L.plan.N);
  const bool want_log = active && !code && P.log_interval > 0 && (L.kg % P.log_interval) == 0;
  if (__any_sync(FULL, finish || want_log)) {
    const MvsMass M = mvs_mass<N, JAC>(L.m, b, base);
    double xo[3], vo[3];
    if (JAC) from_jacobi<N>(L.q, L.u, M.w, b, base, xo, vo);
    else from_dh<N>(L.q, L.u, L.m, M.m0, M.Minv, b, base, xo, vo);
    const double tk = step_time(L.plan, L.kg, L.t0, P.dt);
    if (__any_sync(FULL, want_log)) {  // the energy sum is a warp collective
      double e[4];
      ring_energy<N>(xo, vo, L.m, b, base, e);
      if (want_log && lane_ok && b == 0) write_log(P, B.gidx[L.s], tk, e);
    }
    if (finish && lane_ok) {
#pragma unroll
      for (int c = 0; c < 3; c++) {
        B.x[(size_t)(c * N + b) * SP + L.s] = xo[c];
        B.v[(size_t)(c * N + b) * SP + L.s] = vo[c];
      }
      if (b == 0) {
        B.t[L.s] = tk;
        B.status[L.s] = code ? code : (L.plan.full ? SWARM_SYS_DONE : SWARM_SYS_ACTIVE);
        if (P.counters) {
          atomicAdd(&P.counters[0], (unsigned long long)L.kg);
          atomicAdd(&P.counters[1], NP * (1ull + (unsigned long long)L.kg));
        }
      }
    }
  }
  return finish;
}

// Systems handed out one by one to the warp's groups: take(need, leader, base) gives the group's
// next system or -1 (every lane calls it).  A refill costs the warp one round (the new systems'
// coordinate maps and first evaluation) during which the other groups wait.
template <int N, bool JAC, class Take>
__device__ __forceinline__ void bpl_mvs_run(const BinView &B, const StepParams &P, int ga, Take take) {
  constexpr int G = 32 / N;
  const unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  int grp = lane / N;
  BplBody<N> g;
  g.b = lane - grp * N;
  const bool lane_ok = grp < G;
  if (!lane_ok) {  // spare lanes replicate group 0's, without a system of their own
    grp = 0;
    g.b = lane - G * N;
  }
  g.base = grp * N;
  g.nn = N;
  g.m0 = 1.0;
  g.m0f = g.mf = ff_make(1.0f, 0.0f);
  MvsLane<N, JAC> L;
  L.w = L.gr = L.ei = ff_make(0.0f, 0.0f);
  L.plan.N = 0;
  L.plan.full = L.plan.exact = 1;
  L.plan.h_last = P.dt;
  L.plan.t_end = P.t_end;
  MvsKc<N> kc;
#pragma unroll
  for (int r = 0; r < kRoundsA<N>; r++) kc.kc[r] = kc.kcf[r] = 0.0f;
  const float ejf = P.eject2 > 0.0 ? 0.99999f * (float)P.eject2 : __int_as_float(0x7f800000);
  bool exhausted = !lane_ok || grp >= ga;
  unsigned long long kep_iters = 0;
  for (;;) {
    const bool need = !L.has && !exhausted;
    if (__any_sync(FULL, need)) {
      const int ss = take(need, lane_ok && g.b == 0, g.base);
      const bool got = need && ss >= 0;
      if (need && ss < 0) exhausted = true;
      const BplBody<N> g0 = g;
      mvs_load<N, JAC>(B, P, g0, g, L, got, ss, lane_ok, kc);
      continue;
    }
    if (!__any_sync(FULL, L.has)) break;
    if (mvs_step<N, JAC>(B, P, g, L, lane_ok, kc, ejf, kep_iters)) L.has = false;
  }
  if (P.counters && lane_ok && kep_iters) atomicAdd(&P.counters[2], kep_iters);
}

// one work unit: the G systems from unit * G on
template <int N, bool JAC>
__device__ __noinline__ void bpl_mvs_unit(const BinView &B, const StepParams &P, int unit) {
  constexpr int G = 32 / N;
  bool given = false;
  bpl_mvs_run<N, JAC>(B, P, G, [&](bool need, bool, int base) {
    const int s = unit * G + base / N;
    const bool go = need && !given && s < B.S;
    if (need) given = true;
    return go ? s : -1;
  });
}

// Persistent kernel for one bin: every warp streams systems through its groups until the
// bin's counter runs out (work unit = system).
template <int N, bool JAC>
__global__ void __launch_bounds__(128, 3) mvs_uniform_kernel(BinView B, int nunits, StepParams P) {
  (void)nunits;
  // Groups that take systems: as many per warp as the launch's systems need to be all in
  // flight at once (at most G).
  constexpr int G = 32 / N;
  const long long warps = (long long)gridDim.x * (blockDim.x >> 5);
  const long long per = ((long long)stream_count(B) + warps - 1) / warps;
  const int ga = per < 1 ? 1 : per < G ? (int)per : G;
  bpl_mvs_run<N, JAC>(B, P, ga, [&](bool need, bool leader, int base) {
    int sn = 0;
    if (need && leader) sn = atomicAdd(P.work_next, 1);
    sn = __shfl_sync(0xffffffffu, sn, base);
    return need ? stream_system(B, sn) : -1;
  });
}

template <int N, bool JAC>
cudaError_t launch_mvs_uniform_n(const BinView &B, int nunits, const StepParams &P, int grid, cudaStream_t st) {
  StepParams Q = P;
  Q.fc = fcoef_host(P.dt);
  mvs_uniform_kernel<N, JAC><<<grid, 128, 0, st>>>(B, nunits, Q);
  return cudaGetLastError();
}
template <int N, bool JAC>
int mvs_uniform_blocks_n() {
  int nb = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, mvs_uniform_kernel<N, JAC>, 128, 0);
  return nb;
}

}  // namespace swarm
