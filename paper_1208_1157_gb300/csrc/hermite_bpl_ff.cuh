// Hermite-4, body per lane: the steps of hermite_ff.cuh with lane b of a group holding body b
// (inertial coordinates, FP64), the planets' pairs exchanged by warp shuffles in ring rounds.
//
// Each planet's lane forms body 0's pull on it in FP64 (`star_pull`); the ring runs over the
// n - 1 planets only, in float pairs; body 0's lane takes the sum of the planets' pulls
// (pairs: its own motion has the planets' mass ratio).  Every unordered pair is evaluated
// once per evaluation.  A step of level 2 is one evaluation at the predicted state and FP32
// differences after the corrector's passes, as in spl_hermite_delta_step; in bins below
// kCarryMinSystems the new state is then evaluated afresh, so that a step follows from the
// stored state alone (as does the choice of the kind of step): a call in chunks or from a
// checkpoint repeats the uninterrupted one bit for bit.
//
// Bound: issue slots and the latency of their chains (n = 15: 7200 instructions and 41 FP64
// ones per step of two systems, 0.52 issued per cycle and sub-partition, the FP64 pipe 18 %
// busy), so three CTAs per SM (168 registers).  Per step of 5041 systems, wholly in FP64 ->
// now: n = 3 6.5 -> 4.7 us, 5 20.7 -> 6.5, 8 52.3 -> 9.6, 11 89.4 -> 22.4, 15 120.8 -> 29.8
// (packed over the CTA for n = 7, 11, 15 before); 65536 systems of 3..15 bodies over 100
// steps: 69.2 -> 16.6 ms.  Steps of 0.02 orbits (level 0), 200 of them: 38400 x 8 52.3 -> 55.2 ms,
// 300 x 8 3.82 -> 4.00.  2048 systems of 16..32 bodies (one per warp, n a run-time value) over 50
// steps: 13.6 -> 2.65 ms.
#pragma once
#include "hermite_ff.cuh"
#include "hermite_wide.cuh"

namespace swarm {

// Bins of at least this many systems carry the evaluation of a level-2 step over to the next
// one (one evaluation and two FP32 differences per step); smaller ones evaluate every new
// state afresh (two and one), so that their steps follow from the stored state alone.  The
// line is where a bin comes near one system per SM sub-partition (608): below it a call is
// short, and interactive users compare resumed runs.  Above it the carried evaluation is worth
// more than repeated bits: 65536 systems of 3..15 bodies over 100 steps 16.6 ms, 23.4 without,
// 1024 x 3 over 400 steps 1.87 and 2.28, at the same error against 64 bits.
constexpr int kCarryMinSystems = 512;

__device__ __forceinline__ ff shfl_ff(const ff &a, int src) {
  return ff_make(__shfl_sync(0xffffffffu, a.h, src), __shfl_sync(0xffffffffu, a.l, src));
}

// A body's place in its group, and its masses.  N = 0: a group is the warp, of n bodies (16..32,
// a run-time value).
template <int N>
struct BplBody {
  int b, base, nn;
  double m0;   // body 0's mass
  ff m0f, mf;  // and this body's, as pairs
  float mt;    // what mf leaves of it: in body 0's own acceleration its mass is no small weight, and
               // left out (as would the product of the lower parts, of one sign for truncated
               // pairs) it would be the same relative error at every step
  __device__ __forceinline__ int n() const { return N ? N : nn; }
  __device__ __forceinline__ unsigned mask() const { return n() == 32 ? 0xffffffffu : ((1u << n()) - 1u) << base; }
  // the ring over the n - 1 planets: RF rounds with reaction, and for an even number a last one in
  // which both lanes of a pair take their own share (RT in all)
  __device__ __forceinline__ int RF() const { return (n() - 2) / 2; }
  __device__ __forceinline__ int RT() const { return (n() - 1) / 2; }
  __device__ __forceinline__ int next(int r) const {  // lane r planets after b's
    int p = (b > 0 ? b - 1 : 0) + r;
    if (p >= n() - 1) p -= n() - 1;
    return base + 1 + p;
  }
  __device__ __forceinline__ int prev(int r) const {
    int p = (b > 0 ? b - 1 : 0) - r;
    if (p < 0) p += n() - 1;
    return base + 1 + p;
  }
};
template <int N>
constexpr int kRoundsA = N ? (N > 2 ? (N - 1) / 2 : 1) : kWideRounds;  // sizes of per-round arrays
template <int N>
constexpr int kRingUnroll = N && (N - 1) / 2 <= 2 ? kRoundsA<N> : 1;

// sum over a group's lanes, valid in its first lane
template <int N>
__device__ __forceinline__ ff grp_sum_ff(const BplBody<N> &g, ff t) {
#pragma unroll
  for (int off = 1; off < (N ? N : 32); off <<= 1) {
    ff o = ff_make(__shfl_down_sync(0xffffffffu, t.h, off), __shfl_down_sync(0xffffffffu, t.l, off));
    if (g.b + off >= g.n()) o = ff_make(0.0f, 0.0f);
    t = ff_add_raw(t, o);
  }
  return ff_norm(t);
}

// the same over the planets' lanes alone, whatever body 0's holds: the first level takes two
// lanes at once, so that n - 1 values need no level more than their number does
template <int N>
__device__ __forceinline__ ff grp_planets_ff(const BplBody<N> &g, ff t) {
  const unsigned FULL = 0xffffffffu;
  ff a = ff_make(__shfl_down_sync(FULL, t.h, 1), __shfl_down_sync(FULL, t.l, 1));
  if (N == 2) return a;
  if (g.b + 1 >= g.n()) a = ff_make(0.0f, 0.0f);
  ff o = ff_make(__shfl_down_sync(FULL, t.h, 2), __shfl_down_sync(FULL, t.l, 2));
  if (g.b + 2 >= g.n()) o = ff_make(0.0f, 0.0f);
  t = ff_add_raw(a, o);
#pragma unroll
  for (int off = 2; off < (N ? N : 32) - 1; off <<= 1) {
    o = ff_make(__shfl_down_sync(FULL, t.h, off), __shfl_down_sync(FULL, t.l, off));
    if (g.b + off >= g.n()) o = ff_make(0.0f, 0.0f);
    t = ff_add_raw(t, o);
  }
  return ff_norm(t);
}
template <int N>
__device__ __forceinline__ float grp_planets32(const BplBody<N> &g, float t) {
  const unsigned FULL = 0xffffffffu;
  const float a = __shfl_down_sync(FULL, t, 1), c = __shfl_down_sync(FULL, t, 2);
  t = (g.b + 1 < g.n() ? a : 0.0f) + (g.b + 2 < g.n() ? c : 0.0f);
#pragma unroll
  for (int off = 2; off < (N ? N : 32) - 1; off <<= 1) {
    const float o = __shfl_down_sync(FULL, t, off);
    t += g.b + off < g.n() ? o : 0.0f;
  }
  return t;
}

// an evaluation: acceleration -M dX + P (M, dX FP64; M = 0 on body 0's lane), jerk J, distances
// and what the guard wants
template <int N>
struct BplEval {
  double M, dX[3];
  ff P[3], J[3];
  float q2, e1, S, V2;
  bool range, near;
  float X[3], V[3], s, p, c;  // relative to body 0, for `bpl_delta`
};
// FULL: body 0's pull in FP64 from x, the perturbers' jerks in pairs; else everything from the
// pairs xf, those jerks in FP32.  STATE: the guard's terms too, and whether a pair is near the
// close-encounter limit of `kcf` (indexed by round).  With more than two rounds they are a loop,
// since the kernel's loop has to fit the instruction cache (n = 15, three evaluations per
// step, 5041 systems: 69 us a step unrolled, 45 as a loop).
template <int N, bool FULL, bool STATE>
__device__ __forceinline__ void bpl_eval_ff(const F64k &k, const BplBody<N> &g, const double (&x)[3], const ff (&xf)[3],
                                            const ff (&v)[3], const float *kcf, BplEval<N> &R) {
  constexpr int KS = N ? 1 : 32;  // stride of kcf
  ff X[3], V[3], rho3, rho2, w[3], T[3], Z[3];
  const bool star = g.b == 0;
#pragma unroll
  for (int c = 0; c < 3; c++) V[c] = ff_sub(v[c], shfl_ff(v[c], g.base));
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
    const ff q2 = ff_norm2(X);
    ff_rho3(q2, rho3, rho2);
  }
  R.c = fjerk_dir(X, V, rho2, w);
  R.s = rho3.h;
  R.p = rho2.h;
#pragma unroll
  for (int c = 0; c < 3; c++) {
    T[c] = ff_mul_raw(rho3, X[c]);
    Z[c] = ff_mul_raw(rho3, w[c]);
    R.X[c] = X[c].h;
    R.V[c] = V[c].h;
  }
  ff Q[3];
#pragma unroll
  for (int c = 0; c < 3; c++) R.P[c] = Q[c] = ff_make(0.0f, 0.0f);
  if (STATE) {
    R.near = false;
    R.e1 = (g.m0f.h + g.mf.h) * rho3.h;  // of the relative orbit: body 0 need not be the heavy one
    R.V2 = __fmaf_rn(V[2].h, V[2].h, __fmaf_rn(V[1].h, V[1].h, __fmul_rn(V[0].h, V[0].h)));
    R.range = frange(R.q2) && R.V2 < 0x1p80f;
    R.S = 0.0f;
  }
#pragma unroll kRingUnroll<N>
  for (int r = 1; r <= g.RT(); r++) {
    const int p = g.next(r), q = g.prev(r);
    ff dx[3], u[3], z[3], s3, s2;
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
    if (FULL) {
      ff dv[3], dw[3];
#pragma unroll
      for (int c = 0; c < 3; c++) dv[c] = ff_sub_raw(shfl_ff(V[c], p), V[c]);
      fjerk_dir(dx, dv, s2, dw);
#pragma unroll
      for (int c = 0; c < 3; c++) {
        z[c] = ff_mul_raw(s3, dw[c]);
        Q[c] = ff_fma_raw(mp, z[c], Q[c]);
      }
    } else {
      ff dv[3];
      float dw[3];
#pragma unroll
      for (int c = 0; c < 3; c++) dv[c] = ff_make(__fsub_rn(__shfl_sync(0xffffffffu, V[c].h, p), V[c].h), 0.0f);
      fjerk_dir32(dx, dv, s2.h, dw);
#pragma unroll
      for (int c = 0; c < 3; c++) {
        z[c].h = __fmul_rn(s3.h, dw[c]);
        Q[c].h = __fmaf_rn(mp.h, z[c].h, Q[c].h);
      }
    }
    float sg = 0.0f;
    if (STATE) {  // |X_b| + |X_p| <= sqrt(2 (q2_b + q2_p))
      const float t = R.q2 + __shfl_sync(0xffffffffu, R.q2, p);
      sg = s3.h * (1.41422f * t) * rsqrtf(t);
      R.S = __fmaf_rn(mp.h, sg, R.S);
      R.near |= !(r2.h >= kcf[(r - 1) * KS] * t);
      R.range = R.range && frange(r2.h);
    }
    if (r <= g.RF()) {  // the pair that lane q evaluated with this one
      const ff mq = ff_neg(shfl_ff(g.mf, q));
#pragma unroll
      for (int c = 0; c < 3; c++) {
        R.P[c] = ff_fma_raw(mq, shfl_ff(u[c], q), R.P[c]);
        if (FULL) Q[c] = ff_fma_raw(mq, shfl_ff(z[c], q), Q[c]);
        else Q[c].h = __fmaf_rn(mq.h, __shfl_sync(0xffffffffu, z[c].h, q), Q[c].h);
      }
      if (STATE) R.S = __fmaf_rn(-mq.h, __shfl_sync(0xffffffffu, sg, q), R.S);
    }
  }
#pragma unroll
  for (int c = 0; c < 3; c++) {
    const ff Tn = ff_norm(T[c]);  // (raw lower parts are of one sign, and so is then their rounding)
    ff w = ff_mul_raw(g.mf, Tn);
    w = fast_two_sum(w.h, __fmaf_rn(g.mf.l, Tn.l, __fmaf_rn(g.mt, Tn.h, w.l)));
    const ff sa = grp_planets_ff<N>(g, w), sj = grp_planets_ff<N>(g, ff_mul_raw(g.mf, Z[c]));
    const ff a = FULL ? ff_norm(R.P[c]) : ff_fma(ff_neg(g.m0f), T[c], R.P[c]);
    const ff j = ff_fma(ff_neg(g.m0f), Z[c], Q[c]);
    R.P[c] = ff_sel(star, sa, a);
    R.J[c] = ff_sel(star, sj, j);
  }
}
// The group's level (the least of its planets') for steps of length hf.  Body 0's answer to a
// planet is formed in pairs by its own lane (2^-46 of it: `BplBody::mt` and `star_pull` keep it
// from the biases that the other sums may have), and may weigh up to 3/64 of the relative velocity
// in a step (at level 2 it cannot weigh that much).  Only with a body 0 much lighter than its companion does it weigh more, at 130 steps
// an orbit and fewer (masses 0.03 and 1, 102 steps an orbit: 1.3 to 1.5 times the FP64 steps'
// error without this limit; two equal ones 0.8).
template <int N>
__device__ __forceinline__ int bpl_level(const BplBody<N> &g, const BplEval<N> &R, float hf, bool ok) {
  int lv = 2;
  if (g.b != 0) lv = R.range ? fguard(hf, hf * hf * R.e1, R.S, R.V2) : 0;
  if (!ok) lv = 0;
  const unsigned gm = g.mask();
  unsigned n0 = __ballot_sync(0xffffffffu, lv == 0);
  const unsigned n1 = __ballot_sync(0xffffffffu, lv == 1);
  if (n1) {
    const float w0 = hf * g.mf.h * R.p;
    n0 |= __ballot_sync(0xffffffffu, lv == 1 && !(w0 * w0 <= 0x1.2p-9f * R.V2));
  }
  return n0 & gm ? 0 : n1 & gm ? 1 : 2;
}

// change of the evaluation R when the bodies' positions and velocities move by dX, dV, in FP32
// (see spl_delta); the pairs' geometry is formed again from R's FP32 vectors
template <int N>
__device__ __forceinline__ void bpl_delta(const BplBody<N> &g, const BplEval<N> &R, const float (&dX)[3],
                                          const float (&dV)[3], float (&DA)[3], float (&DJ)[3]) {
  const unsigned FULL = 0xffffffffu;
  const bool star = g.b == 0;
  float d[3], e[3], T[3], Z[3], P[3], Q[3];
#pragma unroll
  for (int c = 0; c < 3; c++) {
    d[c] = dX[c] - __shfl_sync(FULL, dX[c], g.base);
    e[c] = dV[c] - __shfl_sync(FULL, dV[c], g.base);
    P[c] = Q[c] = 0.0f;
  }
  fpair_delta(R.X, R.V, d, e, R.s, R.p, R.c, T, Z);
#pragma unroll kRingUnroll<N>
  for (int r = 1; r <= g.RT(); r++) {
    const int p = g.next(r), q = g.prev(r);
    float x[3], u[3], dd[3], ee[3], t[3], z[3];
    const float mp = __shfl_sync(FULL, g.mf.h, p);
#pragma unroll
    for (int c = 0; c < 3; c++) {
      x[c] = __shfl_sync(FULL, R.X[c], p) - R.X[c];
      u[c] = __shfl_sync(FULL, R.V[c], p) - R.V[c];
      dd[c] = __shfl_sync(FULL, d[c], p) - d[c];
      ee[c] = __shfl_sync(FULL, e[c], p) - e[c];
    }
    const float y = rsqrtf(__fmaf_rn(x[2], x[2], __fmaf_rn(x[1], x[1], x[0] * x[0])));
    const float y2 = y * y;
    const float rv = __fmaf_rn(x[2], u[2], __fmaf_rn(x[1], u[1], x[0] * u[0]));
    fpair_delta(x, u, dd, ee, y2 * y, y2, -3.0f * rv * y2, t, z);
#pragma unroll
    for (int c = 0; c < 3; c++) {
      P[c] = __fmaf_rn(mp, t[c], P[c]);
      Q[c] = __fmaf_rn(mp, z[c], Q[c]);
    }
    if (r <= g.RF()) {
      const float mq = -__shfl_sync(FULL, g.mf.h, q);
#pragma unroll
      for (int c = 0; c < 3; c++) {
        P[c] = __fmaf_rn(mq, __shfl_sync(FULL, t[c], q), P[c]);
        Q[c] = __fmaf_rn(mq, __shfl_sync(FULL, z[c], q), Q[c]);
      }
    }
  }
#pragma unroll
  for (int c = 0; c < 3; c++) {
    const float sa = grp_planets32<N>(g, __fmul_rn(g.mf.h, T[c]));
    const float sj = grp_planets32<N>(g, __fmul_rn(g.mf.h, Z[c]));
    DA[c] = star ? sa : __fmaf_rn(-g.m0f.h, T[c], P[c]);
    DJ[c] = star ? sj : __fmaf_rn(-g.m0f.h, Z[c], Q[c]);
  }
}

// The new (x, v) of a step of C from a state of level 1 (or 2); out of line.
template <int N>
static __device__ __noinline__ void bpl_hermite_ff_advance(const F64k &k, const BplBody<N> &g, const FCoef &C, int n_corr,
                                                    double (&xs)[3], double (&vs)[3], const double (&a0)[3],
                                                    const float (&da)[3], const ff (&j0)[3]) {
  ff V[3], G[3], W[3], af[3], U[3];
  double xp[3], x[3], v[3];
  BplEval<N> R;
#pragma unroll
  for (int c = 0; c < 3; c++) {
    v[c] = vs[c];
    V[c] = ff_from(v[c]);
    af[c] = ff_from(a0[c]);
    af[c] = ff_norm(ff_make(af[c].h, af[c].l + da[c]));
    x[c] = fma(C.h, v[c], xs[c]);
    fpredict(C, af[c], j0[c], G[c], W[c]);
  }
  for (int ic = 1; ic < n_corr; ic++) {
    ff X[3];
#pragma unroll
    for (int c = 0; c < 3; c++) {
      X[c] = ff_add(ff_from(x[c]), G[c]);
      U[c] = ff_add(V[c], W[c]);
    }
    bpl_eval_ff<N, false, false>(k, g, x, X, U, nullptr, R);
#pragma unroll
    for (int c = 0; c < 3; c++)
      fcorrect(C, af[c], ff_sub(R.P[c], af[c]), ff_sub(j0[c], R.J[c]), G[c], W[c], U[c]);
  }
#pragma unroll
  for (int c = 0; c < 3; c++) {
    xp[c] = ff_addto(x[c], ff_norm(G[c]));
    U[c] = ff_add(V[c], W[c]);
  }
  bpl_eval_ff<N, true, false>(k, g, xp, U, U, nullptr, R);
#pragma unroll
  for (int c = 0; c < 3; c++) {
    ff D = ff_from(fma(-R.M, R.dX[c], -a0[c]));
    D = ff_add(ff_make(D.h, D.l - da[c]), R.P[c]);
    fcorrect(C, af[c], D, ff_sub(j0[c], R.J[c]), G[c], W[c], U[c]);
    xs[c] = ff_addto(x[c], G[c]);
    U[c].l = __fmaf_rn(C.f.h, da[c], U[c].l);
    vs[c] = ff_addto(fma(C.h, a0[c], v[c]), ff_norm(U[c]));
  }
}

// an evaluation of a state, out of line (refills)
template <int N>
static __device__ __noinline__ void bpl_eval_ff_call(const F64k &k, const BplBody<N> &g, const double (&x)[3], const ff (&v)[3],
                                              const float *kcf, BplEval<N> &R) {
  BplEval<N> E;
  bpl_eval_ff<N, true, true>(k, g, x, v, v, kcf, E);
  R = E;
}

// ---------------------------------------------------------------- FP64 steps (guard not met)
// Out of line; every lane of the warp takes part in the shuffles.  kc, d2: per round of the ring
// over all n bodies, in registers' place (local memory) or, for N = 0, this lane's column of
// shared memory.  q2: the lane's squared distance to body 0.
template <int N>
struct BplRounds {
  static constexpr int RT = Ring<N>::RT > 0 ? Ring<N>::RT : 1;
  double kc[RT], d2[RT], q2;
  __device__ __forceinline__ double &kcr(int r) { return kc[r - 1]; }
  __device__ __forceinline__ double &d2r(int r) { return d2[r - 1]; }
};
template <>
struct BplRounds<0> {
  double *kc, *d2, q2;
  __device__ __forceinline__ double &kcr(int r) { return kc[(r - 1) * 32]; }
  __device__ __forceinline__ double &d2r(int r) { return d2[(r - 1) * 32]; }
};
template <int N>
static __device__ __noinline__ void bpl_fp64_eval(const F64k &k, const double (&x)[3], const double (&v)[3], double m,
                                                  const BplBody<N> &g, double (&a)[3], double (&j)[3], BplRounds<N> &rd) {
  double a_[3], j_[3], q_;
  if constexpr (N == 0) {
    wring_accjerk<true, 1>(k, x, v, m, g.b, wide_ring(g.nn), a_, j_, q_, rd.d2, 0);
  } else {
    ring_accjerk<N, true, 1>(k, x, v, m, g.b, g.base, a_, j_, q_, rd.d2);
  }
#pragma unroll
  for (int c = 0; c < 3; c++) {
    a[c] = a_[c];
    j[c] = j_[c];
  }
  rd.q2 = q_;
}
// Eq. 5's length in FP64 from a and j (every lane of the warp)
template <int N>
__device__ __forceinline__ double bpl_fp64_eq5(const StepParams &P, const BplBody<N> &g, bool lane_ok, const double (&a)[3],
                                               const double (&j)[3]) {
  const double ratio = (j[0] * j[0] + j[1] * j[1] + j[2] * j[2]) / (a[0] * a[0] + a[1] * a[1] + a[2] * a[2]);
  double ssum;
  if constexpr (N == 0) ssum = warp_sum(lane_ok ? ratio : 0.0);
  else ssum = grp_sum<N>(ratio, g.b, g.base);
  return fabs(P.dt) * rsqrt(ssum);
}
// the monitor's tests at a state evaluated into rd (every lane of the warp)
template <int N>
__device__ __forceinline__ void bpl_fp64_monitor(const StepParams &P, const BplBody<N> &g, const double (&x)[3],
                                                 const double (&v)[3], BplRounds<N> &rd, bool &nf, bool &ej, bool &ce) {
  const double q2 = rd.q2;
  nf = nonfinite(x[0]) | nonfinite(x[1]) | nonfinite(x[2]) | nonfinite(v[0]) | nonfinite(v[1]) | nonfinite(v[2]);
  ej = g.b != 0 && P.eject2 > 0.0 && q2 > P.eject2;
  ce = false;
  const int n = g.n();
  for (int r = 1; r <= n / 2; r++) {
    int p = g.b + r;
    if (p >= n) p -= n;
    const double q2p = shfl(q2, g.base + p);
    const double kc = rd.kcr(r);
    if (kc > 0.0 && close_encounter(P.fk, rd.d2r(r), kc, q2, q2p)) ce = true;
  }
}
// Up to `count` steps in FP64 for the warp's groups of level 0 (`mine`), each from its state's a and j:
// steps of hs, or (ADAPT) that one and then Eq. 5's.  Returns the steps taken, the same for every
// group: before the count is full it ends at a state that a group has to look at, that the
// monitor stops, or that needs no further step.  x, v, a, j and rd are then that state's, hs, ts and
// last those of the step that led there.  clear: the state is
// beyond doubt one for FP64, since a step is too long for the pairs by 1 % (their guard's eta^2
// is good to 2^-20), a distance out of their range, or (free) all of them are.
// In registers from step to step (200 steps of 0.02 orbits, 300 x 8 bodies: 4.5 ms with the evaluation and
// the rest of the step out of line each, 4.0 so, 3.8 in a kernel wholly in FP64).
template <int N, bool ADAPT>
static __device__ __noinline__ int bpl_fp64_run(const StepParams &P, const BplBody<N> &g, bool lane_ok, double m, bool mine,
                                                bool free, int count, BplRounds<N> &rd, double (&xs)[3], double (&vs)[3],
                                                double (&as)[3], double (&js)[3], double &hs, double &ts, double te,
                                                bool &last, bool &clear) {
  const F64k &k = P.fk;
  const unsigned FULL = 0xffffffffu, gm = g.mask();
  const bool printed = P.corr_form != 0;
  const double dir = P.dt > 0 ? 1.0 : -1.0;
  double x[3], v[3], a0[3], j0[3], h = hs, t = ts;
#pragma unroll
  for (int c = 0; c < 3; c++) {
    x[c] = xs[c];
    v[c] = vs[c];
    a0[c] = as[c];
    j0[c] = js[c];
  }
  HCoef C = hcoef(h);
  int s = 0;
  bool cl = false, la = last;
  double hn = 0.0;
  for (;;) {
    double xk[3], vk[3], Xb[3], Vb[3], q2 = 0.0;
    // Eq. 3 predictor and the step-invariant parts of the corrector
#pragma unroll
    for (int c = 0; c < 3; c++) {
      xk[c] = fma(j0[c], C.h3_6, fma(a0[c], C.h2_2, fma(v[c], C.h, x[c])));
      vk[c] = fma(j0[c], C.h2_2, fma(a0[c], C.h, v[c]));
      Vb[c] = fma(j0[c], C.h2_12, fma(a0[c], C.hh, v[c]));
    }
    PCoef PC;
    if (printed) {
      PC = pcoef(h);
#pragma unroll
      for (int c = 0; c < 3; c++) Xb[c] = fma(j0[c], PC.pj, fma(a0[c], PC.pa, xk[c]));
    } else {
#pragma unroll
      for (int c = 0; c < 3; c++) Xb[c] = fma(a0[c], C.h2_12, fma(v[c], C.hh, x[c]));
    }
#pragma unroll 1
    for (int ic = 0;; ic++) {
      if constexpr (N == 0) {
        wring_accjerk<true, 1>(k, xk, vk, m, g.b, wide_ring(g.nn), a0, j0, q2, rd.d2, 0);
      } else {
        ring_accjerk<N, true, (N <= 8 ? Ring<N>::RF : 1)>(k, xk, vk, m, g.b, g.base, a0, j0, q2, rd.d2);
      }
      if (ic == P.n_corr) break;
#pragma unroll
      for (int c = 0; c < 3; c++) vk[c] = fma(-C.h2_12, j0[c], fma(C.hh, a0[c], Vb[c]));
      if (printed) {
#pragma unroll
        for (int c = 0; c < 3; c++) xk[c] = fma(PC.cj, j0[c], fma(PC.ca, a0[c], Xb[c]));
      } else {
#pragma unroll
        for (int c = 0; c < 3; c++) xk[c] = fma(-C.h2_12, a0[c], fma(C.hh, vk[c], Xb[c]));
      }
    }
#pragma unroll
    for (int c = 0; c < 3; c++) {
      x[c] = xk[c];
      v[c] = vk[c];
    }
    rd.q2 = q2;
    s++;
    float hf = P.fc.hf;
    if (ADAPT) {
      hn = bpl_fp64_eq5<N>(P, g, lane_ok, a0, j0);
      hf = f_from(hn);
    }
    const float q = f_from(q2), y = rsqrtf(q);
    const bool far = hf * hf * (g.m0f.h + g.mf.h) * y * y * y > 1.01f * kFFEta2 || q > 0x1.04p40f || q < 0x1.f8p-41f;
    const unsigned fars = __ballot_sync(FULL, g.b != 0 && far);  // (every lane: not behind `free`)
    cl = free || (fars & gm) != 0;
    if (s >= count) break;
    bool nf, ej, ce;
    bpl_fp64_monitor<N>(P, g, x, v, rd, nf, ej, ce);
    bool stop = nf || ej || ce || !cl;
    double tn = t, hx = h;
    bool ln = la;
    if (ADAPT) {
      tn = kadd(k, t, h);
      const double rem = kmul(k, ksub(k, te, tn), dir);
      ln = hn >= rem;
      hx = kmul(k, ln ? rem : hn, dir);
      stop = stop || la || !(hn > 0.0) || nonfinite(hn);
    }
    if (__any_sync(FULL, mine && stop)) break;
    if (ADAPT) {
      t = tn;
      h = hx;
      la = ln;
      C = hcoef(h);
    }
  }
#pragma unroll
  for (int c = 0; c < 3; c++) {
    xs[c] = x[c];
    vs[c] = v[c];
    as[c] = a0[c];
    js[c] = j0[c];
  }
  hs = h;
  ts = t;
  last = la;
  clear = cl;
  return s;
}

// ---------------------------------------------------------------- the integration loop
// Work handed out per system: each of the warp's G groups takes its next system as soon as its
// own one reached its end time or stopped (fixed steps: stops and per-system end times;
// adaptive steps: step counts differ from system to system).  take(need): the group's next
// system, or -1 (every lane calls it).  A refill round loads the new systems and evaluates
// them (the other groups re-evaluate their unchanged state and keep what they have).
// OBS (fixed steps): through the observation times P.t_obs in one launch, leaving the radial
// velocity at each (12 observations 12 steps apart, 257 x 3 systems: 1.14 ms with a launch for
// each, whose cold start costs as much as three steps, 0.85 in one).
template <int N, bool ADAPT, bool OBS, class Take>
__device__ __forceinline__ void bpl_hermite_run(const BinView &B, const StepParams &P, BplRounds<N> &rd, float *kcf,
                                                Take take) {
  constexpr int KS = N ? 1 : 32;
  const bool printed = P.corr_form != 0;  // warp-uniform
  const bool carry = B.S >= kCarryMinSystems;
  BplBody<N> g;
  g.nn = B.n;
  const int n = g.n(), G = N ? 32 / n : 1;
  const int rt = n / 2;  // rounds of the ring over all n bodies
  const unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  int grp = lane / n;
  g.b = lane - grp * n;
  const bool lane_ok = grp < G;
  if (!lane_ok) {  // spare lanes mirror group 0 (same broadcasts, same state)
    grp = 0;
    g.b = lane - G * n;
  }
  g.base = grp * n;
  const int b = g.b;
  const int SP = B.S_pad;
  const unsigned gm = g.mask();
  const double dir = P.dt > 0 ? 1.0 : -1.0;
  const int cap = P.max_steps > 0 ? P.max_steps : kAdaptiveStepCap;
  const ff tau = ff_from(fabs(P.dt));
  const float ejf = P.eject2 > 0.0 ? 0.998f * (float)P.eject2 : __int_as_float(0x7f800000);

  int s = 0, steps = 0, level = 0;
  // fit: scaled, and the state the group began with, or its last FP64 step led to, is one that the
  // pairs can hold (`spl_ff_state` says why the other steps keep it one)
  bool has = false, exhausted = false, scaled = false, fit = false;
  // the state's acceleration is a0 + da; j0: FP64, or (level > 0) the bits of a pair
  double x[3] = {0.0, 0.0, 0.0}, v[3] = {0.0, 0.0, 0.0}, m = 1.0, a0[3] = {0.0, 0.0, 0.0}, j0[3] = {0.0, 0.0, 0.0};
  float da[3] = {0.0f, 0.0f, 0.0f};
  // rd.kc: close-encounter coefficients of the FP64 ring; kcf: the planets' ring's, doubled and
  // rounded up
  LaunchPlan plan;
  plan.N = 0;
  plan.full = 1;
  plan.exact = 1;
  plan.h_last = P.dt;
  plan.t_end = P.t_end;
  double t = 0.0, t0 = 0.0, te = 0.0;  // fixed steps: t is formed from t0 when needed
  ff h = ff_make(0.0f, 0.0f);          // ADAPT: length of the next step of a group in pairs
  g.m0 = 1.0;
  g.m0f = g.mf = ff_make(1.0f, 0.0f);
  g.mt = 0.0f;
  for (int r = 1; r <= rt; r++) rd.kcr(r) = 0.0;
  for (int r = 1; r <= g.RT(); r++) kcf[(r - 1) * KS] = 0.0f;
  auto to_bits = [](const ff &f) { return __hiloint2double(__float_as_int(f.h), __float_as_int(f.l)); };
  auto to_pair = [](double d) { return ff_make(__int_as_float(__double2hiint(d)), __int_as_float(__double2loint(d))); };

  // Eq. 5's step from the acceleration an + dn and the jerk J
  auto eq5 = [&](const double (&an)[3], const float (&dn)[3], const ff (&J)[3]) -> ff {
    ff A[3];
#pragma unroll
    for (int c = 0; c < 3; c++) {
      A[c] = ff_from(an[c]);
      A[c] = ff_norm(ff_make(A[c].h, A[c].l + dn[c]));
    }
    const ff sum = shfl_ff(grp_sum_ff<N>(g, ff_eq5_term(A, J)), g.base);
    return ff_mul(tau, ff_rsqrt(sum));
  };

  // the observations [from, to) at the present state, and the plan from t0 on towards the first
  // of the others that lies ahead (those that do not are made here); plan.N = 0: none is left
  int obs = 0;
  auto next_obs = [&](int from, int to) {
    for (obs = from;; obs++) {
      if (obs >= to) {
        if (obs >= P.n_obs) {
          plan.N = 0;
          return;
        }
        plan = launch_plan_to(P, P.t_obs[obs], t0, true);
        if (plan.N > 0) return;
      }
      if (lane_ok && b == 0)
        P.rv[obs * P.rv_stride + B.gidx[s]] = v[0] * P.los[0] + v[1] * P.los[1] + v[2] * P.los[2];
    }
  };

  for (;;) {
    // ---- refill: groups without a system take their next one
    const bool need = !has && !exhausted;
    if (__any_sync(FULL, need)) {
      const int ss = take(need, lane_ok && b == 0, g.base);
      const bool got = need && ss >= 0;
      if (need && ss < 0) exhausted = true;
      if (got) {
        s = ss;
#pragma unroll
        for (int c = 0; c < 3; c++) {
          x[c] = B.x[(size_t)(c * n + b) * SP + s];
          v[c] = B.v[(size_t)(c * n + b) * SP + s];
        }
        m = B.m[(size_t)b * SP + s];
      }
      const double m0 = shfl(m, g.base);
      const bool sc = (__ballot_sync(FULL, !fmass_ok(m, b == 0)) & gm) == 0 && fscale(P.dt, -60, 40);
      for (int r = 1; r <= rt; r++) {
        int p = b + r;
        if (p >= n) p -= n;
        const double mp = shfl(m, g.base + p);
        const double kk = (b != 0 && p != 0) ? hill_kc(P.ce_factor, m, mp, m0) : 0.0;
        if (got) rd.kcr(r) = kk;
      }
      for (int r = 1; r <= g.RT(); r++) {
        const double mp = shfl(m, g.next(r));
        const float kk = 2.004f * (float)hill_kc(P.ce_factor, m, mp, m0);
        if (got) kcf[(r - 1) * KS] = kk;
      }
      if (got) {
        scaled = sc;
        g.m0 = m0;
        g.m0f = ff_from(m0);
        g.mf = ff_norm(ff_from(m));
        g.mt = (float)((m - (double)g.mf.h) - (double)g.mf.l);
      }
      const bool tm = (__ballot_sync(FULL, !ff_tame(x, v)) & gm) == 0;
      if (got) fit = scaled && tm;
      double an[3] = {0.0, 0.0, 0.0}, jn[3] = {0.0, 0.0, 0.0};
      ff hn = h;
      int lv = 0;
      if (!printed) {
        BplEval<N> E;
        ff V[3];
#pragma unroll
        for (int c = 0; c < 3; c++) V[c] = ff_norm(ff_from(v[c]));
        bpl_eval_ff_call<N>(P.fk, g, x, V, kcf, E);
#pragma unroll
        for (int c = 0; c < 3; c++) {
          an[c] = fma(-E.M, E.dX[c], ff_double(E.P[c]));
          jn[c] = to_bits(E.J[c]);
        }
        float hf = P.fc.hf, zero[3] = {0.0f, 0.0f, 0.0f};
        if (ADAPT) {
          hn = eq5(an, zero, E.J);
          hf = hn.h;
        }
        lv = bpl_level<N>(g, E, hf, fit && hf > 0.0f);
      }
      if (__any_sync(FULL, got && !lv)) {
        double a_[3], j_[3];
        bpl_fp64_eval<N>(P.fk, x, v, m, g, a_, j_, rd);
        if (!lv)
#pragma unroll
          for (int c = 0; c < 3; c++) {
            an[c] = a_[c];
            jn[c] = j_[c];
          }
      }
      if (got) {
#pragma unroll
        for (int c = 0; c < 3; c++) {
          a0[c] = an[c];
          j0[c] = jn[c];
          da[c] = 0.0f;
        }
        level = lv;
        h = hn;
        t0 = t = B.t[s];
        steps = 0;
        const bool runnable = B.status[s] <= SWARM_SYS_DONE;
        if (!ADAPT) {
          if constexpr (OBS) next_obs(0, runnable ? 0 : P.n_obs);
          else plan = launch_plan(B, P, s, t0, runnable);
          has = runnable && plan.N > 0;
        } else {
          te = adaptive_end(B, P, s);
          has = runnable && ((te - t0) * dir > 1e-12 * fmax(1.0, fabs(te)));
        }
        if (runnable && !has && lane_ok && b == 0) B.status[s] = SWARM_SYS_DONE;
      }
      continue;
    }
    if (!__any_sync(FULL, has)) break;

    // ---- one step for every group holding a system
    const bool alive = has;
    bool last, bad = false;
    double hd = P.dt;
    int kind = level;  // of this step
    if (!ADAPT) {
      last = steps + 1 == plan.N;
      if (last && !plan.exact) {  // the shortened last step is FP64
        hd = plan.h_last;
        if (kind)
#pragma unroll
          for (int c = 0; c < 3; c++) {
            j0[c] = ff_double(to_pair(j0[c]));
            a0[c] += (double)da[c];
          }
        kind = 0;
      }
    } else {
      double hs = ff_double(h);
      if (__any_sync(FULL, alive && !kind)) {
        const double e = bpl_fp64_eq5<N>(P, g, lane_ok, a0, j0);
        if (!kind) hs = e;
      }
      const double rem = kmul(P.fk, ksub(P.fk, te, t), dir);
      last = hs >= rem;
      bad = !(hs > 0.0) || nonfinite(hs);
      hd = kmul(P.fk, last ? rem : hs, dir);
    }
    const bool active = alive && !bad;
    FCoef Cad;
    if (ADAPT) Cad = fcoef(hd);
    const FCoef &C = ADAPT ? Cad : P.fc;
    const bool any2 = __any_sync(FULL, active && kind == 2);
    const bool rest = __any_sync(FULL, active && kind != 2);
    double an[3], jn[3];
    float dn[3] = {0.0f, 0.0f, 0.0f};
    bool fp64 = false, clear = false;
    if (rest) {  // groups of level 1, groups in FP64
      double xn[3], vn[3];
      const bool any1 = __any_sync(FULL, active && kind == 1);
      if (any1) {
        ff jf[3];
#pragma unroll
        for (int c = 0; c < 3; c++) {
          xn[c] = x[c];
          vn[c] = v[c];
          jf[c] = to_pair(j0[c]);
        }
        bpl_hermite_ff_advance<N>(P.fk, g, C, P.n_corr, xn, vn, a0, da, jf);
        if (active && kind == 1)
#pragma unroll
          for (int c = 0; c < 3; c++) {
            x[c] = xn[c];
            v[c] = vn[c];
          }
      }
      if (__any_sync(FULL, active && kind == 0)) {  // several steps where no group of the warp is in pairs
        const bool alone = !any1 && !any2;
        int count = 1;
        if (alone) {
          int c = 1 << 30;
          if (active) {
            c = ADAPT ? cap - steps : max(1, (plan.exact ? plan.N : plan.N - 1) - steps);
            if (P.log_interval > 0) c = min(c, P.log_interval - steps % P.log_interval);
          }
          count = __reduce_min_sync(FULL, c);
        }
        double a_[3], j_[3], hx = hd, tx = t;
        bool lx = last, cl;
#pragma unroll
        for (int c = 0; c < 3; c++) {
          xn[c] = x[c];
          vn[c] = v[c];
          a_[c] = a0[c];
          j_[c] = j0[c];
        }
        const int done = bpl_fp64_run<N, ADAPT>(P, g, lane_ok, m, active && !kind, printed || !scaled, count, rd, xn, vn, a_, j_,
                                                hx, tx, te, lx, cl);
        fp64 = true;
        const bool tm = (__ballot_sync(FULL, !ff_tame(xn, vn)) & gm) == 0;
        if (active && !kind) {
          fit = scaled && tm;
          clear = cl;
          if (ADAPT) {
            hd = hx;
            t = tx;
            last = lx;
          } else {
            last = steps + done == plan.N;
          }
          steps += done - 1;
#pragma unroll
          for (int c = 0; c < 3; c++) {
            x[c] = xn[c];
            v[c] = vn[c];
            an[c] = a_[c];
            jn[c] = j_[c];
          }
        }
      }
    }
    // Level 2: phase 0 evaluates the prediction and corrects it (spl_hermite_delta_step); then,
    // for every group or (carry) those of the other kinds, phase 1 evaluates the new state.
    // One copy of the evaluation serves both phases (instruction cache).  Neither for a warp none of
    // whose systems the pairs could take or hold, nor for the printed corrector, whose steps are FP64.
    int lv = 0;
    bool near = true;
    ff hn = h;
    int phase = 0;
    if (!any2) phase = !printed && __any_sync(FULL, alive && fit && !clear) ? 1 : 2;
#pragma unroll 1
    for (; phase < (rest || !carry ? 2 : 1); phase++) {
      BplEval<N> E;
      ff G[3], W[3], V[3];
      double xe[3];
#pragma unroll
      for (int c = 0; c < 3; c++) {
        V[c] = ff_norm(ff_from(v[c]));
        xe[c] = x[c];
        if (phase == 0) {
          const ff a = ff_from(a0[c]);
          fpredict(C, ff_norm(ff_make(a.h, a.l + da[c])), to_pair(j0[c]), G[c], W[c]);
          G[c] = ff_norm(ff_add_raw(fstep(C, V[c]), G[c]));
          V[c] = ff_add(V[c], W[c]);
          xe[c] = ff_addto(x[c], G[c]);
        }
      }
      bpl_eval_ff<N, true, true>(P.fk, g, xe, V, V, kcf, E);
      const bool mine = phase == 0 ? (carry && kind == 2) : !(carry && kind == 2);
      float hf = ADAPT ? 1.25f * C.hf : P.fc.hf;
      double aE[3];
#pragma unroll
      for (int c = 0; c < 3; c++) aE[c] = fma(-E.M, E.dX[c], ff_double(E.P[c]));
      if (phase == 1 && ADAPT) {
        const float zero[3] = {0.0f, 0.0f, 0.0f};
        const ff hs = eq5(aE, zero, E.J);
        if (mine) hn = hs;
        hf = hs.h;
      }
      const int lE = bpl_level<N>(g, E, hf, fit && hf > 0.0f);
      if (mine) {
        lv = lE;
        near = !lE || (b != 0 && (E.near || !(E.q2 < ejf)));
      }
      if (phase == 0) {
        ff D[3], F[3];
        float DJ[3] = {0.0f, 0.0f, 0.0f}, dA[3] = {0.0f, 0.0f, 0.0f}, dX[3], dV[3];
#pragma unroll
        for (int c = 0; c < 3; c++) {
          const ff jf = to_pair(j0[c]);
          ff d = ff_from(fma(-E.M, E.dX[c], -a0[c]));
          d = ff_add_raw(ff_make(d.h, d.l - da[c]), E.P[c]);
          D[c] = ff_norm(ff_fma_raw(ff_neg(C.f), jf, d));
          F[c] = ff_norm(ff_sub_raw(E.J[c], jf));
        }
#pragma unroll 1
        for (int ic = 1; ic <= P.n_corr; ic++) {
#pragma unroll
          for (int c = 0; c < 3; c++)
            fcorrect_delta32(C, D[c].h + dA[c], F[c].h + DJ[c], dX[c], dV[c]);
          if (ic == P.n_corr) {
#pragma unroll
            for (int c = 0; c < 3; c++) {
              ff y, u;
              fcorrect_delta(C, ff_make(D[c].h, D[c].l + dA[c]), ff_make(F[c].h, F[c].l + DJ[c]), y, u);
              if (active && kind == 2) {
                x[c] = ff_addto(x[c], ff_add(G[c], y));
                v[c] = ff_addto(v[c], ff_add(W[c], u));
              }
            }
            if (!carry) break;
          }
          bpl_delta<N>(g, E, dX, dV, dA, DJ);
        }
        if (carry && kind == 2) {
          ff J[3];
#pragma unroll
          for (int c = 0; c < 3; c++) {
            an[c] = aE[c];
            dn[c] = dA[c];
            J[c] = ff_norm(ff_make(E.J[c].h, E.J[c].l + DJ[c]));
            jn[c] = to_bits(J[c]);
          }
        }
        if (ADAPT && carry) {
          ff J[3];
#pragma unroll
          for (int c = 0; c < 3; c++) J[c] = ff_norm(ff_make(E.J[c].h, E.J[c].l + DJ[c]));
          const ff hs = eq5(aE, dA, J);
          if (kind == 2) {
            hn = hs;
            if (!(hs.h > 0.0f && hs.h <= hf)) lv = 0;
          }
        }
      } else if (mine && (lE || kind)) {
#pragma unroll
        for (int c = 0; c < 3; c++) {
          an[c] = aE[c];
          jn[c] = to_bits(E.J[c]);
        }
      }
    }
    if (carry && kind == 2 && !lv) near = true;
    int code = 0;
    if (__any_sync(FULL, alive && near)) {  // in FP64: a0, j0 of groups that need them, the exact tests
      if (!fp64 || __any_sync(FULL, alive && near && kind != 0)) {
        double a_[3], j_[3];
        bpl_fp64_eval<N>(P.fk, x, v, m, g, a_, j_, rd);
        if (!lv)
#pragma unroll
          for (int c = 0; c < 3; c++) {
            an[c] = a_[c];
            jn[c] = j_[c];
            dn[c] = 0.0f;
          }
      }
      bool nf, ej, ce;
      bpl_fp64_monitor<N>(P, g, x, v, rd, nf, ej, ce);
      const unsigned bnf = __ballot_sync(FULL, alive && (nf || bad)) & gm;
      const unsigned bej = __ballot_sync(FULL, active && ej) & gm;
      const unsigned bce = __ballot_sync(FULL, active && ce) & gm;
      code = bnf ? SWARM_SYS_NONFINITE : bej ? SWARM_SYS_EJECTED : bce ? SWARM_SYS_CLOSE_ENCOUNTER : 0;
    } else if (__any_sync(FULL, bad && alive)) {
      code = (__ballot_sync(FULL, alive && bad) & gm) ? SWARM_SYS_NONFINITE : 0;
    }
    if (!alive) code = 0;
    if (active) {
#pragma unroll
      for (int c = 0; c < 3; c++) {
        a0[c] = an[c];
        j0[c] = jn[c];
        da[c] = dn[c];
      }
      level = lv;
      h = hn;
      steps++;
      if (ADAPT) t = last ? te : kadd(P.fk, t, hd);
    }
    const bool reached = active && last && !code;
    const bool capped = ADAPT && active && steps >= cap;
    const bool finish = alive && (code != 0 || reached || capped);
    if (!ADAPT && (finish || (P.log_interval > 0 && active && (steps % P.log_interval) == 0)))
      t = step_time(plan, steps, t0, P.dt);
    if (P.log_interval > 0) {
      const bool need_log = active && !code && (steps % P.log_interval) == 0;
      if (__any_sync(FULL, need_log)) {
        double e4[4];
        if constexpr (N == 0) wring_energy(x, v, m, b, lane_ok, wide_ring(n), e4);
        else ring_energy<N>(x, v, m, b, g.base, e4);
        if (need_log && lane_ok && b == 0) write_log(P, B.gidx[s], t, e4);
      }
    }
    bool end = finish;
    if constexpr (OBS) if (finish) {
      const bool count = obs == P.n_obs - 1;  // the counters are the last interval's
      if (b == 0 && lane_ok && P.counters && steps > 0 && count) {
        atomicAdd(&P.counters[0], (unsigned long long)steps);
        const unsigned long long NP = (unsigned long long)n * (n - 1) / 2;
        atomicAdd(&P.counters[1], NP * (1ull + (unsigned long long)steps * (P.n_corr + 1)));
      }
      t0 = t;
      steps = 0;
      next_obs(obs, code ? P.n_obs : obs + 1);
      end = plan.N == 0;
    }
    if (end && lane_ok) {
#pragma unroll
      for (int c = 0; c < 3; c++) {
        B.x[(size_t)(c * n + b) * SP + s] = x[c];
        B.v[(size_t)(c * n + b) * SP + s] = v[c];
      }
      if (b == 0) {
        B.t[s] = t;
        if (code) B.status[s] = code;
        else if (ADAPT) B.status[s] = reached ? SWARM_SYS_DONE : SWARM_SYS_ACTIVE;
        else B.status[s] = plan.full ? SWARM_SYS_DONE : SWARM_SYS_ACTIVE;
        if (P.counters && steps > 0) {
          atomicAdd(&P.counters[0], (unsigned long long)steps);
          const unsigned long long NP = (unsigned long long)n * (n - 1) / 2;
          atomicAdd(&P.counters[1], NP * (1ull + (unsigned long long)steps * (P.n_corr + 1)));
        }
      }
    }
    if (end) has = false;
  }
}
// the bin's next systems, one by one
template <int N, bool ADAPT, bool OBS = false>
__device__ __forceinline__ void bpl_hermite_stream(const BinView &B, const StepParams &P) {
  BplRounds<N> rd;
  float kcf[kRoundsA<N>];
  bpl_hermite_run<N, ADAPT, OBS>(B, P, rd, kcf, [&](bool need, bool leader, int base) {
    int sn = 0;
    if (need && leader) sn = atomicAdd(P.work_next, 1);
    sn = __shfl_sync(0xffffffffu, sn, base);
    return stream_system(B, sn);
  });
}
// one work unit: a warp's G = 32/N systems
template <int N, bool ADAPT>
__device__ __forceinline__ void bpl_hermite_body(const BinView &B, const StepParams &P, int unit) {
  bool taken = false;
  BplRounds<N> rd;
  float kcf[kRoundsA<N>];
  bpl_hermite_run<N, ADAPT, false>(B, P, rd, kcf, [&](bool, bool, int base) {
    const int s = taken ? -1 : unit * (32 / N) + base / N;
    taken = true;
    return s < B.S ? s : -1;
  });
}

// systems of 16..32 bodies, one per warp; shared memory of the warp: kc, d2 [16][32] FP64, kcf
// [16][32] FP32
template <bool ADAPT>
__device__ __forceinline__ void wide_hermite_stream(const BinView &B, const StepParams &P, double *kc, double *d2,
                                                    float *kcf) {
  const int lane = threadIdx.x & 31;
  BplRounds<0> rd;
  rd.kc = kc + lane;
  rd.d2 = d2 + lane;
  bpl_hermite_run<0, ADAPT, false>(B, P, rd, kcf + lane, [&](bool need, bool leader, int base) {
    int sn = 0;
    if (need && leader) sn = atomicAdd(P.work_next, 1);
    sn = __shfl_sync(0xffffffffu, sn, base);
    return stream_system(B, sn);
  });
}

}  // namespace swarm
