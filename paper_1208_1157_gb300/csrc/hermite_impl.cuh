// Hermite-4 work-unit functions (Algorithm 1 with the Algorithm 2 propagator) in the
// two thread mappings; instantiated per body count in hermite_units_*.cu.
#pragma once
#include "hermite.cuh"
#include "hermite_block.cuh"
#include "hermite_ff.cuh"
#include "kernels.h"

namespace swarm {

// ---------------------------------------------------------------- body per lane
// One work unit = one warp's G = 32/N systems of a bin, integrated for the whole call.
template <int N>
__device__ __forceinline__ void bpl_hermite_body(const BinView &B, const StepParams &P, int unit) {
  const bool printed = P.corr_form != 0;  // warp-uniform
  using R = Ring<N>;
  constexpr int G = R::G;
  constexpr int RT = R::RT > 0 ? R::RT : 1;
  const unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  int g = lane / N, b = lane - g * N;
  const bool lane_ok = g < G;
  if (!lane_ok) {  // spare lanes mirror group 0 so every shuffle stays well defined
    g = 0;
    b = lane - G * N;
  }
  const int base = g * N;
  const int s0 = unit * G;
  int s = s0 + g;
  const bool sys_ok = lane_ok && s < B.S;
  if (s >= B.S) s = s0;
  const int SP = B.S_pad;

  double x[3], v[3];
#pragma unroll
  for (int c = 0; c < 3; c++) {
    x[c] = B.x[(size_t)(c * N + b) * SP + s];
    v[c] = B.v[(size_t)(c * N + b) * SP + s];
  }
  const double m = B.m[(size_t)b * SP + s];
  const double t0 = B.t[s];
  const int st0 = B.status[s];
  const double m0 = shfl(m, base);
  const bool runnable = sys_ok && st0 <= SWARM_SYS_DONE;
  const LaunchPlan plan = launch_plan(B, P, s, t0, runnable);
  const int Ns = plan.N;
  const int Nmax = __reduce_max_sync(FULL, Ns);
  if (Nmax == 0) {
    if (runnable && b == 0) B.status[s] = SWARM_SYS_DONE;
    return;
  }

  // close-encounter coefficients of this lane's pairs (planet pairs only)
  double kc[RT];
#pragma unroll
  for (int r = 1; r <= RT; r++) {
    int p = b + r;
    if (p >= N) p -= N;
    double mp = shfl(m, base + p);
    kc[r - 1] = (b != 0 && p != 0 && RT == R::RT) ? hill_kc(P.ce_factor, m, mp, m0) : 0.0;
  }

  double a0[3], j0[3], q2, d2[RT];
  ring_accjerk<N, false>(P.fk, x, v, m, b, base, a0, j0, q2, d2);
  const HCoef cdt = hcoef(P.dt);
  const HCoef clast = hcoef(plan.h_last);
  bool alive = runnable;
  int steps_done = 0;

  for (int k = 1; k <= Nmax; k++) {
    const bool active = alive && (k <= Ns);
    if (!__any_sync(FULL, active)) break;
    const HCoef C = hsel(k == Ns && !plan.exact, clast, cdt);
    // Eq. 3 predictor and the step-invariant parts of the corrector
    double xk[3], vk[3], Xb[3], Vb[3];
#pragma unroll
    for (int c = 0; c < 3; c++) {
      xk[c] = fma(j0[c], C.h3_6, fma(a0[c], C.h2_2, fma(v[c], C.h, x[c])));
      vk[c] = fma(j0[c], C.h2_2, fma(a0[c], C.h, v[c]));
      Vb[c] = fma(j0[c], C.h2_12, fma(a0[c], C.hh, v[c]));
    }
    PCoef PC;
    if (printed) {
      PC = pcoef(C.h);
#pragma unroll
      for (int c = 0; c < 3; c++) Xb[c] = fma(j0[c], PC.pj, fma(a0[c], PC.pa, xk[c]));
    } else {
#pragma unroll
      for (int c = 0; c < 3; c++) Xb[c] = fma(a0[c], C.h2_12, fma(v[c], C.hh, x[c]));
    }
    // corrector passes (time-symmetric form of Eq. 4)
    for (int ic = 0; ic < P.n_corr; ic++) {
      double ak[3], jk[3];
      ring_accjerk<N, false>(P.fk, xk, vk, m, b, base, ak, jk, q2, d2);
#pragma unroll
      for (int c = 0; c < 3; c++) vk[c] = fma(-C.h2_12, jk[c], fma(C.hh, ak[c], Vb[c]));
      if (printed) {
#pragma unroll
        for (int c = 0; c < 3; c++) xk[c] = fma(PC.cj, jk[c], fma(PC.ca, ak[c], Xb[c]));
      } else {
#pragma unroll
        for (int c = 0; c < 3; c++) xk[c] = fma(-C.h2_12, ak[c], fma(C.hh, vk[c], Xb[c]));
      }
    }
    // third evaluation: next step's a0, j0 and the monitor's distances
    double an[3], jn[3];
    ring_accjerk<N, true>(P.fk, xk, vk, m, b, base, an, jn, q2, d2);
    if (active) {
#pragma unroll
      for (int c = 0; c < 3; c++) {
        x[c] = xk[c];
        v[c] = vk[c];
        a0[c] = an[c];
        j0[c] = jn[c];
      }
      steps_done = k;
    }
    // monitor
    const bool nf = nonfinite(x[0]) | nonfinite(x[1]) | nonfinite(x[2]) | nonfinite(v[0]) | nonfinite(v[1]) |
                    nonfinite(v[2]);
    const bool ej = (b != 0) && (P.eject2 > 0.0) && (q2 > P.eject2);
    bool ce = false;
#pragma unroll
    for (int r = 1; r <= RT; r++) {
      int p = b + r;
      if (p >= N) p -= N;
      double q2p = shfl(q2, base + p);
      if (kc[r - 1] > 0.0 && close_encounter(P.fk, d2[r - 1], kc[r - 1], q2, q2p)) ce = true;
    }
    const unsigned gm = ((1u << N) - 1u) << base;
    const unsigned bnf = __ballot_sync(FULL, active && nf) & gm;
    const unsigned bej = __ballot_sync(FULL, active && ej) & gm;
    const unsigned bce = __ballot_sync(FULL, active && ce) & gm;
    const int code = bnf ? SWARM_SYS_NONFINITE : bej ? SWARM_SYS_EJECTED : bce ? SWARM_SYS_CLOSE_ENCOUNTER : 0;
    if (active && code) {
      const double tk = step_time(plan, k, t0, P.dt);
      if (sys_ok) {
#pragma unroll
        for (int c = 0; c < 3; c++) {
          B.x[(size_t)(c * N + b) * SP + s] = x[c];
          B.v[(size_t)(c * N + b) * SP + s] = v[c];
        }
        if (b == 0) {
          B.t[s] = tk;
          B.status[s] = code;
        }
      }
      alive = false;
    }
    if (P.log_interval > 0 && (k % P.log_interval) == 0) {
      double e[4];
      ring_energy<N>(x, v, m, b, base, e);
      if (active && !code && b == 0 && sys_ok) write_log(P, B.gidx[s], step_time(plan, k, t0, P.dt), e);
    }
  }
  if (alive && sys_ok) {
    if (Ns > 0) {
#pragma unroll
      for (int c = 0; c < 3; c++) {
        B.x[(size_t)(c * N + b) * SP + s] = x[c];
        B.v[(size_t)(c * N + b) * SP + s] = v[c];
      }
    }
    if (b == 0) {
      if (Ns > 0) B.t[s] = step_time(plan, Ns, t0, P.dt);
      B.status[s] = plan.full ? SWARM_SYS_DONE : SWARM_SYS_ACTIVE;
    }
  }
  if (P.counters && sys_ok && b == 0 && steps_done > 0) {
    constexpr unsigned long long NP = (unsigned long long)N * (N - 1) / 2;
    atomicAdd(&P.counters[0], (unsigned long long)steps_done);
    atomicAdd(&P.counters[1], NP * (1ull + (unsigned long long)steps_done * (P.n_corr + 1)));
  }
}

// ---------------------------------------------------------------- system per lane
// Each lane integrates one system in coordinates relative to body 0, X_k = x_k - x_0 and
// V_k = v_k - v_0 (k >= 1), plus the uniform motion of the barycentre.  Every operation
// of the Hermite step (Eqs. 3-4) is linear in (x, v, a, jerk) and A_k = a_k - a_0, so this
// is the step of the inertial coordinates in exact arithmetic (the barycentre of the
// inertial step moves by h v_cm, its accelerations summing to zero); it drops body 0's
// predictor and corrector and the coordinate differences of body 0's pairs.  Inertial
// coordinates are rebuilt at log points and at the end:
//   x_0 = X_cm - sum_{k>=1} m_k X_k / M,  x_k = X_k + x_0   (likewise v),
// X_cm moved by its velocity times the time elapsed.
//
// The steps are those of hermite_ff.cuh.  Bound: the FP64 pipe and the issue slots about
// evenly (57 and 58 % at n = 3, two warps per sub-partition at 255 registers; a 3-warp build
// at 168 registers spills and misses the instruction cache: 9 % slower).  131072 x 3 systems
// over 400 steps: 37.0 ms wholly in FP64 (413 FP64 slots per step, the pipe 97 % busy), 8.0 ms
// with 50 FP64 and 3250 other instructions per step; 16384 x 4 over 400 steps 10.8 -> 4.1 ms;
// steps of 0.003 and 0.02 orbits (levels 1 and 0), 100 of them: 9.5 -> 4.1 and 9.6 ms.
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

template <int N>
__device__ __forceinline__ void spl_hermite_body(const BinView &B, const StepParams &P, int unit) {
  const bool printed = P.corr_form != 0;  // warp-uniform
  const int s = unit * 32 + (threadIdx.x & 31);
  if (s >= B.S) return;
  const int SP = B.S_pad;
  double x[N][3], v[N][3], m[N];
#pragma unroll
  for (int i = 0; i < N; i++) {
    m[i] = B.m[(size_t)i * SP + s];
#pragma unroll
    for (int c = 0; c < 3; c++) {
      x[i][c] = B.x[(size_t)(c * N + i) * SP + s];
      v[i][c] = B.v[(size_t)(c * N + i) * SP + s];
    }
  }
  const double t0 = B.t[s];
  if (B.status[s] > SWARM_SYS_DONE) return;
  const LaunchPlan plan = launch_plan(B, P, s, t0, true);
  const int Ns = plan.N;
  if (Ns == 0) {
    B.status[s] = SWARM_SYS_DONE;
    return;
  }
  const FLimits<N> L = flimits<N>(m, P.ce_factor, P.eject2);
  double Minv, Xc[3], Vc[3];
  spl_to_rel<N>(m, x, v, Minv, Xc, Vc);
  FMass<N> F = fmass<N>(m);
  F.ok = F.ok && fscale(P.dt, -60, 40) && !printed;
  double a0[N][3];
  ff j0[N][3], sa[3], sj[3];
  float da[N][3], q2[N], d2[N][N];
  int level = spl_ff_state_call<N, false>(P.fk, F, P.fc.hf, x, v, a0, da, j0, q2, d2, sa, sj);
  int k = 0, code = 0;  // steps done
  const int whole = plan.exact ? Ns : Ns - 1;
  while (k < Ns) {
    if (level == 2 && k < whole) {
      k++;
      level = spl_hermite_delta_step<N, false>(P.fk, F, P.fc, P.fc.hf, P.n_corr, x, v, a0, da, j0, q2, d2, sa, sj);
      code = spl_ff_monitor<N>(P.fk, level, L, q2, d2, x, v, P.eject2);
    } else if (level && k < whole) {
      k++;
      level = spl_hermite_ff_step_call<N, false>(P.fk, F, P.fc, P.fc.hf, P.n_corr, x, v, a0, da, j0, q2, d2, sa, sj);
      code = spl_ff_monitor<N>(P.fk, level, L, q2, d2, x, v, P.eject2);
    } else {
      int count = k < whole ? min(whole - k, kFP64Run) : 1;
      if (P.log_interval > 0) count = min(count, P.log_interval - k % P.log_interval);
      const double h = k < whole ? P.dt : plan.h_last;
      double t = 0.0;
      bool reached = false;
      code = printed ? spl_hermite_fp64_run<N, false, true>(P.fk, m, L.kc, P.eject2, h, P.n_corr, count, true, x, v, a0, j0, k, t, t, reached)
                     : spl_hermite_fp64_run<N, false, false>(P.fk, m, L.kc, P.eject2, h, P.n_corr, count, true, x, v, a0, j0, k, t, t, reached);
      if (!code && k < Ns && !printed) level = spl_ff_state_call<N, false>(P.fk, F, P.fc.hf, x, v, a0, da, j0, q2, d2, sa, sj);
    }
    if (code) break;
    if (P.log_interval > 0 && (k % P.log_interval) == 0) {
      const double tk = step_time(plan, k, t0, P.dt);
      spl_write<N>(B, s, m, x, v, Minv, Xc, Vc, tk - t0, &P, tk);
    }
  }
  const double tk = step_time(plan, k, t0, P.dt);
  spl_write<N>(B, s, m, x, v, Minv, Xc, Vc, tk - t0, nullptr, tk);
  B.t[s] = tk;
  B.status[s] = code ? code : (plan.full ? SWARM_SYS_DONE : SWARM_SYS_ACTIVE);
  if (P.counters) {
    constexpr unsigned long long NP = (unsigned long long)N * (N - 1) / 2;
    atomicAdd(&P.counters[0], (unsigned long long)k);
    atomicAdd(&P.counters[1], NP * (1ull + (unsigned long long)k * (P.n_corr + 1)));
  }
}

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

template <int N>
__device__ __forceinline__ void bpl_hermite_adaptive_body(const BinView &B, const StepParams &P, int unit) {
  const bool printed = P.corr_form != 0;  // warp-uniform
  using R = Ring<N>;
  constexpr int G = R::G;
  constexpr int RT = R::RT > 0 ? R::RT : 1;
  const unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  int g = lane / N, b = lane - g * N;
  const bool lane_ok = g < G;
  if (!lane_ok) {
    g = 0;
    b = lane - G * N;
  }
  const int base = g * N;
  const int s0 = unit * G;
  int s = s0 + g;
  const bool sys_ok = lane_ok && s < B.S;
  if (s >= B.S) s = s0;
  const int SP = B.S_pad;
  double x[3], v[3];
#pragma unroll
  for (int c = 0; c < 3; c++) {
    x[c] = B.x[(size_t)(c * N + b) * SP + s];
    v[c] = B.v[(size_t)(c * N + b) * SP + s];
  }
  const double m = B.m[(size_t)b * SP + s];
  const double t0 = B.t[s];
  const int st0 = B.status[s];
  const double m0 = shfl(m, base);
  const bool runnable = sys_ok && st0 <= SWARM_SYS_DONE;
  const double te = adaptive_end(B, P, s);
  const double tau = fabs(P.dt), dir = P.dt > 0 ? 1.0 : -1.0;
  bool alive = runnable && ((te - t0) * dir > 1e-12 * fmax(1.0, fabs(te)));
  if (!__any_sync(FULL, alive)) {
    if (runnable && b == 0) B.status[s] = SWARM_SYS_DONE;
    return;
  }
  double kc[RT];
#pragma unroll
  for (int r = 1; r <= RT; r++) {
    int p = b + r;
    if (p >= N) p -= N;
    double mp = shfl(m, base + p);
    kc[r - 1] = (b != 0 && p != 0 && RT == R::RT) ? hill_kc(P.ce_factor, m, mp, m0) : 0.0;
  }
  double a0[3], j0[3], q2, d2[RT];
  ring_accjerk<N, false>(P.fk, x, v, m, b, base, a0, j0, q2, d2);
  const int cap = P.max_steps > 0 ? P.max_steps : kAdaptiveStepCap;
  double t = t0;
  int steps_done = 0, code = 0;
  bool reached = false, ran = alive;
  for (int k = 1; k <= cap; k++) {
    if (!__any_sync(FULL, alive)) break;
    // Eq. 5 over the system's bodies (group sum of this lane's |j|^2/|a|^2)
    const double ratio = (j0[0] * j0[0] + j0[1] * j0[1] + j0[2] * j0[2]) / (a0[0] * a0[0] + a0[1] * a0[1] + a0[2] * a0[2]);
    const double ssum = grp_sum<N>(ratio, b, base);
    double h = tau * rsqrt(ssum);
    const double rem = kmul(P.fk, ksub(P.fk, te, t), dir);
    const bool last = h >= rem;
    const bool bad = !(h > 0.0) || nonfinite(h);
    h = kmul(P.fk, last ? rem : h, dir);
    const HCoef C = hcoef(P.fk, h);
    double xk[3], vk[3], Xb[3], Vb[3];
#pragma unroll
    for (int c = 0; c < 3; c++) {
      xk[c] = fma(j0[c], C.h3_6, fma(a0[c], C.h2_2, fma(v[c], C.h, x[c])));
      vk[c] = fma(j0[c], C.h2_2, fma(a0[c], C.h, v[c]));
      Vb[c] = fma(j0[c], C.h2_12, fma(a0[c], C.hh, v[c]));
    }
    PCoef PC;
    if (printed) {
      PC = pcoef(C.h);
#pragma unroll
      for (int c = 0; c < 3; c++) Xb[c] = fma(j0[c], PC.pj, fma(a0[c], PC.pa, xk[c]));
    } else {
#pragma unroll
      for (int c = 0; c < 3; c++) Xb[c] = fma(a0[c], C.h2_12, fma(v[c], C.hh, x[c]));
    }
    for (int ic = 0; ic < P.n_corr; ic++) {
      double ak[3], jk[3];
      ring_accjerk<N, false>(P.fk, xk, vk, m, b, base, ak, jk, q2, d2);
#pragma unroll
      for (int c = 0; c < 3; c++) vk[c] = fma(-C.h2_12, jk[c], fma(C.hh, ak[c], Vb[c]));
      if (printed) {
#pragma unroll
        for (int c = 0; c < 3; c++) xk[c] = fma(PC.cj, jk[c], fma(PC.ca, ak[c], Xb[c]));
      } else {
#pragma unroll
        for (int c = 0; c < 3; c++) xk[c] = fma(-C.h2_12, ak[c], fma(C.hh, vk[c], Xb[c]));
      }
    }
    double an[3], jn[3];
    ring_accjerk<N, true>(P.fk, xk, vk, m, b, base, an, jn, q2, d2);
    const bool active = alive && !bad;
    if (active) {
#pragma unroll
      for (int c = 0; c < 3; c++) {
        x[c] = xk[c];
        v[c] = vk[c];
        a0[c] = an[c];
        j0[c] = jn[c];
      }
      steps_done = k;
      t = last ? te : kadd(P.fk, t, h);
    }
    const bool nf = nonfinite(x[0]) | nonfinite(x[1]) | nonfinite(x[2]) | nonfinite(v[0]) | nonfinite(v[1]) |
                    nonfinite(v[2]);
    const bool ej = (b != 0) && (P.eject2 > 0.0) && (q2 > P.eject2);
    bool ce = false;
#pragma unroll
    for (int r = 1; r <= RT; r++) {
      int p = b + r;
      if (p >= N) p -= N;
      double q2p = shfl(q2, base + p);
      if (kc[r - 1] > 0.0 && close_encounter(P.fk, d2[r - 1], kc[r - 1], q2, q2p)) ce = true;
    }
    const unsigned gm = ((1u << N) - 1u) << base;
    const unsigned bnf = __ballot_sync(FULL, alive && (nf || bad)) & gm;
    const unsigned bej = __ballot_sync(FULL, active && ej) & gm;
    const unsigned bce = __ballot_sync(FULL, active && ce) & gm;
    const int c2 = bnf ? SWARM_SYS_NONFINITE : bej ? SWARM_SYS_EJECTED : bce ? SWARM_SYS_CLOSE_ENCOUNTER : 0;
    if (alive && c2) {
      code = c2;
      alive = false;
    } else if (active && last) {
      reached = true;
      alive = false;
    }
    if (P.log_interval > 0 && (k % P.log_interval) == 0) {
      double e[4];
      ring_energy<N>(x, v, m, b, base, e);
      if (active && !c2 && b == 0 && sys_ok) write_log(P, B.gidx[s], t, e);
    }
  }
  if (sys_ok && ran) {
#pragma unroll
    for (int c = 0; c < 3; c++) {
      B.x[(size_t)(c * N + b) * SP + s] = x[c];
      B.v[(size_t)(c * N + b) * SP + s] = v[c];
    }
    if (b == 0) {
      B.t[s] = t;
      B.status[s] = code ? code : (reached ? SWARM_SYS_DONE : SWARM_SYS_ACTIVE);
    }
  } else if (runnable && b == 0) {
    B.status[s] = SWARM_SYS_DONE;  // already at its end time
  }
  if (P.counters && sys_ok && b == 0 && steps_done > 0) {
    constexpr unsigned long long NP = (unsigned long long)N * (N - 1) / 2;
    atomicAdd(&P.counters[0], (unsigned long long)steps_done);
    atomicAdd(&P.counters[1], NP * (1ull + (unsigned long long)steps_done * (P.n_corr + 1)));
  }
}

// Adaptive steps, system per lane, with work handed out per lane: a lane whose system
// reached its end time (or stopped) takes its next system at once, so the warp does not wait
// for the lane with the most steps (adaptive step counts differ from system to system).  One
// loop, each round either loads a new system (that lane only) or takes one step.  take(): the
// lane's next system, or -1.  Steps as in spl_hermite_body, with Eq. 5's length in pairs.  The guard of a state wants the length of
// the step from it, which follows from that state's evaluation: it is given 1.25 times the
// present length, and a longer step is taken in FP64.  A system that comes to level 0 stays
// in FP64 (eta is about tau / sqrt 2 all along an orbit, and lanes that change back and forth
// at their own times would make a warp take both kinds of step).  131072 x 3 systems over a
// quarter of an inner period: 37.4 -> 18 ms; the loop is long enough to miss the instruction
// cache (lanes are at different points of their systems).
template <int N, class Take>
__device__ __forceinline__ void spl_hermite_adaptive_run(const BinView &B, const StepParams &P, Take take) {
  const bool printed = P.corr_form != 0;  // warp-uniform
  const unsigned FULL = 0xffffffffu;
  const int SP = B.S_pad;
  const double dir = P.dt > 0 ? 1.0 : -1.0;
  const ff tau = ff_from(fabs(P.dt));
  const int cap = P.max_steps > 0 ? P.max_steps : kAdaptiveStepCap;
  double x[N][3], v[N][3], m[N], a0[N][3];
  ff j0[N][3], sa[3], sj[3], h;
  float da[N][3], q2[N], d2[N][N], hf = 0.0f;
  FLimits<N> L;
  FMass<N> F;
  double Minv = 1.0, Xc[3] = {0.0, 0.0, 0.0}, Vc[3] = {0.0, 0.0, 0.0};
  double t = 0.0, t0 = 0.0, te = 0.0;
  int s = 0, steps = 0, level = 0;
  bool carried = false;  // a0, j0 are those of an FP64 step
  bool has = false, exhausted = false;
  auto next_step = [&]() {
    h = spl_ff_eq5<N>(tau, a0, da, j0, sa, sj);
    if (!(h.h > 0.0f && h.h <= hf)) level = 0;
  };
  auto look = [&]() {  // at a state whose step length is not known yet
    spl_ff_state_call<N, true>(P.fk, F, 0.0f, x, v, a0, da, j0, q2, d2, sa, sj);
    h = spl_ff_eq5<N>(tau, a0, da, j0, sa, sj);
    hf = 1.25f * h.h;
    level = spl_ff_state_call<N, true>(P.fk, F, hf, x, v, a0, da, j0, q2, d2, sa, sj);
    next_step();
  };
  for (;;) {
    if (!has && !exhausted) {
      s = take();
      if (s < 0) {
        exhausted = true;
      } else if (B.status[s] <= SWARM_SYS_DONE) {
#pragma unroll
        for (int i = 0; i < N; i++) {
          m[i] = B.m[(size_t)i * SP + s];
#pragma unroll
          for (int c = 0; c < 3; c++) {
            x[i][c] = B.x[(size_t)(c * N + i) * SP + s];
            v[i][c] = B.v[(size_t)(c * N + i) * SP + s];
          }
        }
        t0 = t = B.t[s];
        te = adaptive_end(B, P, s);
        if (!((te - t) * dir > 1e-12 * fmax(1.0, fabs(te)))) {
          B.status[s] = SWARM_SYS_DONE;
        } else {
          L = flimits<N>(m, P.ce_factor, P.eject2);
          F = fmass<N>(m);
          F.ok = F.ok && fscale(P.dt, -60, 40) && !printed;
          spl_to_rel<N>(m, x, v, Minv, Xc, Vc);
          look();
          steps = 0;
          carried = false;
          has = true;
        }
      }
    }
    if (!__any_sync(FULL, has || !exhausted)) break;
    if (!has) continue;
    int code = 0;
    bool reached = false;
    if (level) {
      const double rem = kmul(P.fk, ksub(P.fk, te, t), dir);
      double hd = ff_double(h);
      // compared in FP32 first (FP64 compares are slow)
      const bool last = h.h >= 0.999f * f_from(rem) && hd >= rem;
      if (last) hd = rem;
      hd = kmul(P.fk, hd, dir);
      const FCoef C = fcoef(hd);
      hf = 1.25f * C.hf;
      if (level == 2) {
        level = spl_hermite_delta_step<N, true>(P.fk, F, C, hf, P.n_corr, x, v, a0, da, j0, q2, d2, sa, sj);
      } else {
        level = spl_hermite_ff_step_call<N, true>(P.fk, F, C, hf, P.n_corr, x, v, a0, da, j0, q2, d2, sa, sj);
      }
      steps++;
      t = last ? te : kadd(P.fk, t, hd);
      code = spl_ff_monitor<N>(P.fk, level, L, q2, d2, x, v, P.eject2);
      reached = last && !code;
      next_step();
    } else {
      code = printed ? spl_hermite_fp64_run<N, true, true>(P.fk, m, L.kc, P.eject2, P.dt, P.n_corr, 1, !carried, x, v, a0, j0, steps, t, te, reached)
                     : spl_hermite_fp64_run<N, true, false>(P.fk, m, L.kc, P.eject2, P.dt, P.n_corr, 1, !carried, x, v, a0, j0, steps, t, te, reached);
      carried = true;
    }
    if (!code && P.log_interval > 0 && steps > 0 && (steps % P.log_interval) == 0)
      spl_write<N>(B, s, m, x, v, Minv, Xc, Vc, t - t0, &P, t);
    if (code != 0 || reached || steps >= cap) {
      spl_write<N>(B, s, m, x, v, Minv, Xc, Vc, t - t0, nullptr, t);
      B.t[s] = t;
      B.status[s] = code ? code : (reached ? SWARM_SYS_DONE : SWARM_SYS_ACTIVE);
      if (P.counters && steps > 0) {
        constexpr unsigned long long NP = (unsigned long long)N * (N - 1) / 2;
        atomicAdd(&P.counters[0], (unsigned long long)steps);
        atomicAdd(&P.counters[1], NP * (1ull + (unsigned long long)steps * (P.n_corr + 1)));
      }
      has = false;
    }
  }
}
template <int N>
__device__ __forceinline__ void spl_hermite_adaptive_stream(const BinView &B, const StepParams &P) {
  spl_hermite_adaptive_run<N>(B, P, [&]() { return stream_system(B, atomicAdd(P.work_next, 1)); });
}
// one unit: 32 consecutive entries of the launch's system order
template <int N>
__device__ __forceinline__ void spl_hermite_adaptive_body(const BinView &B, const StepParams &P, int unit) {
  bool taken = false;
  spl_hermite_adaptive_run<N>(B, P, [&]() {
    const int s = taken ? -1 : stream_system(B, unit * 32 + (threadIdx.x & 31));
    taken = true;
    return s;
  });
}

// Body per lane with work handed out per system: each of the warp's G groups takes the
// bin's next system as soon as its own one reached its end time or stopped (fixed steps:
// stops and per-system end times; adaptive steps: step counts differ from system to
// system).  A refill round loads the new systems and evaluates their a0, j0 (the other
// groups re-evaluate their unchanged state, which gives the same values); per system
// the arithmetic is that of bpl_hermite_body / bpl_hermite_adaptive_body.
template <int N, bool ADAPT>
__device__ __forceinline__ void bpl_hermite_stream(const BinView &B, const StepParams &P) {
  const bool printed = P.corr_form != 0;  // warp-uniform
  using R = Ring<N>;
  constexpr int G = R::G;
  constexpr int RT = R::RT > 0 ? R::RT : 1;
  constexpr unsigned long long NP = (unsigned long long)N * (N - 1) / 2;
  const unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  int g = lane / N, b = lane - g * N;
  const bool lane_ok = g < G;
  if (!lane_ok) {  // spare lanes mirror group 0 (same broadcasts, same state)
    g = 0;
    b = lane - G * N;
  }
  const int base = g * N;
  const int SP = B.S_pad;
  const unsigned gm = ((1u << N) - 1u) << base;
  const double tau = fabs(P.dt), dir = P.dt > 0 ? 1.0 : -1.0;
  const int cap = P.max_steps > 0 ? P.max_steps : kAdaptiveStepCap;
  const HCoef cdt = hcoef(P.dt);

  int s = 0;
  bool has = false, exhausted = false;
  double x[3] = {0.0, 0.0, 0.0}, v[3] = {0.0, 0.0, 0.0}, m = 1.0, a0[3], j0[3], kc[RT];
  LaunchPlan plan;
  plan.N = 0;
  plan.full = 1;
  plan.exact = 1;
  plan.h_last = P.dt;
  plan.t_end = P.t_end;
  HCoef clast = cdt;  // coefficients of a shortened last step (fixed steps)
  double t = 0.0, t0 = 0.0, te = 0.0;  // fixed steps: t is formed from t0 when needed
  int steps = 0;
#pragma unroll
  for (int r = 0; r < RT; r++) kc[r] = 0.0;

  for (;;) {
    // ---- refill: groups without a system take the bin's next one
    const bool need = !has && !exhausted;
    if (__any_sync(FULL, need)) {
      int sn = 0;
      if (need && lane_ok && b == 0) sn = atomicAdd(P.work_next, 1);
      sn = __shfl_sync(FULL, sn, base);
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
      const double m0 = shfl(m, base);
#pragma unroll
      for (int r = 1; r <= RT; r++) {
        int p = b + r;
        if (p >= N) p -= N;
        double mp = shfl(m, base + p);
        const double k = (b != 0 && p != 0 && RT == R::RT) ? hill_kc(P.ce_factor, m, mp, m0) : 0.0;
        if (take) kc[r - 1] = k;
      }
      double an[3], jn[3], q2, d2[RT];
      ring_accjerk<N, false>(P.fk, x, v, m, b, base, an, jn, q2, d2);
      if (take) {
#pragma unroll
        for (int c = 0; c < 3; c++) {
          a0[c] = an[c];
          j0[c] = jn[c];
        }
        t0 = B.t[s];
        t = t0;
        steps = 0;
        const bool runnable = B.status[s] <= SWARM_SYS_DONE;
        bool go;
        if (!ADAPT) {
          plan = launch_plan(B, P, s, t0, runnable);
          go = runnable && plan.N > 0;
          clast = hcoef(plan.exact ? P.dt : plan.h_last);
        } else {
          te = adaptive_end(B, P, s);
          go = runnable && ((te - t0) * dir > 1e-12 * fmax(1.0, fabs(te)));
        }
        has = go;
        if (runnable && !go && lane_ok && b == 0) B.status[s] = SWARM_SYS_DONE;
      }
      continue;
    }
    if (!__any_sync(FULL, has)) break;

    // ---- one step for every group holding a system
    const bool alive = has;
    HCoef C;
    bool last, bad = false;
    double h = 0.0;
    if (!ADAPT) {
      last = steps + 1 == plan.N;
      C = hsel(last, clast, cdt);
    } else {
      const double ratio = (j0[0] * j0[0] + j0[1] * j0[1] + j0[2] * j0[2]) / (a0[0] * a0[0] + a0[1] * a0[1] + a0[2] * a0[2]);
      const double ssum = grp_sum<N>(ratio, b, base);
      h = tau * rsqrt(ssum);
      const double rem = kmul(P.fk, ksub(P.fk, te, t), dir);
      last = h >= rem;
      bad = !(h > 0.0) || nonfinite(h);
      h = kmul(P.fk, last ? rem : h, dir);
      C = hcoef(P.fk, h);
    }
    double xk[3], vk[3], Xb[3], Vb[3];
#pragma unroll
    for (int c = 0; c < 3; c++) {
      xk[c] = fma(j0[c], C.h3_6, fma(a0[c], C.h2_2, fma(v[c], C.h, x[c])));
      vk[c] = fma(j0[c], C.h2_2, fma(a0[c], C.h, v[c]));
      Vb[c] = fma(j0[c], C.h2_12, fma(a0[c], C.hh, v[c]));
    }
    PCoef PC;
    if (printed) {
      PC = pcoef(C.h);
#pragma unroll
      for (int c = 0; c < 3; c++) Xb[c] = fma(j0[c], PC.pj, fma(a0[c], PC.pa, xk[c]));
    } else {
#pragma unroll
      for (int c = 0; c < 3; c++) Xb[c] = fma(a0[c], C.h2_12, fma(v[c], C.hh, x[c]));
    }
    double q2, d2[RT];
    for (int ic = 0; ic < P.n_corr; ic++) {
      double ak[3], jk[3];
      ring_accjerk<N, false>(P.fk, xk, vk, m, b, base, ak, jk, q2, d2);
#pragma unroll
      for (int c = 0; c < 3; c++) vk[c] = fma(-C.h2_12, jk[c], fma(C.hh, ak[c], Vb[c]));
      if (printed) {
#pragma unroll
        for (int c = 0; c < 3; c++) xk[c] = fma(PC.cj, jk[c], fma(PC.ca, ak[c], Xb[c]));
      } else {
#pragma unroll
        for (int c = 0; c < 3; c++) xk[c] = fma(-C.h2_12, ak[c], fma(C.hh, vk[c], Xb[c]));
      }
    }
    double an[3], jn[3];
    ring_accjerk<N, true>(P.fk, xk, vk, m, b, base, an, jn, q2, d2);
    const bool active = alive && !bad;
    if (active) {
#pragma unroll
      for (int c = 0; c < 3; c++) {
        x[c] = xk[c];
        v[c] = vk[c];
        a0[c] = an[c];
        j0[c] = jn[c];
      }
      steps++;
      if (ADAPT) t = last ? te : kadd(P.fk, t, h);
    }
    const bool nf = nonfinite(x[0]) | nonfinite(x[1]) | nonfinite(x[2]) | nonfinite(v[0]) | nonfinite(v[1]) |
                    nonfinite(v[2]);
    const bool ej = (b != 0) && (P.eject2 > 0.0) && (q2 > P.eject2);
    bool ce = false;
#pragma unroll
    for (int r = 1; r <= RT; r++) {
      int p = b + r;
      if (p >= N) p -= N;
      double q2p = shfl(q2, base + p);
      if (kc[r - 1] > 0.0 && close_encounter(P.fk, d2[r - 1], kc[r - 1], q2, q2p)) ce = true;
    }
    const unsigned bnf = __ballot_sync(FULL, alive && (nf || bad)) & gm;
    const unsigned bej = __ballot_sync(FULL, active && ej) & gm;
    const unsigned bce = __ballot_sync(FULL, active && ce) & gm;
    int code = bnf ? SWARM_SYS_NONFINITE : bej ? SWARM_SYS_EJECTED : bce ? SWARM_SYS_CLOSE_ENCOUNTER : 0;
    if (!alive) code = 0;
    const bool reached = active && last && !code;
    const bool capped = ADAPT && active && steps >= cap;
    const bool finish = alive && (code != 0 || reached || capped);
    if (!ADAPT && (finish || (P.log_interval > 0 && active && (steps % P.log_interval) == 0)))
      t = step_time(plan, steps, t0, P.dt);
    if (P.log_interval > 0) {
      const bool need_log = active && !code && (steps % P.log_interval) == 0;
      if (__any_sync(FULL, need_log)) {
        double e4[4];
        ring_energy<N>(x, v, m, b, base, e4);
        if (need_log && lane_ok && b == 0) write_log(P, B.gidx[s], t, e4);
      }
    }
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
        if (P.counters && steps > 0) {
          atomicAdd(&P.counters[0], (unsigned long long)steps);
          atomicAdd(&P.counters[1], NP * (1ull + (unsigned long long)steps * (P.n_corr + 1)));
        }
      }
    }
    if (finish) has = false;
  }
}

// Out-of-line copies called by the multi-body-count dispatcher kernel.
template <int N>
__device__ __noinline__ void bpl_hermite_unit(const BinView &B, const StepParams &P, int unit) {
  bpl_hermite_body<N>(B, P, unit);
}
template <int N>
__device__ __noinline__ void spl_hermite_unit(const BinView &B, const StepParams &P, int unit) {
  spl_hermite_body<N>(B, P, unit);
}
template <int N>
__device__ __noinline__ void bpl_hermite_adaptive_unit(const BinView &B, const StepParams &P, int unit) {
  bpl_hermite_adaptive_body<N>(B, P, unit);
}
template <int N>
__device__ __noinline__ void spl_hermite_adaptive_unit(const BinView &B, const StepParams &P, int unit) {
  spl_hermite_adaptive_body<N>(B, P, unit);
}

// Persistent kernel for one bin (one body count, one mapping): the unit body is inlined,
// so registers are allocated for this n alone.  Warps pull unit indices from a counter.
template <int MAP, int N, bool ADAPT = false>
__global__ void __launch_bounds__(128, 2) hermite_uniform_kernel(BinView B, int nunits, StepParams P) {
  if (ADAPT && MAP == SWARM_MAP_SYSTEM_PER_LANE) {  // work unit = system (per-lane refill)
    spl_hermite_adaptive_stream<N>(B, P);
    return;
  }
  if (MAP == SWARM_MAP_BODY_PER_LANE) {  // work unit = system (per-group refill)
    bpl_hermite_stream<N, ADAPT>(B, P);
    return;
  }
  const int lane = threadIdx.x & 31;
  for (;;) {
    int w = 0;
    if (lane == 0) w = atomicAdd(P.work_next, 1);
    w = __shfl_sync(0xffffffffu, w, 0);
    if (w >= nunits) break;
    spl_hermite_body<N>(B, P, w);
  }
}

template <int MAP, int N, bool ADAPT = false>
cudaError_t launch_hermite_uniform_n(const BinView &B, int nunits, const StepParams &P, int grid, cudaStream_t st) {
  StepParams Q = P;
  Q.fc = fcoef_host(P.dt);
  hermite_uniform_kernel<MAP, N, ADAPT><<<grid, 128, 0, st>>>(B, nunits, Q);
  return cudaGetLastError();
}
template <int MAP, int N, bool ADAPT = false>
int hermite_uniform_blocks_n() {
  int nb = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, hermite_uniform_kernel<MAP, N, ADAPT>, 128, 0);
  return nb;
}
// adaptive (Eq. 5) single-bin kernels: both mappings, registers sized for 2 CTAs per SM
template <int MAP, int N>
cudaError_t launch_hermite_uniform_pick(const BinView &B, int nunits, const StepParams &P, int grid, cudaStream_t st,
                                        int *blocks, bool adaptive) {
  if (adaptive) {
    if (blocks) *blocks = hermite_uniform_blocks_n<MAP, N, true>();
    return grid > 0 ? launch_hermite_uniform_n<MAP, N, true>(B, nunits, P, grid, st) : cudaSuccess;
  }
  // fixed steps, body per lane, n >= 5: systems packed across the CTA (hermite_block.cuh)
  // when the bin fills a wave of those CTAs; a smaller bin's step latency is the limit,
  // and the warp ring's shuffles are shorter than the block ring's barriers there
  if constexpr (MAP == SWARM_MAP_BODY_PER_LANE && N >= kBlockRingMinN) {
    if (block_ring_pays(B, N, BlockRing<N>::T, BlockRing<N>::CPS, P.concurrent != 0)) return launch_hermite_block_n<N>(B, nunits, P, grid, st, blocks);
  }
  if (blocks) *blocks = hermite_uniform_blocks_n<MAP, N>();
  return grid > 0 ? launch_hermite_uniform_n<MAP, N>(B, nunits, P, grid, st) : cudaSuccess;
}

}  // namespace swarm
