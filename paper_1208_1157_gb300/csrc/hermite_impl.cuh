// Hermite-4 work-unit functions (Algorithm 1 with the Algorithm 2 propagator) in the
// two thread mappings; instantiated per body count in hermite_units_*.cu.
#pragma once
#include "hermite.cuh"
#include "hermite_block.cuh"
#include "hermite_bpl_ff.cuh"
#include "hermite_ff.cuh"
#include "kernels.h"

namespace swarm {

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
// evenly (60 and 65 % at n = 3, two warps per sub-partition at 255 registers; a 3-warp build
// at 168 registers spills and misses the instruction cache: 9 % slower).  131072 x 3 systems
// over 400 steps: 37.0 ms wholly in FP64 (413 FP64 slots per step, the pipe 97 % busy), 7.8 ms
// with 47 FP64 and 3210 other instructions per step; widely spaced systems, 300 steps of 0.003 and 0.02
// orbits (levels 1 and 0): 27.8 -> 11.1 and 28.3 -> 28.8 ms.
template <int N>
__device__ __forceinline__ void spl_hermite_body(const BinView &B, const StepParams &P, int unit) {
  const bool printed = P.corr_form != 0;  // warp-uniform
  const int s = unit * 32 + (threadIdx.x & 31);
  double t0 = 0.0;
  LaunchPlan plan;
  plan.N = 0;
  if (s < B.S && B.status[s] <= SWARM_SYS_DONE) {
    t0 = B.t[s];
    plan = launch_plan(B, P, s, t0, true);
    if (plan.N == 0) B.status[s] = SWARM_SYS_DONE;
  }
  const int Ns = plan.N;
  const unsigned lanes = __ballot_sync(0xffffffffu, Ns > 0);  // those with a system to integrate
  if (Ns == 0) return;
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
  auto log = [&]() {
    if (!code && P.log_interval > 0 && (k % P.log_interval) == 0) {
      const double tk = step_time(plan, k, t0, P.dt);
      spl_write<N>(B, s, m, x, v, Minv, Xc, Vc, tk - t0, &P, tk);
    }
  };
  // kStepRun steps of the lanes in pairs, then as many of those in FP64: lanes of compact systems
  // change back and forth, each at its own time, and one run of FP64 steps for all that wait costs
  // the warp as much as one for a single lane.  131072 compact systems over 300 steps of 0.005 and
  // 0.01 orbits: n = 3 87 and 103 ms with a run at once for each lane, now 57 and 53 (wholly FP64
  // 28); n = 4 270 and 254, now 178 and 204 (55).  What is left is fetching three kinds of steps of
  // 50 KB and more; widely spaced systems, all of one kind: n = 3 11 ms, n = 4 37.
  while (__any_sync(lanes, k < Ns && !code)) {
    if (!__any_sync(lanes, level == 1 && k < whole && !code)) {  // the loop that fits the instruction cache
      for (int c = 0; c < kStepRun && level == 2 && k < whole && !code; c++) {
        k++;
        level = spl_hermite_delta_step<N, false>(P.fk, F, P.fc, P.fc.hf, P.n_corr, x, v, a0, da, j0, q2, d2, sa, sj);
        code = spl_ff_monitor<N>(P.fk, level, L, q2, d2, x, v, P.eject2);
        log();
      }
    } else {
      for (int c = 0; c < kStepRun && level && k < whole && !code; c++) {
        k++;
        level = level == 2 ? spl_hermite_delta_step_call<N>(P.fk, F, P.fc, P.fc.hf, P.n_corr, x, v, a0, da, j0, q2, d2, sa, sj)
                           : spl_hermite_ff_step_call<N, false>(P.fk, F, P.fc, P.fc.hf, P.n_corr, x, v, a0, da, j0, q2, d2, sa, sj);
        code = spl_ff_monitor<N>(P.fk, level, L, q2, d2, x, v, P.eject2);
        log();
      }
    }
    __syncwarp(lanes);
    if ((level == 0 || k >= whole) && k < Ns && !code) {
      int count = k < whole ? min(whole - k, kStepRun) : 1;
      if (P.log_interval > 0) count = min(count, P.log_interval - k % P.log_interval);
      const double h = k < whole ? P.dt : plan.h_last;
      double t = 0.0;
      bool reached = false;
      code = printed ? spl_hermite_fp64_run<N, false, true>(P.fk, m, L.kc, P.eject2, h, P.n_corr, count, true, x, v, a0, j0, k, t, t, reached)
                     : spl_hermite_fp64_run<N, false, false>(P.fk, m, L.kc, P.eject2, h, P.n_corr, count, true, x, v, a0, j0, k, t, t, reached);
      if (!code && k < Ns && !printed) level = spl_ff_state_call<N, false>(P.fk, F, P.fc.hf, x, v, a0, da, j0, q2, d2, sa, sj);
      log();
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

// Adaptive steps, system per lane, with work handed out per lane: a lane whose system
// reached its end time (or stopped) takes its next system at once, so the warp does not wait
// for the lane with the most steps (adaptive step counts differ from system to system).  One
// loop, each round either loads a new system (that lane only) or takes one step.  take(): the
// lane's next system, or -1.  Steps as in spl_hermite_body, with Eq. 5's length in pairs.  The guard of a state wants the length of
// the step from it, which follows from that state's evaluation: it is given 1.25 times the
// present length, and a longer step is taken in FP64.  A system that comes to level 0 stays
// in FP64 (eta is about tau / sqrt 2 all along an orbit, and lanes that change back and forth
// at their own times would make a warp take both kinds of step).  131072 x 3 systems over a
// quarter of an inner period: 37.4 ms wholly in FP64, now 15.
// CTA: the warps of a CTA take their steps together.  The loop is longer than the instruction
// cache (4500 instructions), and warps at different places of it would each fetch all of it for
// themselves: 131072 systems over a quarter period 18.5 -> 15.0 ms, 65536 11.1 -> 10.2, 30011
// 5.1 either way (the longest system's chain); adaptive Cash-Karp, 131072 systems 20.8 -> 10.6.
template <int N, bool CTA, class Take>
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
    bool more = __any_sync(FULL, has || !exhausted);
    if (CTA) more = __syncthreads_or(more);
    if (!more) break;
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
  spl_hermite_adaptive_run<N, true>(B, P, [&]() { return stream_system(B, atomicAdd(P.work_next, 1)); });
}
// one unit: 32 consecutive entries of the launch's system order
template <int N>
__device__ __forceinline__ void spl_hermite_adaptive_body(const BinView &B, const StepParams &P, int unit) {
  bool taken = false;
  spl_hermite_adaptive_run<N, false>(B, P, [&]() {
    const int s = taken ? -1 : stream_system(B, unit * 32 + (threadIdx.x & 31));
    taken = true;
    return s;
  });
}

// Out-of-line copies called by the multi-body-count dispatcher kernel.
template <int N>
__device__ __noinline__ void bpl_hermite_unit(const BinView &B, const StepParams &P, int unit) {
  bpl_hermite_body<N, false>(B, P, unit);
}
template <int N>
__device__ __noinline__ void spl_hermite_unit(const BinView &B, const StepParams &P, int unit) {
  spl_hermite_body<N>(B, P, unit);
}
template <int N>
__device__ __noinline__ void bpl_hermite_adaptive_unit(const BinView &B, const StepParams &P, int unit) {
  bpl_hermite_body<N, true>(B, P, unit);
}
template <int N>
__device__ __noinline__ void spl_hermite_adaptive_unit(const BinView &B, const StepParams &P, int unit) {
  spl_hermite_adaptive_body<N>(B, P, unit);
}

// Persistent kernel for one bin (one body count, one mapping): the unit body is inlined,
// so registers are allocated for this n alone.  Warps pull unit indices from a counter.
// Body per lane: three CTAs per SM, or two where the step's latency is all that counts, up to
// four bodies (a bin that fills the chip runs system per lane) and observations on the way
// (without the spills 1024 x 3 systems over 400 steps take 1.88 instead of 1.92 ms).  P: its address
// goes to functions out of line, and the loop is to read it from constant memory all the same.
template <int MAP, int N, bool ADAPT = false, bool OBS = false>
__global__ void __launch_bounds__(128, MAP == SWARM_MAP_BODY_PER_LANE && N > 4 && !OBS ? 3 : 2) hermite_uniform_kernel(BinView B, int nunits, const __grid_constant__ StepParams P) {
  if (ADAPT && MAP == SWARM_MAP_SYSTEM_PER_LANE) {  // work unit = system (per-lane refill)
    spl_hermite_adaptive_stream<N>(B, P);
    return;
  }
  if (MAP == SWARM_MAP_BODY_PER_LANE) {  // work unit = system (per-group refill)
    bpl_hermite_stream<N, ADAPT, OBS>(B, P);
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

template <int MAP, int N, bool ADAPT = false, bool OBS = false>
cudaError_t launch_hermite_uniform_n(const BinView &B, int nunits, const StepParams &P, int grid, cudaStream_t st) {
  StepParams Q = P;
  Q.fc = fcoef_host(P.dt);
  hermite_uniform_kernel<MAP, N, ADAPT, OBS><<<grid, 128, 0, st>>>(B, nunits, Q);
  return cudaGetLastError();
}
template <int MAP, int N, bool ADAPT = false, bool OBS = false>
int hermite_uniform_blocks_n() {
  int nb = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, hermite_uniform_kernel<MAP, N, ADAPT, OBS>, 128, 0);
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
  // the printed corrector's steps are FP64: body per lane, n >= 5, packed across the CTA
  // (hermite_block.cuh) when the bin fills a wave of those CTAs; a smaller bin's step latency
  // is the limit, and the warp ring's shuffles are shorter than the block ring's barriers
  // there
  if constexpr (MAP == SWARM_MAP_BODY_PER_LANE && N >= kBlockRingMinN) {
    if (P.corr_form && block_ring_pays(B, N, BlockRing<N>::T, BlockRing<N>::CPS, P.concurrent != 0)) return launch_hermite_block_n<N>(B, nunits, P, grid, st, blocks);
  }
  if (blocks) *blocks = hermite_uniform_blocks_n<MAP, N>();
  return grid > 0 ? launch_hermite_uniform_n<MAP, N>(B, nunits, P, grid, st) : cudaSuccess;
}

}  // namespace swarm
