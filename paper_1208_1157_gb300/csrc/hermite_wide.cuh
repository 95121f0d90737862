// Hermite-4 (Sec. 2.2.1, Algorithm 2) for larger systems, 16..32 bodies: one system per
// warp, body b in lane b, with the body count a run-time value.  The paper's second
// gravitation variant for larger n (Sec. 4.2) trades shared memory for recomputed square
// roots; here every unordered pair is still evaluated once per evaluation (ring rounds as
// in the body-per-lane mapping, the reaction handed back by shuffle), and only the
// monitor's per-pair data (Hill coefficients and squared distances, up to 16 rounds)
// live in shared memory instead of registers.  The Hermite step itself is
// hermite_bpl_ff.cuh's with the warp as the group; this file holds its FP64 evaluation (and
// what the Runge-Kutta and MVS kernels of these sizes use).
#pragma once
#include "hermite.cuh"

namespace swarm {

constexpr int kWideMaxN = SWARM_MAX_N;
constexpr int kWideRounds = kWideMaxN / 2;  // ring rounds of the largest system
constexpr int kWideWarps = 4;               // warps per CTA of the wide kernel

struct WideRing {
  int n;     // bodies
  int RF;    // rounds with reaction
  int RT;    // all rounds (RF, plus one self-sufficient round when n is even)
};
__device__ __forceinline__ WideRing wide_ring(int n) {
  WideRing R;
  R.n = n;
  R.RF = (n - 1) / 2;
  R.RT = R.RF + ((n & 1) ? 0 : 1);
  return R;
}

// sum over the warp's 32 lanes, result in every lane
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
  return v;
}

// Acceleration and jerk of body b (Eq. 1 and its time derivative).  MON: also q2 (squared
// distance to body 0) and, per round r, the squared distance of this lane's pair
// (b, b + r mod n) in d2s[(r - 1) * 32 + lane].
template <bool MON, int UNROLL = kWideRounds>
__device__ __forceinline__ void wring_accjerk(const F64k &k, const double (&x)[3], const double (&v)[3], double m, int b,
                                              const WideRing &R, double (&a)[3], double (&jk)[3], double &q2,
                                              double *d2s, int lane) {
#pragma unroll
  for (int c = 0; c < 3; c++) {
    a[c] = 0.0;
    jk[c] = 0.0;
  }
  q2 = 0.0;
#pragma unroll UNROLL
  for (int r = 1; r <= kWideRounds; r++) {
    if (r > R.RT) break;  // warp-uniform
    const bool full = r <= R.RF;
    int p = b + r;
    if (p >= R.n) p -= R.n;
    int q = b - r;
    if (q < 0) q += R.n;
    double xj[3], vj[3];
#pragma unroll
    for (int c = 0; c < 3; c++) {
      xj[c] = shfl(x[c], p);
      vj[c] = shfl(v[c], p);
    }
    const double mj = shfl(m, p);
    double dx[3], w[3], rho3, r2;
    pair_geom(k, x, v, xj, vj, dx, w, rho3, r2);
    const double sj = kmul(k, mj, rho3);
#pragma unroll
    for (int c = 0; c < 3; c++) {
      a[c] = fma(sj, dx[c], a[c]);
      jk[c] = fma(sj, w[c], jk[c]);
    }
    if (full) {  // reaction from lane q, which evaluated the pair (q, b)
      const double si = kmul(k, m, rho3);
      double rdx[3], rw[3];
#pragma unroll
      for (int c = 0; c < 3; c++) {
        rdx[c] = shfl(dx[c], q);
        rw[c] = shfl(w[c], q);
      }
      const double rs = shfl(si, q);
#pragma unroll
      for (int c = 0; c < 3; c++) {
        a[c] = fma(-rs, rdx[c], a[c]);
        jk[c] = fma(-rs, rw[c], jk[c]);
      }
      if (MON) {
        const double rr2 = shfl(r2, q);
        if (q == 0) q2 = rr2;
      }
    }
    if (MON) {
      if (p == 0) q2 = r2;
      d2s[(r - 1) * 32 + lane] = r2;
    }
  }
}

// Acceleration only (Eq. 1) of body b, with the pair distances of each round in
// d2s[(r - 1) * 32 + lane] (used by the monitor when the state is the accepted one).
__device__ __forceinline__ void wring_acc(const F64k &k, const double (&x)[3], double m, int b, const WideRing &R,
                                          double (&a)[3], double *d2s, int lane) {
#pragma unroll
  for (int c = 0; c < 3; c++) a[c] = 0.0;
#pragma unroll
  for (int r = 1; r <= kWideRounds; r++) {
    if (r > R.RT) break;  // warp-uniform
    const bool full = r <= R.RF;
    int p = b + r;
    if (p >= R.n) p -= R.n;
    int q = b - r;
    if (q < 0) q += R.n;
    double dx[3];
#pragma unroll
    for (int c = 0; c < 3; c++) dx[c] = ksub(k, shfl(x[c], p), x[c]);
    const double mp = shfl(m, p);
    double r2 = kmul(k, dx[0], dx[0]);
    r2 = fma(dx[1], dx[1], r2);
    r2 = fma(dx[2], dx[2], r2);
    const double rho = rsqrt(r2);
    const double rho3 = kmul(k, kmul(k, rho, rho), rho);
    const double sp = kmul(k, mp, rho3);
#pragma unroll
    for (int c = 0; c < 3; c++) a[c] = fma(sp, dx[c], a[c]);
    if (full) {  // reaction from lane q, which evaluated the pair (q, b)
      const double si = kmul(k, m, rho3);
      double rdx[3];
#pragma unroll
      for (int c = 0; c < 3; c++) rdx[c] = shfl(dx[c], q);
      const double rs = shfl(si, q);
#pragma unroll
      for (int c = 0; c < 3; c++) a[c] = fma(-rs, rdx[c], a[c]);
    }
    d2s[(r - 1) * 32 + lane] = r2;
  }
}

// maximum over the warp's 32 lanes (idle lanes pass 0), result in every lane
__device__ __forceinline__ double warp_max(double v) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, off));
  return v;
}

// Energy (Eq. 6, pairs once) and angular momentum of the warp's system, in every lane.
__device__ __forceinline__ void wring_energy(const double (&x)[3], const double (&v)[3], double m, int b, bool real,
                                             const WideRing &R, double (&out)[4]) {
  double e = 0.5 * m * (v[0] * v[0] + v[1] * v[1] + v[2] * v[2]);
  double L0 = m * (x[1] * v[2] - x[2] * v[1]);
  double L1 = m * (x[2] * v[0] - x[0] * v[2]);
  double L2 = m * (x[0] * v[1] - x[1] * v[0]);
  const int half = R.n / 2;
#pragma unroll
  for (int r = 1; r <= kWideRounds; r++) {
    if (r > half) break;
    int p = b + r;
    if (p >= R.n) p -= R.n;
    const double d0 = shfl(x[0], p) - x[0];
    const double d1 = shfl(x[1], p) - x[1];
    const double d2 = shfl(x[2], p) - x[2];
    const double mp = shfl(m, p);
    double pot = m * mp * rsqrt(d0 * d0 + d1 * d1 + d2 * d2);
    if (!(R.n & 1) && r == half) pot *= 0.5;  // both lanes of the pair count it
    e -= pot;
  }
  out[0] = warp_sum(real ? e : 0.0);
  out[1] = warp_sum(real ? L0 : 0.0);
  out[2] = warp_sum(real ? L1 : 0.0);
  out[3] = warp_sum(real ? L2 : 0.0);
}

}  // namespace swarm
