// Pairs of FP32 numbers ("float-float", 48 significant bits) on the FP32 and integer pipes.
//
// What bounds this chip's kernels here is the FP64 pipe: one FP64 warp instruction holds an
// SM sub-partition's pipe for 64 cycles (76 for DADD/DMUL, 64 for a float<->double
// conversion), while an FP32 instruction takes 1 cycle, an integer one 2 and a shuffle 4
// (measured with chains of each, 1-4 warps per sub-partition; 32 FP32 instructions issued
// next to each DFMA cost 4 cycles more than the DFMA alone at two warps).  A pair product is
// 7 FP32 instructions and a pair sum 11, so work whose weight in the result is 2^-8 or less
// runs 5-9x cheaper as pairs than as FP64 and still lands below half a unit in the last
// place of the FP64 value that it is added to.  Each use states that weight and checks it.
//
// Error-free transformations after Dekker (1971) and Knuth; pair algorithms after Hida, Li
// & Bailey (2001), "sloppy" sums: error below 2^-45 relative to the larger operand.
#pragma once
#include "common.cuh"

namespace swarm {

__device__ __forceinline__ ff ff_make(float h, float l) {
  ff r;
  r.h = h;
  r.l = l;
  return r;
}
__device__ __forceinline__ constexpr ff ff_const(double d) { return ff{(float)d, (float)(d - (double)(float)d)}; }
__device__ __forceinline__ ff ff_sel(bool p, const ff &a, const ff &b) { return ff_make(p ? a.h : b.h, p ? a.l : b.l); }
__device__ __forceinline__ ff ff_neg(const ff &a) { return ff_make(-a.h, -a.l); }
// a + b exactly (|a| >= |b| or a = 0)
__device__ __forceinline__ ff fast_two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  return ff_make(s, __fsub_rn(b, __fsub_rn(s, a)));
}
// a + b exactly
__device__ __forceinline__ ff two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  const float t = __fsub_rn(s, a);
  return ff_make(s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t)));
}
// a b exactly
__device__ __forceinline__ ff two_prod(float a, float b) {
  const float p = __fmul_rn(a, b);
  return ff_make(p, __fmaf_rn(a, b, -p));
}
// The _raw forms leave out the final normalisation (3 instructions): l may overlap h by some
// bits, which later sums and products take as it is; `ff_pack` and `ff_double` want a
// normalised pair.
__device__ __forceinline__ ff ff_norm(const ff &a) { return fast_two_sum(a.h, a.l); }
__device__ __forceinline__ ff ff_add_raw(const ff &a, const ff &b) {
  const ff s = two_sum(a.h, b.h);
  return ff_make(s.h, __fadd_rn(s.l, __fadd_rn(a.l, b.l)));
}
__device__ __forceinline__ ff ff_sub_raw(const ff &a, const ff &b) { return ff_add_raw(a, ff_neg(b)); }
__device__ __forceinline__ ff ff_mul_raw(const ff &a, const ff &b) {
  const ff p = two_prod(a.h, b.h);
  return ff_make(p.h, __fmaf_rn(a.h, b.l, __fmaf_rn(a.l, b.h, p.l)));
}
__device__ __forceinline__ ff ff_fma_raw(const ff &a, const ff &b, const ff &c) { return ff_add_raw(c, ff_mul_raw(a, b)); }
__device__ __forceinline__ ff ff_add(const ff &a, const ff &b) { return ff_norm(ff_add_raw(a, b)); }
__device__ __forceinline__ ff ff_sub(const ff &a, const ff &b) { return ff_add(a, ff_neg(b)); }
__device__ __forceinline__ ff ff_mul(const ff &a, const ff &b) {
  const ff p = ff_mul_raw(a, b);
  return fast_two_sum(p.h, p.l);
}
__device__ __forceinline__ ff ff_mulf(const ff &a, float b) {
  const ff p = two_prod(a.h, b);
  return fast_two_sum(p.h, __fmaf_rn(a.l, b, p.l));
}
// c + a b
__device__ __forceinline__ ff ff_fma(const ff &a, const ff &b, const ff &c) { return ff_norm(ff_fma_raw(a, b, c)); }
// |a|^2 and a . b (three components, one normalisation)
__device__ __forceinline__ ff ff_dot(const ff (&a)[3], const ff (&b)[3]) {
  return ff_norm(ff_fma_raw(a[2], b[2], ff_fma_raw(a[1], b[1], ff_mul_raw(a[0], b[0]))));
}
__device__ __forceinline__ ff ff_norm2(const ff (&a)[3]) {
  ff p = ff_make(0.0f, 0.0f);
#pragma unroll
  for (int c = 0; c < 3; c++) {
    ff q = two_prod(a[c].h, a[c].h);
    q.l = __fmaf_rn(__fadd_rn(a[c].h, a[c].h), a[c].l, q.l);
    if (c == 0) {
      p = q;
    } else {  // squares: the running sum is not always the larger one
      p = ff_add_raw(p, q);
    }
  }
  return ff_norm(p);
}

// Double -> pair on the integer pipe (the conversion instructions run on the FP64 pipe): the
// upper 24 bits truncated, the other 29 rounded to 24, so 2^-48 relative; doubles below
// 2^-126 become 0 (or a subnormal), values of 2^128 and above are not representable (callers
// check their range).
__device__ __forceinline__ ff ff_from(double d) {
  const int hi = __double2hiint(d), lo = __double2loint(d);
  const int e = max((hi & 0x7fffffff) - (896 << 20), 0);
  const int t = (__funnelshift_l(lo, e, 3) & 0x7fffffff) | (hi & 0x80000000);
  const float sc = __int_as_float(t & 0xff800000);  // +-2^E
  const float r = __fmul_rn(__int2float_rn(lo & 0x1fffffff), 0x1p-52f);
  return ff_make(__int_as_float(t), __fmul_rn(r, sc));
}
// its upper part alone (truncated to 24 bits)
__device__ __forceinline__ float f_from(double d) {
  const int hi = __double2hiint(d);
  const int e = max((hi & 0x7fffffff) - (896 << 20), 0);
  return __int_as_float((__funnelshift_l(__double2loint(d), e, 3) & 0x7fffffff) | (hi & 0x80000000));
}

// a double's 53 bits as three floats
struct ff3 {
  float h, l, t;
};
__device__ __forceinline__ ff3 ff3_from(double d) {
  const int hi = __double2hiint(d), lo = __double2loint(d);
  const int e = max((hi & 0x7fffffff) - (896 << 20), 0);
  ff3 r;
  const int top = (__funnelshift_l(lo, e, 3) & 0x7fffffff) | (hi & 0x80000000);
  const float sc = __int_as_float(top & 0xff800000);
  r.h = __int_as_float(top);
  r.l = __fmul_rn(__fmul_rn(__int2float_rn(lo & 0x1fffffe0), 0x1p-52f), sc);
  r.t = __fmul_rn(__fmul_rn(__int2float_rn(lo & 31), 0x1p-52f), sc);
  return r;
}

// Whether every value is below 2^64 in size, and neither NaN nor infinite (exponent bits, integer
// pipe).  NaN, infinity and what is beyond 2^128 come out of the conversions above as ordinary
// numbers (the exponent's upper bits are dropped), so a test of those does not see them.
__device__ __forceinline__ bool ff_tame(const double (&a)[3], const double (&b)[3]) {
  int e = 0;
#pragma unroll
  for (int c = 0; c < 3; c++) e = max(e, max(__double2hiint(a[c]) & 0x7fffffff, __double2hiint(b[c]) & 0x7fffffff));
  return e < (1023 + 64) << 20;
}

// Pair -> double times 2^-896, on the integer pipe: the float's exponent field is taken over
// without its rebias, which the DFMA that adds it supplies (`ff_addto`); the lower part is
// scaled to the double's last place and added to the bits.  Exact for a normalised pair.
constexpr double kFFScale = 0x1p896;
__device__ __forceinline__ double ff_pack(const ff &a) {
  const int t = __float_as_int(a.h);
  const int mag = t & 0x7fffffff;
  // +-2^-E of the upper part, so that l * 2^(52-E) counts units of the double's last place
  const float sc = __int_as_float((0x7f000000 - (t & 0x7f800000)) | (t & 0x80000000));
  const int q = __float2int_rn(__fmul_rn(__fmul_rn(a.l, sc), 0x1p52f));
  const long long top = ((long long)(mag >> 3) << 32) | (unsigned)(mag << 29);
  long long b = top + (long long)q;
  // below a power of two the last place halves: the lower part counts twice there
  if (q < 0 && (((int)(b >> 32) ^ (int)(top >> 32)) & 0x7ff00000)) b += (long long)q;
  return __longlong_as_double(b | ((long long)(t & 0x80000000) << 32));
}
// x + a in one DFMA
__device__ __forceinline__ double ff_addto(double x, const ff &a) { return fma(ff_pack(a), kFFScale, x); }
// the pair as a double
__device__ __forceinline__ double ff_double(const ff &a) {
  const double p = ff_pack(a);
  const int hi = __double2hiint(p);
  return __hiloint2double((hi & 0x7fffffff) ? hi + (896 << 20) : hi, __double2loint(p));
}

// 1/sqrt(a)^3 as a pair, and 1/a (rho2), from the hardware's FP32 reciprocal root y:
// t = 1 - a y^2, rho^2 = y^2 / (1 - t), rho^3 = y^3 (1 - t)^(-3/2).  |t| < 2^-21 (the root's
// error is 2 units at most), so the dropped cubes are below 2^-61.
__device__ __forceinline__ void ff_rho3(const ff &a, ff &rho3, ff &rho2) {
  const float y = rsqrtf(a.h);
  const ff y2 = two_prod(y, y);
  const ff p = ff_mul_raw(a, y2);
  const float t = __fsub_rn(__fsub_rn(1.0f, p.h), p.l);
  const float q2 = __fmaf_rn(t, t, t);
  const float q3 = __fmul_rn(t, __fmaf_rn(t, 1.875f, 1.5f));
  rho2 = fast_two_sum(y2.h, __fmaf_rn(y2.h, q2, y2.l));
  const ff y3 = two_prod(y2.h, y);
  rho3 = fast_two_sum(y3.h, __fmaf_rn(y3.h, q3, __fmaf_rn(y2.l, y, y3.l)));
}

}  // namespace swarm
