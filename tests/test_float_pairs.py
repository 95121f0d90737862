"""The float-pair arithmetic of csrc/ff.cuh (compiled from its source as host code) against
exact rationals, at the edges of its conversions."""
import os
import re
import shutil
import subprocess
from fractions import Fraction

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1208_1157_gb300", "csrc")

SHIMS = r"""
#include <cmath>
#include <cstdio>
#include <cstring>
#include <algorithm>
using std::fma; using std::max;
#define __device__
#define __forceinline__ inline
static inline int __double2hiint(double a) { long long b; memcpy(&b, &a, 8); return (int)(b >> 32); }
static inline int __double2loint(double a) { long long b; memcpy(&b, &a, 8); return (int)b; }
static inline double __hiloint2double(int h, int l) { long long b = ((long long)h << 32) | (unsigned)l; double d; memcpy(&d, &b, 8); return d; }
static inline double __longlong_as_double(long long b) { double d; memcpy(&d, &b, 8); return d; }
static inline int __float_as_int(float f) { int i; memcpy(&i, &f, 4); return i; }
static inline float __int_as_float(int i) { float f; memcpy(&f, &i, 4); return f; }
static inline float __fadd_rn(float a, float b) { return a + b; }
static inline float __fsub_rn(float a, float b) { return a - b; }
static inline float __fmul_rn(float a, float b) { return a * b; }
static inline float __fmaf_rn(float a, float b, float c) { return std::fmaf(a, b, c); }
static inline float __int2float_rn(int i) { return (float)i; }
static inline int __float2int_rn(float f) { return (int)nearbyintf(f); }
static inline unsigned __funnelshift_l(unsigned lo, unsigned hi, int s) { return (hi << s) | (lo >> (32 - s)); }
static inline float rsqrtf(float x) { return (float)(1.0 / std::sqrt((double)x)); }
struct ff { float h, l; };
"""

MAIN = r"""
int main() {
  double x, y;
  while (scanf("%la %la", &x, &y) == 2) {
    const ff a = ff_from(x), b = ff_from(y), s = ff_add(a, b), p = ff_mul(a, b);
    ff r3, r2;
    ff_rho3(ff_from(fabs(x)), r3, r2);
    printf("%a %a %a %a %a %a %a %a %a\n", ff_double(a), ff_addto(y, a), (double)s.h, (double)s.l, (double)p.h, (double)p.l,
           (double)r3.h + (double)r3.l, (double)r2.h + (double)r2.l, (double)f_from(x));
  }
}
"""


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("no g++")
    src = open(os.path.join(CSRC, "ff.cuh")).read()
    src = re.sub(r"#(pragma once|include .*)\n", "", src)
    d = tmp_path_factory.mktemp("ff")
    (d / "f.cpp").write_text(SHIMS + src + "using namespace swarm;\n" + MAIN)
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-Wno-unknown-pragmas", "-o", str(d / "f"),
                    str(d / "f.cpp")], check=True)
    return str(d / "f")


def test_pairs_against_exact_rationals(exe):
    rng = np.random.default_rng(3)
    # mantissas around powers of two (the packing's borrow crosses a binade there), all ones,
    # random ones, and zero; both signs
    m = np.concatenate([1.0 + np.arange(-40, 41) * 2.0 ** -50, 1.0 + np.arange(1, 40) * 2.0 ** -26, 2.0 - 2.0 ** -np.arange(20, 53),
                        1.0 - 2.0 ** -np.arange(20, 53.0), 1.0 + rng.random(3000)])
    x = m * 2.0 ** rng.integers(-12, 12, len(m)) * rng.choice([-1, 1], len(m))
    x = np.concatenate([x, [0.0, 2.0 ** -20, -2.0 ** 20]])
    y = rng.uniform(0.5, 2.0, len(x)) * 2.0 ** rng.integers(-3, 4, len(x)) * rng.choice([-1, 1], len(x))
    text = "\n".join(f"{float(a).hex()} {float(b).hex()}" for a, b in zip(x, y))
    out = subprocess.run([exe], input=text, capture_output=True, text=True, check=True).stdout.split("\n")
    for a, b, line in zip(x, y, out):
        back, added, sh, sl, ph, pl, r3, r2, hi = map(float.fromhex, line.split())
        A, B = Fraction(float(a)), Fraction(float(b))
        # the conversion: 24 bits truncated, the other 29 rounded to 24
        assert abs(Fraction(back) - A) <= abs(A) / 2 ** 47
        assert hi == 0.0 or abs(Fraction(hi) - A) < abs(A) / 2 ** 23 and abs(hi) <= abs(float(a))
        # one DFMA's rounding (2^-53) on top of it
        assert abs(Fraction(added) - (A + B)) <= abs(A) / 2 ** 47 + abs(A + B) / 2 ** 53
        assert abs(Fraction(sh) + Fraction(sl) - (A + B)) <= max(abs(A), abs(B)) / 2 ** 45
        assert abs(Fraction(ph) + Fraction(pl) - A * B) <= abs(A * B) / 2 ** 44
        if a != 0.0:
            q = abs(A)
            # two roundings of 2^-48 and the conversion's, tripled by the power
            assert abs(Fraction(r2) * q - 1) <= Fraction(1, 2 ** 44)
            assert abs(Fraction(r3) ** 2 * q ** 3 - 1) <= Fraction(1, 2 ** 43)
