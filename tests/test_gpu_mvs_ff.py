"""GPU parity of the mixed-variable steps in FP64 and float pairs (csrc/mvs_ff.cuh,
csrc/kepler_ff.cuh) at the sizes, masses and step lengths where parts of a step change form."""
import math

import numpy as np
import pytest

import oracle as O
from gpu_util import TWO_PI, assert_parity, oracle_sensitivity, run_gpu, run_oracle
from test_gpu_hermite_ff import planets

pytestmark = pytest.mark.gpu


# dt in inner periods (1/20: the short drift; 1/5 and e 0.6: past a radian of eccentric anomaly,
# the FP64 drift); mass: the planets' factor (1e-6..1e-4 times it: at 500 the interactions and
# the reflex drift are FP64, at 1e-20 the planets are test particles)
@pytest.mark.parametrize("kind", [O.MVS_DH, O.MVS_JACOBI])
@pytest.mark.parametrize("n,n_sys,dt,e_max,mass", [(2, 33, 0.05, 0.1, 1), (3, 11, 0.05, 0.6, 1), (4, 41, 0.05, 0.1, 500),
                                                   (5, 7, 0.2, 0.1, 1), (7, 9, -0.05, 0.1, 10), (8, 5, 0.05, 0.1, 1e-20),
                                                   (11, 3, 0.01, 0.3, 20), (12, 13, 0.05, 0.05, 1), (15, 3, 0.05, 0.05, 1)])
def test_steps_across_the_forms(kind, n, n_sys, dt, e_max, mass):
    ens = planets(n_sys, n, e_max, seed=300 + n)
    m = ens["mass"].reshape(n_sys, n)
    m[:, 1:] *= mass
    ens["mass"] = m.ravel()
    h = dt * TWO_PI
    t_end = 100.4 * h  # a shortened last step
    ce = 0.0 if mass == 500 else 3.0
    o = run_oracle(ens, t_end, kind, h, ce=ce, ej=500.0)
    sens = oracle_sensitivity(ens, t_end, kind, h, ce=ce, ej=500.0)
    for single in (0, 1):
        g = run_gpu(ens, t_end, kind, h, ce=ce, ej=500.0, single_launch=single)
        assert_parity(ens, g, o, sens=sens, steps=101)
