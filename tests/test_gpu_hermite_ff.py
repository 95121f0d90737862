"""GPU parity of the Hermite steps in FP64 and float pairs (csrc/hermite_ff.cuh) at the step
lengths, orbits and sizes where the kind of step changes."""
import math

import numpy as np
import pytest

import oracle as O
from gpu_util import TWO_PI, assert_parity, oracle_sensitivity, run_gpu, run_oracle
from paper_1208_1157_gb300 import ics

pytestmark = pytest.mark.gpu
DT = TWO_PI * 1e-3


def planets(n_sys, n, e_max, seed, flat=False):
    """Systems of a star and n - 1 planets on widely spaced orbits of eccentricity up to e_max."""
    rng = np.random.default_rng(seed)
    p = n - 1
    a = 1.7 ** np.arange(p)[None, :] * rng.uniform(0.97, 1.03, (n_sys, p))
    m = np.exp(rng.uniform(math.log(1e-6), math.log(1e-4), (n_sys, p)))
    ang = lambda: rng.uniform(0, TWO_PI, (n_sys, p))
    inc = np.zeros((n_sys, p)) if flat else rng.uniform(0, 0.3, (n_sys, p))
    x, v = ics.elements_to_cartesian(1.0 + m, a, rng.uniform(0, e_max, (n_sys, p)), inc, ang(), ang(), ang())
    z = np.zeros((n_sys, 1, 3))
    return {"n_body": np.full(n_sys, n, np.int32), "mass": np.concatenate([np.ones((n_sys, 1)), m], 1).ravel(),
            "pos": np.concatenate([z, x], 1).reshape(-1, 3), "vel": np.concatenate([z, v], 1).reshape(-1, 3)}


# dt in thousandths of the inner period: FP32 differences up to about 2.1, pairs up to about 10,
# FP64 steps above; e_max 0.6 makes one orbit pass through several of them
@pytest.mark.parametrize("mapping", [1, 2])
@pytest.mark.parametrize("n,n_sys,dt,e_max", [(5, 9, 1.0, 0.3), (6, 520, 1.0, 0.05), (8, 33, 2.1, 0.05), (9, 5, 6.0, 0.05),
                                              (15, 3, 1.0, 0.05), (14, 600, 1.0, 0.02), (7, 530, 25.0, 0.05), (2, 31, 1.0, 0.05), (3, 33, 1.0, 0.6), (3, 65, 2.1, 0.05), (3, 32, 6.0, 0.05),
                                              (3, 40, 25.0, 0.05), (4, 33, 1.0, 0.3), (4, 7, 9.5, 0.1)])
def test_fixed_steps_across_the_levels(mapping, n, n_sys, dt, e_max):
    if mapping == 1 and n > 4:
        pytest.skip("a system per lane: up to four bodies")
    ens = planets(n_sys, n, e_max, seed=100 + n_sys, flat=n == 2)
    t_end = 150.4 * dt * DT  # a shortened last step
    o = run_oracle(ens, t_end, O.HERMITE, dt * DT, ce=3.0, ej=100.0)
    sens = oracle_sensitivity(ens, t_end, O.HERMITE, dt * DT, ce=3.0, ej=100.0)
    g = run_gpu(ens, t_end, 1, dt * DT, mapping=mapping, ce=3.0, ej=100.0, single_launch=0)
    assert_parity(ens, g, o, sens=sens, steps=151)
    if n == 2:  # a flat system stays exactly flat
        assert np.all(g["pos"][:, 2] == 0.0) and np.all(g["vel"][:, 2] == 0.0)


@pytest.mark.parametrize("mapping", [1, 2])
@pytest.mark.parametrize("n,tau,e_max", [(2, 0.01, 0.1), (3, 0.01, 0.5), (3, 0.05, 0.1), (4, 0.2, 0.1), (9, 0.01, 0.3), (13, 0.02, 0.1)])
def test_adaptive_steps_across_the_levels(mapping, n, tau, e_max):
    if mapping == 1 and n > 4:
        pytest.skip("a system per lane: up to four bodies")
    ens = planets(37, n, e_max, seed=200 + n)
    o = run_oracle(ens, 1.5, O.HERMITE_ADAPTIVE, tau, ce=3.0, ej=100.0)
    sens = oracle_sensitivity(ens, 1.5, O.HERMITE_ADAPTIVE, tau, ce=3.0, ej=100.0)
    g = run_gpu(ens, 1.5, 4, tau, mapping=mapping, ce=3.0, ej=100.0, single_launch=0)
    assert_parity(ens, g, o, sens=sens, steps=1000)
