"""Ensembles in units that the pairs of FP32 numbers do not hold (kilometres and km^3/s^2, masses of
2^44, distances of 2^-24), which are stepped in FP64, and adaptive bins of 512 systems and more,
which carry an evaluation: against the oracle."""
import numpy as np
import pytest

import oracle as O
from gpu_util import TWO_PI, assert_parity, oracle_sensitivity, run_gpu, run_oracle
from test_gpu_hermite_ff import planets

pytestmark = pytest.mark.gpu
DT = TWO_PI * 1e-3


# integrator, mapping, bodies, step in thousandths of the inner period, steps
RUNS = [(1, 1, 3, 1.0, 60.4), (1, 2, 2, 1.0, 60.4), (1, 2, 3, 1.0, 60.4), (1, 2, 8, 1.0, 60.4), (1, 2, 18, 1.0, 30.4),
        (5, 2, 3, 1.0, 60.4), (5, 2, 4, 1.0, 60.4), (5, 2, 9, 1.0, 60.4), (6, 2, 3, 10.0, 20.0), (6, 2, 6, 10.0, 20.0),
        (2, 2, 3, 50.0, 40.4), (2, 2, 9, 50.0, 40.4), (3, 2, 4, 50.0, 40.4), (3, 2, 9, 50.0, 40.4)]


@pytest.mark.parametrize("length,mass", [(2.0 ** 27, 2.0 ** 37), (1.0, 2.0 ** 44), (2.0 ** -24, 1.0)])
@pytest.mark.parametrize("integrator,mapping,n,dt,steps", RUNS)
def test_other_units(length, mass, integrator, mapping, n, dt, steps):
    ens = planets(23, n, 0.05, seed=80 + n, flat=n == 2)
    ens["mass"], ens["pos"], ens["vel"] = ens["mass"] * mass, ens["pos"] * length, ens["vel"] * np.sqrt(mass / length)
    h = dt * DT * np.sqrt(length ** 3 / mass)
    kw = dict(ce=3.0, ej=1e5 * length)
    o = run_oracle(ens, steps * h, integrator, h, **kw)
    g = run_gpu(ens, steps * h, integrator, h, mapping=mapping, single_launch=0, **kw)
    assert_parity(ens, g, o, sens=oracle_sensitivity(ens, steps * h, integrator, h, **kw), stop_time_rtol=1e-9 if integrator == 6 else None)


@pytest.mark.parametrize("n,n_sys,tau,e_max", [(2, 520, 0.01, 0.1), (3, 530, 0.01, 0.3), (3, 600, 0.05, 0.1), (9, 512, 0.01, 0.1), (18, 514, 0.01, 0.02)])
def test_adaptive_bins_that_carry(n, n_sys, tau, e_max):
    ens = planets(n_sys, n, e_max, seed=90 + n)
    o = run_oracle(ens, 1.0, O.HERMITE_ADAPTIVE, tau, ce=3.0, ej=1e5)
    g = run_gpu(ens, 1.0, 4, tau, mapping=2, ce=3.0, ej=1e5, single_launch=0)
    assert_parity(ens, g, o, sens=oracle_sensitivity(ens, 1.0, O.HERMITE_ADAPTIVE, tau, ce=3.0, ej=1e5), steps=1000)
