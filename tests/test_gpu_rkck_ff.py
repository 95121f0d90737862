"""GPU parity of the Cash-Karp steps in FP64 and float pairs (csrc/rkck_ff.cuh) at the step
lengths, orbits and sizes where a step changes form."""
import pytest

import oracle as O
from gpu_util import TWO_PI, assert_parity, oracle_sensitivity, run_gpu, run_oracle
from test_gpu_hermite_ff import planets

pytestmark = pytest.mark.gpu


# dt in thousandths of the inner period: pairs up to about 20, FP64 steps above; e_max 0.7 makes
# one orbit pass through both
@pytest.mark.parametrize("n,n_sys,dt,e_max", [(2, 33, 1.0, 0.1), (3, 65, 1.0, 0.05), (3, 40, 15.0, 0.7), (3, 7, 40.0, 0.05),
                                              (4, 9, 1.0, 0.05), (5, 33, 15.0, 0.5), (8, 5, 40.0, 0.05), (11, 13, 1.0, 0.05),
                                              (15, 3, 10.0, 0.05)])
def test_fixed_steps_across_the_forms(n, n_sys, dt, e_max):
    ens = planets(n_sys, n, e_max, seed=400 + n)
    h = dt * 1e-3 * TWO_PI
    t_end = 100.4 * h  # a shortened last step
    o = run_oracle(ens, t_end, O.RKCK, h, ce=3.0, ej=500.0)
    sens = oracle_sensitivity(ens, t_end, O.RKCK, h, ce=3.0, ej=500.0)
    g = run_gpu(ens, t_end, 5, h, ce=3.0, ej=500.0, single_launch=0)
    assert_parity(ens, g, o, sens=sens, steps=101)


@pytest.mark.parametrize("n,n_sys,eps,e_max", [(2, 33, 1e-12, 0.1), (3, 70, 1e-12, 0.6), (3, 20, 1e-6, 0.1), (4, 9, 1e-12, 0.3),
                                               (9, 5, 1e-9, 0.1), (13, 3, 1e-12, 0.1)])
def test_adaptive_steps_across_the_forms(n, n_sys, eps, e_max):
    ens = planets(n_sys, n, e_max, seed=500 + n)
    t_end, h = 2.5, 0.02
    o = run_oracle(ens, t_end, O.RKCK_ADAPTIVE, h, ce=3.0, ej=500.0, rk_eps=eps)
    sens = oracle_sensitivity(ens, t_end, O.RKCK_ADAPTIVE, h, ce=3.0, ej=500.0, rk_eps=eps)
    g = run_gpu(ens, t_end, 6, h, ce=3.0, ej=500.0, rk_eps=eps, single_launch=0)
    assert_parity(ens, g, o, sens=sens, steps=1000, stop_time_rtol=1e-9)
