"""Body per lane, states that go between FP64 steps and pairs: a step's form follows from the state
alone (bins below 512 systems), so a call in chunks repeats the whole one bit for bit, and the
states are the oracle's."""
import numpy as np
import pytest

import oracle as O
from gpu_util import TWO_PI, assert_parity, oracle_sensitivity, run_gpu, run_oracle
from test_gpu_hermite_ff import planets

pytestmark = pytest.mark.gpu
DT = TWO_PI * 1e-3


# dt in thousandths of the inner period; eccentric orbits cross the limit (about 10) within one
# orbit, the last case is FP64 throughout
@pytest.mark.parametrize("n,n_sys,dt,e_max", [(2, 31, 8.0, 0.5), (3, 100, 8.0, 0.5), (6, 33, 9.8, 0.02), (8, 65, 6.0, 0.6),
                                              (15, 9, 8.0, 0.4), (18, 7, 8.0, 0.4), (9, 40, 25.0, 0.05)])
def test_chunks_repeat_the_whole_call(n, n_sys, dt, e_max):
    ens = planets(n_sys, n, e_max, seed=70 + n, flat=n == 2)
    t_end = 90 * dt * DT  # whole steps: a shortened last one takes its length from the chunk's own times
    whole = run_gpu(ens, t_end, 1, dt * DT, mapping=2, ce=3.0, ej=1e5, single_launch=0)
    parts = run_gpu(ens, t_end, 1, dt * DT, mapping=2, ce=3.0, ej=1e5, single_launch=0, steps_per_launch=7)
    for k in ("pos", "vel", "status"):
        assert np.array_equal(whole[k], parts[k]), k
    o = run_oracle(ens, t_end, O.HERMITE, dt * DT, ce=3.0, ej=1e5)
    assert_parity(ens, whole, o, sens=oracle_sensitivity(ens, t_end, O.HERMITE, dt * DT, ce=3.0, ej=1e5), steps=90)
