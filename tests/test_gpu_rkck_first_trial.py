"""Adaptive Cash-Karp from a first trial longer than the call: the first step is the whole call, at
any length that a double holds."""
import numpy as np
import pytest

from gpu_util import run_gpu
from test_gpu_hermite_ff import planets

pytestmark = pytest.mark.gpu


# 2^385 and 2^300 are 0 and 2^44 where only eight bits of the exponent are looked at
@pytest.mark.parametrize("n", [2, 3, 4, 9])
@pytest.mark.parametrize("dt", [2.0 ** 128, 2.0 ** 300, 2.0 ** 385, 2.0 ** 1000])
def test_a_first_trial_of_any_length(n, dt):
    ens = planets(21, n, 0.05, seed=40 + n)
    a = run_gpu(ens, 0.3, 6, dt, single_launch=0)
    b = run_gpu(ens, 0.3, 6, 1.0, single_launch=0)
    assert np.all(a["status"] == 1)
    for k in ("pos", "vel", "time", "status"):
        assert np.array_equal(a[k], b[k]), k
