"""The adaptive step's length (Eq. 5) with planets light enough that body 0's own acceleration,
which has their mass, squares out of FP32's range: the times after 8 and 16 steps against the
oracle's.  The length is good to 2^-44 (6e-14), a sum of 16 of them to no less, and the orbits'
rounding moves it by less: bound 1e-12.  2^-38 of a step at 1e-17 and 2^-23 at 1e-19 before."""
import numpy as np
import pytest

import oracle as O
from gpu_util import run_gpu, run_oracle
from test_gpu_hermite_ff import planets

pytestmark = pytest.mark.gpu


# 1e-28: 2^-93, below which the terms are taken in FP64
@pytest.mark.parametrize("mapping,n,n_sys", [(1, 2, 33), (1, 3, 40), (1, 4, 33), (2, 2, 33), (2, 3, 40), (2, 3, 520), (2, 9, 21), (2, 18, 5)])
@pytest.mark.parametrize("mass", [1e-5, 1e-12, 1e-17, 1e-19, 1e-24, 1e-28])
def test_step_lengths(mapping, n, n_sys, mass):
    ens = planets(n_sys, n, 0.1, seed=60 + n)
    m = ens["mass"].reshape(n_sys, n)
    m[:, 1:] *= mass / 1e-5
    ens["mass"] = m.ravel()
    g = run_gpu(ens, 0.5, 4, 0.01, mapping=mapping, log_interval=8, log_cap=64, single_launch=0)
    o = run_oracle(ens, 0.5, O.HERMITE_ADAPTIVE, 0.01, log_interval=8, log_cap=64)
    for s in range(n_sys):
        a, b = g["logs"][s][:2], o["log"][s, :2]
        assert a.shape == b.shape and o["log_count"][s] >= 2
        np.testing.assert_allclose(a[:, 0], b[:, 0], rtol=1e-12)
