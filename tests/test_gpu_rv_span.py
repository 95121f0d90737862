"""The limit of 2e9 steps holds for each interval of swarm_observe_rv, not for their sum."""
import numpy as np
import pytest

from gpu_util import TWO_PI
from paper_1208_1157_gb300 import ics

pytestmark = pytest.mark.gpu
DT = TWO_PI * 1e-3
LOS = (0.6, 0.0, 0.8)


@pytest.mark.parametrize("integrator", [1, 3])
def test_the_limit_is_an_intervals(integrator):
    from paper_1208_1157_gb300 import swarm as S

    ens = ics.ragged(20, seed=54, n_max=6)
    with S.Ensemble(ens) as e:
        e.set_state(status=np.full(20, S.EJECTED, np.int32))  # no system takes a step
        here = e.rv(LOS)
        rv = e.observe_rv(np.array([1.5e9, 3e9, 4.5e9]) * DT, integrator, DT, LOS)
        assert np.array_equal(rv, np.stack([here] * 3))
        with pytest.raises(S.SwarmError):  # one interval of 2.5e9
            e.observe_rv(np.array([4.6e9, 7.1e9]) * DT, integrator, DT, LOS)
