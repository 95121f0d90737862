"""swarm_observe_rv through one launch per body count against a call per observation time."""
import numpy as np
import pytest

from gpu_util import TWO_PI
from paper_1208_1157_gb300 import ics

pytestmark = pytest.mark.gpu
DT = TWO_PI * 1e-3
LOS = (0.6, 0.0, 0.8)


# bins below 512 systems evaluate every state afresh, so the two are equal bit for bit; larger ones
# carry an evaluation over a step, which a new call does not (round-off of 60 steps)
@pytest.mark.parametrize("make,tol", [(lambda: ics.ragged(150, seed=51, n_max=15), 0.0), (lambda: ics.three_body(33, seed=52), 0.0),
                                      (lambda: ics.three_body(1500, seed=53), 1e-13)])
def test_one_launch_equals_a_call_per_time(make, tol):
    from paper_1208_1157_gb300 import swarm as S

    ens = make()
    # the present time, whole steps, shortened ones, the same time twice
    t_obs = np.array([0.0, 12.0, 24.0, 24.0, 30.5, 30.5, 31.0, 60.25]) * DT
    n = len(ens["n_body"])
    status = np.zeros(n, np.int32)
    status[::7] = S.EJECTED  # never run
    with S.Ensemble(ens) as e:
        e.set_stop(3.3, 100.0)
        e.set_state(status=status)
        rv = e.observe_rv(t_obs, S.HERMITE4, DT, LOS)
        got, steps = e.state(), e.stats()["system_steps"]
    with S.Ensemble(ens) as e:
        e.set_stop(3.3, 100.0)
        e.set_state(status=status)
        want = []
        for t in t_obs:
            e.integrate(t, S.HERMITE4, DT)
            want.append(e.rv(LOS))
        ref, ref_steps = e.state(), e.stats()["system_steps"]
    assert np.array_equal(got["status"], ref["status"]) and np.array_equal(got["time"], ref["time"]) and steps == ref_steps
    for a, b in ((rv, np.array(want)), (got["pos"], ref["pos"]), (got["vel"], ref["vel"])):
        assert np.abs(a - b).max() <= tol * np.abs(b).max()
