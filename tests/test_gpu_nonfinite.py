"""States that are not finite, put in through the device path (swarm_set_state_dev does not look
at the values): the system stops at its first step, the others of its bin take no notice."""
import math

import numpy as np
import pytest

from gpu_util import TWO_PI
from paper_1208_1157_gb300 import ics
from test_gpu_hermite_ff import planets

pytestmark = pytest.mark.gpu
DT = TWO_PI * 1e-3
STEPS = 5
HUGE = 1e80  # finite, and outside FP32's range with an exponent that wraps into it
VALUES = [math.nan, -math.nan, math.inf, -math.inf, HUGE]


def poisoned(ens, n, adaptive):
    """ens with one component of every third system replaced: a value of VALUES in the position or
    the velocity of the star or the last planet.  Returns it, those systems and their values."""
    values = VALUES[:4] if adaptive else VALUES
    pos, vel = ens["pos"].reshape(-1, n, 3).copy(), ens["vel"].reshape(-1, n, 3).copy()
    which = np.arange(0, len(pos), 3)
    put = []
    for k, s in enumerate(which):
        val = values[k % len(values)]
        where = (k // len(values)) % 12
        (pos, vel)[where // 6][s, (0, n - 1)[where // 3 % 2], where % 3] = val
        put.append(val)
    return pos.reshape(-1, 3), vel.reshape(-1, 3), which, np.array(put)


def run_dev(ens, pos, vel, t_end, integrator, dt, mapping, single):
    import torch
    from paper_1208_1157_gb300 import swarm as S

    with S.Ensemble(ens) as e:
        e.set_option(S.OPT_MAPPING, mapping)
        e.set_option(S.OPT_SINGLE_LAUNCH, single)
        e.set_stop(3.0, 1e5)
        dev = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")
        p, v = dev(pos), dev(vel)
        torch.cuda.synchronize()
        e.set_state_dev(p, v, None, None)
        e.integrate(t_end, integrator, dt)
        return e.state()


# (integrator, mapping, bodies, systems, single launch): Hermite a system and a body per lane, below
# and above the 512 systems from which an evaluation is carried, one system per warp, and from the
# shared launch; Cash-Karp a system per lane, a body per lane and one system per warp
FIXED = [(1, 1, 3, 180, 0), (1, 1, 4, 180, 1), (1, 2, 2, 180, 0), (1, 2, 3, 180, 0), (1, 2, 8, 180, 0), (1, 2, 3, 540, 0),
         (1, 2, 8, 540, 0), (1, 2, 15, 540, 1), (1, 2, 18, 180, 0), (5, 2, 2, 180, 0), (5, 2, 3, 180, 0), (5, 2, 5, 180, 0),
         (5, 2, 13, 180, 0), (5, 2, 18, 180, 0), (2, 2, 5, 180, 0), (3, 2, 5, 180, 0)]
ADAPTIVE = [(4, 1, 3, 144, 0), (4, 2, 3, 144, 0), (4, 2, 8, 540, 0), (4, 2, 18, 144, 0), (6, 2, 3, 144, 0), (6, 2, 5, 144, 0)]


def check(integrator, mapping, n, n_sys, single):
    adaptive = integrator in (4, 6)
    dt = {1: DT, 5: DT, 2: 20 * DT, 3: 20 * DT, 4: 0.01, 6: 10 * DT}[integrator]
    t_end = STEPS * (dt if not adaptive else 4 * DT)
    ens = planets(n_sys, n, 0.05, seed=900 + n, flat=n == 2)
    pos, vel, which, put = poisoned(ens, n, adaptive)
    if single:  # the shared launch wants a second body count
        more = planets(9, 5, 0.05, seed=950)
        ens = ics.concat(ens, more)
        pos, vel = np.concatenate([pos, more["pos"]]), np.concatenate([vel, more["vel"]])
    good = run_dev(ens, ens["pos"], ens["vel"], t_end, integrator, dt, mapping, single)
    got = run_dev(ens, pos, vel, t_end, integrator, dt, mapping, single)
    stopped, huge = which[put != HUGE], which[put == HUGE]
    assert np.all(got["status"][stopped] == 5), got["status"][stopped]
    if adaptive:  # a step's length is that of no other system
        assert np.all(got["time"][stopped] < t_end)
    else:
        assert np.all(got["time"][stopped] <= dt)
        # wholly in FP64: ejected at once, or in the step where its square leaves FP64's range
        assert np.all(np.isin(got["status"][huge], (3, 4, 5))), got["status"][huge]
        assert np.all(got["time"][huge] <= dt)
    rest = np.setdiff1d(np.arange(n_sys), which)
    for k in ("pos", "vel"):
        assert np.array_equal(got[k][:n_sys * n].reshape(-1, n, 3)[rest], good[k][:n_sys * n].reshape(-1, n, 3)[rest]), k
    assert np.array_equal(got["time"][rest], good["time"][rest]) and np.array_equal(got["status"][rest], good["status"][rest])


@pytest.mark.parametrize("integrator,mapping,n,n_sys,single", FIXED)
def test_fixed_steps(integrator, mapping, n, n_sys, single):
    check(integrator, mapping, n, n_sys, single)


@pytest.mark.parametrize("integrator,mapping,n,n_sys,single", ADAPTIVE)
def test_adaptive_steps(integrator, mapping, n, n_sys, single):
    check(integrator, mapping, n, n_sys, single)
