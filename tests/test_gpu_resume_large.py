"""Hermite bins of 512 systems and more carry an evaluation from step to step: a call in chunks, or
resumed from a checkpoint, agrees with the whole one to rounding, not bit for bit.

Bound: at each of the at most 40 boundaries the state's evaluation differs by its own rounding
(2^-46 of a step's dv, 2^-53 of v and less), as FP64's at every step; over 200 steps of 1/1000
orbit on well-spaced orbits that moves a state by about 200 x 2^-53 x (a radian's growth), below
1e-13 of its size."""
import numpy as np
import pytest

from gpu_util import TWO_PI, per_system_errors, run_gpu
from test_gpu_hermite_ff import planets

pytestmark = pytest.mark.gpu
DT = TWO_PI * 1e-3


@pytest.mark.parametrize("n,n_sys", [(3, 520), (3, 2000), (8, 700), (15, 512)])
def test_chunked_and_resumed_agree_to_rounding(n, n_sys, tmp_path):
    from paper_1208_1157_gb300 import swarm as S

    ens = planets(n_sys, n, 0.05, seed=30 + n)
    t_end = 200 * DT
    whole = run_gpu(ens, t_end, 1, DT, mapping=2, single_launch=0)
    parts = run_gpu(ens, t_end, 1, DT, mapping=2, single_launch=0, steps_per_launch=5)
    with S.Ensemble(ens) as e:
        e.set_option(S.OPT_MAPPING, S.MAP_BODY_PER_LANE)
        e.integrate(77 * DT, S.HERMITE4, DT)
        S.save_checkpoint(e, str(tmp_path / "ck.npz"))
    with S.resume(S.load_checkpoint(str(tmp_path / "ck.npz"))) as e:
        e.set_option(S.OPT_MAPPING, S.MAP_BODY_PER_LANE)
        e.integrate(t_end, S.HERMITE4, DT)
        resumed = e.state()
    for got in (parts, resumed):
        assert np.array_equal(got["status"], whole["status"])
        ex, ev = per_system_errors(ens, got, whole)
        assert max(ex.max(), ev.max()) < 1e-13, (ex.max(), ev.max())
