"""The printed corrector in bins of five bodies and more: the kernel packed across the CTA (bins that
fill a wave of it) against the warp ring, and against the oracle."""
import numpy as np
import pytest

import oracle as O
from gpu_util import TWO_PI, assert_parity, block_ring_wave
from paper_1208_1157_gb300 import ics

pytestmark = pytest.mark.gpu
DT = TWO_PI * 1e-3


def run(ens, steps, single):
    from paper_1208_1157_gb300 import swarm as S

    with S.Ensemble(ens) as e:
        e.set_option(S.OPT_MAPPING, S.MAP_BODY_PER_LANE)
        e.set_option(S.OPT_CORRECTOR, 1)
        e.set_option(S.OPT_SINGLE_LAUNCH, single)
        e.set_option(S.OPT_LOG_CAPACITY, 4)
        e.set_option(S.OPT_LOG_INTERVAL, 20)
        e.set_stop(3.0, 100.0)
        e.integrate(steps * DT, S.HERMITE4, DT)
        out = e.state()
        out["logs"] = [e.log(s) for s in range(e.n_sys)]
    return out


@pytest.mark.parametrize("ns", [(5, 6), (7, 9), (11, 12), (13, 14), (15, 10)])
def test_packed_equals_warp_ring_and_oracle(ns):
    import torch

    sms = torch.cuda.get_device_properties(0).multi_processor_count
    ens = ics.concat(*[ics.request_ensemble({"n_sys": block_ring_wave(n, sms) + 37, "n": n, "seed": 800 + n}) for n in ns])
    a = run(ens, 60.5, 0)
    b = run(ens, 60.5, 1)  # the shared launch: the warp ring
    for k in ("pos", "vel", "time", "status"):
        assert np.array_equal(a[k], b[k]), k
    assert all(np.array_equal(x, y) for x, y in zip(a["logs"], b["logs"]))
    idx = np.sort(np.random.default_rng(4).choice(len(ens["n_body"]), 24, replace=False))
    sub = ics.subset(ens, idx)
    offs = np.concatenate([[0], np.cumsum(ens["n_body"])])
    rows = np.concatenate([np.arange(offs[s], offs[s + 1]) for s in idx])
    o = O.integrate(sub, 60.5 * DT, DT, O.HERMITE, ce_factor=3.0, eject_radius=100.0, corr_form=O.CORR_PRINTED)
    assert_parity(sub, {"pos": a["pos"][rows], "vel": a["vel"][rows], "time": a["time"][idx], "status": a["status"][idx]}, o, steps=61)
