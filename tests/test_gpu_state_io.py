"""State in and out of ensembles whose bins go together in one launch, alone, or some of each way."""
import numpy as np
import pytest

from paper_1208_1157_gb300 import ics

pytestmark = pytest.mark.gpu


def part(n_sys, n, rng):
    return {"n_body": np.full(n_sys, n, np.int32), "mass": np.exp(rng.uniform(-9, 0, n_sys * n)),
            "pos": rng.normal(size=(n_sys * n, 3)), "vel": rng.normal(size=(n_sys * n, 3))}


@pytest.mark.parametrize("scattered", [False, True])
@pytest.mark.parametrize("bins", [[(40000, 3)], [(16383, 3), (16384, 4)], [(20000, 2), (33, 5), (1, 32)], [(32768, 6), (32767, 5)],
                                  [(17000, 3), (33000, 9), (7, 16), (500, 4)], [(5, n) for n in range(2, 33)]])
def test_round_trip(bins, scattered):
    import torch
    from paper_1208_1157_gb300 import swarm as S

    rng = np.random.default_rng(5)
    ens = ics.concat(*[part(s, n, rng) for s, n in bins]) if len(bins) > 1 else part(*bins[0], rng)
    if scattered:
        ens = ics.subset(ens, rng.permutation(len(ens["n_body"])))
    n_sys, n_rows = len(ens["n_body"]), len(ens["mass"])
    with S.Ensemble(ens) as e:
        got = e.state()
        assert np.array_equal(got["pos"], ens["pos"]) and np.array_equal(got["vel"], ens["vel"])
        energy, _ = e.diagnostics()  # takes the masses
        first = np.concatenate([[0], np.cumsum(ens["n_body"])])
        s = n_sys // 2
        m, x, v = (ens[k][first[s]:first[s + 1]] for k in ("mass", "pos", "vel"))
        d = np.linalg.norm(x[:, None] - x[None], axis=-1)
        i, j = np.triu_indices(len(m), 1)
        want = 0.5 * np.sum(m * np.sum(v * v, 1)) - np.sum(m[i] * m[j] / d[i, j])
        assert abs(energy[s] - want) < 1e-12 * (0.5 * np.sum(m * np.sum(v * v, 1)) + np.sum(m[i] * m[j] / d[i, j]))
        pos, vel = rng.normal(size=(n_rows, 3)), rng.normal(size=(n_rows, 3))
        time, status = rng.normal(size=n_sys), rng.integers(0, 5, n_sys).astype(np.int32)
        dev = lambda a: torch.as_tensor(a, device="cuda")
        a = [dev(pos), dev(vel), dev(time), dev(status)]
        b = [torch.zeros_like(t) for t in a]
        torch.cuda.synchronize()
        e.set_state_dev(*a)
        e.state_dev(*b)
        e.synchronize()
        assert all(torch.equal(x, y) for x, y in zip(a, b))
        e.set_state_dev(a[1], None, None, None)  # positions alone
        e.state_dev(b[0], b[1], b[2], b[3])
        e.synchronize()
        assert torch.equal(b[0], a[1]) and torch.equal(b[1], a[1]) and torch.equal(b[2], a[2])
