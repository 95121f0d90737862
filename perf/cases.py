"""Performance cases: what users of the library have it do, through its public entry points.

Each case is one pass of a user's program over an ensemble it holds: put the state in, advance
it, take the state (or the observable) out.  Sizes, step lengths and distributions are those of
the package's own workloads (three-body, ragged, compact and wide planetary ensembles).
"""
import math

import numpy as np
import torch

from paper_1208_1157_gb300 import server as SV
from paper_1208_1157_gb300 import swarm as S
from paper_1208_1157_gb300 import tune

TWO_PI = 2.0 * math.pi
DT = 1e-3 * TWO_PI       # Hermite and Runge-Kutta: a thousandth of the inner period
DT_MVS = TWO_PI / 20     # mixed-variable symplectic: a twentieth of it
CE, EJECT = 3.0, 100.0   # stop conditions: 3 mutual Hill radii, 100 AU
TAU, EPS = 0.01, 1e-12   # adaptive Hermite's step factor, adaptive Runge-Kutta's tolerance
LOS = (0.0, 0.6, 0.8)

# kind -> (smallest, largest) number of systems that draw() takes, (fewest, most) steps
RANGES = {
    "rv": ((33, 1500), (6, 24)),
    "hermite3": ((64, 131072), (100, 400)),
    "hermite_ragged": ((100, 65536), (20, 100)),
    "hermite_wide": ((50, 2500), (20, 60)),
    "hermite_adaptive3": ((500, 65536), (100, 250)),
    "mvs_jacobi": ((200, 16384), (100, 500)),
    "mvs_dh_ragged": ((200, 9000), (50, 300)),
    "rkck_ragged": ((100, 20000), (20, 60)),
    "rkck_adaptive3": ((500, 30000), (250, 1000)),
    "serve": ((6, 24), (60, 240)),
}


def listed():
    return [
        # one likelihood evaluation of a radial-velocity fit: a few hundred candidate systems from the
        # host, advanced through 12 observation times, the star's velocities back on the host
        {"name": "rv_fit_257x3", "kind": "rv", "systems": 257, "steps": 12},
        # a small ensemble, where the latency of a step counts
        {"name": "hermite_1024x3", "kind": "hermite3", "systems": 1024, "steps": 400},
        # the paper-shaped ensemble with its stop conditions
        {"name": "hermite_131072x3", "kind": "hermite3", "systems": 131072, "steps": 400},
        # ensembles of mixed body counts (3..15): an odd small one and the full one
        {"name": "hermite_ragged_777", "kind": "hermite_ragged", "systems": 777, "steps": 100},
        {"name": "hermite_ragged_65536", "kind": "hermite_ragged", "systems": 65536, "steps": 100},
        # many-planet systems (16..32 bodies)
        {"name": "hermite_wide_2048", "kind": "hermite_wide", "systems": 2048, "steps": 50},
        # the adaptive step over a fraction of an inner period
        {"name": "hermite_adaptive_30011x3", "kind": "hermite_adaptive3", "systems": 30011, "steps": 250},
        # long-term stability runs of compact systems: Wisdom-Holman map, both coordinate choices
        {"name": "mvs_jacobi_16384x8", "kind": "mvs_jacobi", "systems": 16384, "steps": 500},
        {"name": "mvs_dh_ragged_3001", "kind": "mvs_dh_ragged", "systems": 3001, "steps": 300},
        # Runge-Kutta with fixed steps on mixed body counts, and adaptive on three bodies
        {"name": "rkck_ragged_9001", "kind": "rkck_ragged", "systems": 9001, "steps": 60},
        {"name": "rkck_adaptive_20000x3", "kind": "rkck_adaptive3", "systems": 20000, "steps": 1000},
        # the serving loop: requests of different sizes, body counts and integrators until all are done
        {"name": "serve_24_requests", "kind": "serve", "systems": 24, "steps": 240},
    ]


def draw(rng):
    kind = rng.choice(sorted(RANGES))
    (lo, hi), (s0, s1) = RANGES[kind]
    n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    return {"kind": kind, "systems": min(hi, max(lo, n | rng.randrange(2))), "steps": rng.randint(s0, s1)}


# ---------------------------------------------------------------------------------------- inputs
def _cartesian(mu, a, e, inc, node, peri, E):
    b = a * np.sqrt(1 - e * e)
    w = np.sqrt(mu / a ** 3) / (1 - e * np.cos(E))
    xo, yo, vx, vy = a * (np.cos(E) - e), b * np.sin(E), -a * np.sin(E) * w, b * np.cos(E) * w
    cO, sO, cw, sw, ci, si = np.cos(node), np.sin(node), np.cos(peri), np.sin(peri), np.cos(inc), np.sin(inc)
    p = np.stack([cO * cw - sO * sw * ci, sO * cw + cO * sw * ci, sw * si], -1)
    q = np.stack([-cO * sw - sO * cw * ci, -sO * sw + cO * cw * ci, cw * si], -1)
    return xo[..., None] * p + yo[..., None] * q, vx[..., None] * p + vy[..., None] * q


def _systems(n_body, rng, e_max, m_lo, m_hi, three=False, a_cap=None):
    """Seeded planetary systems: a star of one solar mass and n - 1 planets, barycentric."""
    n_body = np.asarray(n_body, dtype=np.int32)
    s, p = len(n_body), int(n_body.max()) - 1
    live = np.arange(p)[None, :] < (n_body - 1)[:, None]

    def spaced(k):
        m = np.exp(rng.uniform(math.log(m_lo), math.log(m_hi), (k, p)))
        a = np.ones((k, p))
        if three:
            a[:, 1] = rng.uniform(1.6, 3.0, k)
            return m, a
        for j in range(1, p):
            x = 0.5 * rng.uniform(3.0, 8.0, k) * np.cbrt((m[:, j - 1] + m[:, j]) / 3.0)
            a[:, j] = a[:, j - 1] * (1 + x) / (1 - x)
        return m, a

    m, a = spaced(s)
    while a_cap is not None and (far := np.nonzero(a[:, -1] > a_cap)[0]).size:
        m[far], a[far] = spaced(far.size)
    e, inc = rng.uniform(0, e_max, (s, p)), rng.uniform(0, 0.01, (s, p))
    node, peri, E = (rng.uniform(0, TWO_PI, (s, p)) for _ in range(3))
    x, v = _cartesian(1.0 + m, a, e, inc, node, peri, E)
    mass = np.concatenate([np.ones((s, 1)), np.where(live, m, 0.0)], 1)
    zero = np.zeros((s, 1, 3))
    x, v = np.concatenate([zero, x], 1), np.concatenate([zero, v], 1)
    total = mass.sum(1)[:, None, None]
    x = x - (mass[..., None] * x).sum(1, keepdims=True) / total
    v = v - (mass[..., None] * v).sum(1, keepdims=True) / total
    keep = np.concatenate([np.ones((s, 1), bool), live], 1)
    return {"n_body": n_body, "mass": mass[keep], "pos": x[keep], "vel": v[keep]}


def _ensemble(case, seed):
    rng, kind, s = np.random.default_rng([seed, 7]), case["kind"], case["systems"]
    counts = np.random.default_rng(s)  # the body counts are the case's, the systems the seed's
    if kind == "mvs_jacobi":
        return _systems(np.full(s, 8), rng, 0.1, 1e-5, 1e-3, a_cap=45.0)
    if kind == "hermite_wide":
        return _systems(counts.integers(16, 33, s), rng, 0.1, 1e-7, 1e-5)
    if kind in ("hermite_ragged", "mvs_dh_ragged", "rkck_ragged"):
        return _systems(counts.integers(3, 16, s), rng, 0.1, 1e-5, 1e-3)
    return _systems(np.full(s, 3), rng, 0.05, 1e-5, 1e-3, three=True)


def _requests(case, seed):
    """Requests of 1..512 systems (log-uniform), 3..15 bodies, alternately Hermite and MVS; end times
    from a quarter of `steps` to all of them."""
    rng, shape, got = np.random.default_rng([seed, 8]), np.random.default_rng(case["steps"]), []
    for k in range(case["systems"]):
        s, n = int(round(math.exp(shape.uniform(0.0, math.log(512.0))))), int(shape.integers(3, 16))
        steps = int(shape.integers(max(1, case["steps"] // 4), case["steps"] + 1))
        integ, dt = (S.HERMITE4, DT) if k % 2 == 0 else (S.MVS_DH, DT_MVS)
        got.append((_systems(np.full(s, n), rng, 0.1, 1e-5, 1e-3), steps * dt, integ))
    return got


def _plan(case):
    """(integrator, dt or tau or first trial, end time)"""
    kind, steps = case["kind"], case["steps"]
    if kind.startswith("mvs"):
        return (S.MVS_JACOBI if kind == "mvs_jacobi" else S.MVS_DH), DT_MVS, steps * DT_MVS
    if kind == "hermite_adaptive3":
        return S.HERMITE4_ADAPTIVE, TAU, steps * DT
    if kind == "rkck_adaptive3":
        return S.RKCK_ADAPTIVE, 10 * DT, steps * DT
    return (S.RKCK if kind == "rkck_ragged" else S.HERMITE4), DT, steps * DT


def prepare(case, seed):
    S.tuner_load(tune.DEFAULT_PATH)
    if case["kind"] == "serve":
        return {"kind": "serve", "requests": _requests(case, seed),
                "server": SV.Server(slots_per_pool=1024, quantum_steps=60, hermite_dt=DT, mvs_dt=DT_MVS,
                                    ce_hill_factor=CE, eject_radius=EJECT)}
    ics = _ensemble(case, seed)
    e = S.Ensemble(ics)
    integ, dt, t_end = _plan(case)
    s, b = e.n_sys, e.n_bodies
    state = {"kind": case["kind"], "ens": e, "integ": integ, "dt": dt, "t_end": t_end, "ics": ics}
    if case["kind"] == "rv":
        state |= {"t_obs": DT * case["steps"] * np.arange(1, 13), "time": np.zeros(s), "status": np.zeros(s, np.int32)}
        return state
    e.set_stop(CE, EJECT)
    e.set_tolerance(EPS)
    dev = lambda a, t: torch.as_tensor(a, dtype=t, device="cuda")
    state |= {"pos": dev(ics["pos"], torch.float64), "vel": dev(ics["vel"], torch.float64),
              "time": torch.zeros(s, dtype=torch.float64, device="cuda"),
              "status": torch.zeros(s, dtype=torch.int32, device="cuda"), "bodies": b, "systems": s}
    return state


def run(state):
    if state["kind"] == "serve":
        sv = state["server"]
        ids = [sv.submit(ens, t_end, integ) for ens, t_end, integ in state["requests"]]
        done = 0
        while done < len(ids):
            done += sv.step()
        out = {}
        for k, (rid, (ens, _, _)) in enumerate(zip(ids, state["requests"])):
            got = sv.poll(rid, len(ens["n_body"]), int(ens["n_body"][0]))[1]
            out["r%02d" % k] = np.concatenate([got["pos"].ravel(), got["vel"].ravel(), got["time"]])
            sv.release(rid)
        return out
    e = state["ens"]
    if state["kind"] == "rv":
        e.set_state(state["ics"]["pos"], state["ics"]["vel"], state["time"], state["status"])
        return {"rv": e.observe_rv(state["t_obs"], state["integ"], state["dt"], LOS)}
    e.set_state_dev(state["pos"], state["vel"], state["time"], state["status"])
    e.integrate(state["t_end"], state["integ"], state["dt"], sync=False)
    new = lambda *d: torch.empty(d, dtype=torch.float64, device="cuda")
    out = {"pos": new(state["bodies"], 3), "vel": new(state["bodies"], 3), "time": new(state["systems"]),
           "status": torch.empty(state["systems"], dtype=torch.int32, device="cuda")}
    e.state_dev(out["pos"], out["vel"], out["time"], out["status"])
    return out


# ---------------------------------------------------------------------------------------- work
def _flops_per_step(kind, n, integ=None):
    pairs = n * (n - 1) / 2
    if kind.startswith("hermite") or kind == "rv" or integ == S.HERMITE4:
        return 3 * pairs * 58 + 3 * n * 34
    if kind.startswith("rkck"):
        return 6 * pairs * 25 + 3 * n * 54
    return 25 * pairs + (n - 1) * 100 + 6 * n


def work(case):
    kind, s, steps = case["kind"], case["systems"], case["steps"]
    if kind == "serve":
        sys_mean = 511.0 / math.log(512.0)  # mean of a log-uniform 1..512
        per = [(sum(_flops_per_step("", n, i) for n in range(3, 16)) / 13) for i in (S.HERMITE4, S.MVS_DH)]
        return {"bytes": s * sys_mean * 9 * 104.0, "flops": s * sys_mean * 0.625 * steps * sum(per) / 2}
    ns = range(16, 33) if kind == "hermite_wide" else range(3, 16) if "ragged" in kind else [8] if kind == "mvs_jacobi" else [3]
    flops = sum(_flops_per_step(kind, n) for n in ns) / len(ns)
    bodies = sum(ns) / len(ns)
    if kind == "rv":
        return {"bytes": s * (3 * 56.0 + 12 * 8), "flops": 12.0 * steps * s * flops}
    # adaptive: about 1.4 (Eq. 5) and 0.1 (error control at 1e-12) steps per dt of the fixed-step workloads
    steps *= {"hermite_adaptive3": 1.4, "rkck_adaptive3": 0.1}.get(kind, 1.0)
    return {"bytes": s * (bodies * 104.0 + 24), "flops": s * steps * flops}


# ---------------------------------------------------------------------------------------- in plain 64 bits
def _accjerk(m, x, v):
    d, u = x[:, None] - x[:, :, None], v[:, None] - v[:, :, None]
    r2 = (d * d).sum(-1)
    r2 = r2 + torch.eye(x.shape[1], dtype=x.dtype, device=x.device)
    s = m[:, None] / (r2 * r2.sqrt())
    q = 3 * (d * u).sum(-1) / r2
    return (s[..., None] * d).sum(2), (s[..., None] * (u - q[..., None] * d)).sum(2)


def _acc(m, x, star=True):
    d = x[:, None] - x[:, :, None]
    r2 = (d * d).sum(-1) + torch.eye(x.shape[1], dtype=x.dtype, device=x.device)
    s = m[:, None] / (r2 * r2.sqrt())
    if not star:
        s = torch.cat([torch.zeros_like(s[..., :1]), s[..., 1:]], -1)
    return (s[..., None] * d).sum(2)


def _stopped(m, x):
    """1 done, 2 close encounter, 3 ejected, after a step."""
    q = x[:, 1:] - x[:, :1]
    r = (q * q).sum(-1).sqrt()
    d = q[:, None] - q[:, :, None]
    d = (d * d).sum(-1).sqrt()
    hill = ((m[:, None, 1:] + m[:, 1:, None]) / (3 * m[:, :1, None])) ** (1.0 / 3) * (r[:, None] + r[:, :, None]) / 2
    off = ~torch.eye(r.shape[1], dtype=torch.bool, device=x.device)
    ce = ((d < CE * hill) & off).any(-1).any(-1)
    return torch.where((r > EJECT).any(-1), 3, torch.where(ce, 2, 0)).to(torch.int32)


def _hermite_step(m, x, v, a, j, h):
    xk, vk = x + h * (v + h * (a / 2 + h * j / 6)), v + h * (a + h * j / 2)
    for _ in range(2):
        ak, jk = _accjerk(m, xk, vk)
        vk = v + h / 2 * (a + ak) + h * h / 12 * (j - jk)
        xk = x + h / 2 * (v + vk) + h * h / 12 * (a - ak)
    return xk, vk


_C = ((), (1 / 5,), (3 / 40, 9 / 40), (3 / 10, -9 / 10, 6 / 5), (-11 / 54, 5 / 2, -70 / 27, 35 / 27),
      (1631 / 55296, 175 / 512, 575 / 13824, 44275 / 110592, 253 / 4096))
_B5 = (37 / 378, 0.0, 250 / 621, 125 / 594, 0.0, 512 / 1771)
_B4 = (2825 / 27648, 0.0, 18575 / 48384, 13525 / 55296, 277 / 14336, 1 / 4)


def _rkck_step(m, x, v, h):
    kx, kv = [], []
    for row in _C:
        xs = x + h * sum((c * k for c, k in zip(row, kx)), torch.zeros_like(x))
        vs = v + h * sum((c * k for c, k in zip(row, kv)), torch.zeros_like(v))
        kx.append(vs)
        kv.append(_acc(m, xs))
    mix = lambda w, ks: h * sum(c * k for c, k in zip(w, ks))
    db = [p - q for p, q in zip(_B5, _B4)]
    size = lambda u: (u * u).sum(-1).sqrt().amax(-1)
    err = torch.maximum(size(mix(db, kx)) / size(x), size(mix(db, kv)) / size(v))
    return x + mix(_B5, kx), v + mix(_B5, kv), err


def _series(z, terms=15):
    """Stumpff functions c2, c3 for |z| of order one."""
    c2 = sum((-z) ** k / float(math.factorial(2 * k + 2)) for k in range(terms - 1, -1, -1))
    c3 = sum((-z) ** k / float(math.factorial(2 * k + 3)) for k in range(terms - 1, -1, -1))
    return c2, c3


def _kepler(mu, r, v, h):
    """Universal variables, Newton; steps of a small part of an orbit (|z| of order one)."""
    r0, sig = (r * r).sum(-1).sqrt(), (r * v).sum(-1)
    smu = mu.sqrt()
    alpha = 2 / r0 - (v * v).sum(-1) / mu
    chi = smu * h / r0
    for _ in range(9):
        c2, c3 = _series(alpha * chi * chi)
        f = sig / smu * chi ** 2 * c2 + (1 - alpha * r0) * chi ** 3 * c3 + r0 * chi - smu * h
        df = sig / smu * chi * (1 - alpha * chi * chi * c3) + (1 - alpha * r0) * chi ** 2 * c2 + r0
        chi = chi - f / df
    z = alpha * chi * chi
    c2, c3 = _series(z)
    f, g = 1 - chi ** 2 * c2 / r0, h - chi ** 3 * c3 / smu
    rn = f[..., None] * r + g[..., None] * v
    r1 = (rn * rn).sum(-1).sqrt()
    fd, gd = smu / (r1 * r0) * chi * (z * c3 - 1), 1 - chi ** 2 * c2 / r1
    return rn, fd[..., None] * r + gd[..., None] * v


def _jacobi_to(m, x):
    eta = m.cumsum(1)[..., None]
    c = (m[..., None] * x).cumsum(1) / eta
    return torch.cat([c[:, -1:], x[:, 1:] - c[:, :-1]], 1)


def _jacobi_from(m, r):
    eta, out, c = m.cumsum(1), [None] * r.shape[1], r[:, 0]
    for i in range(r.shape[1] - 1, 0, -1):
        c = c - (m[:, i] / eta[:, i])[:, None] * r[:, i]
        out[i] = r[:, i] + c
    out[0] = c
    return torch.stack(out, 1)


def _mvs(m, x, v, h, steps, jacobi, live, after):
    eta, m0 = m.cumsum(1), m[:, :1]
    if jacobi:
        q, u = _jacobi_to(m, x), _jacobi_to(m, v)
        mu = m0 * eta[:, 1:] / eta[:, :-1]

        def kick(q):
            a = _acc(m, _jacobi_from(m, q))
            r = q[:, 1:]
            return _jacobi_to(m, a)[:, 1:] + mu[..., None] * r / (r * r).sum(-1, keepdim=True) ** 1.5

        back = lambda q, u: (_jacobi_from(m, q), _jacobi_from(m, u))
        drift = lambda q, u, h: q
    else:
        mean = lambda y: (m[..., None] * y).sum(1, keepdim=True) / m.sum(1)[:, None, None]
        xc, vc = mean(x), mean(v)
        q, u = torch.cat([xc, x[:, 1:] - x[:, :1]], 1), torch.cat([vc, v[:, 1:] - vc], 1)
        mu = m0.expand(-1, m.shape[1] - 1)
        kick = lambda q: _acc(m, q, star=False)[:, 1:]

        def drift(q, u, h):
            p = (m[:, 1:, None] * u[:, 1:]).sum(1, keepdim=True) / m0[..., None]
            return torch.cat([q[:, :1] + h * u[:, :1], q[:, 1:] + h * p], 1)

        def back(q, u):
            x0 = q[:, :1] - (m[:, 1:, None] * q[:, 1:]).sum(1, keepdim=True) / m.sum(1)[:, None, None]
            v0 = u[:, :1] - (m[:, 1:, None] * u[:, 1:]).sum(1, keepdim=True) / m0[..., None]
            return torch.cat([x0, q[:, 1:] + x0], 1), torch.cat([v0, u[:, 1:] + u[:, :1]], 1)

    a = kick(q)
    for k in range(steps):
        qn = drift(q, u, h / 2)
        w = u[:, 1:] + h / 2 * a
        if jacobi:
            qn = torch.cat([qn[:, :1] + h * u[:, :1], qn[:, 1:]], 1)
        r, w = _kepler(mu, qn[:, 1:], w, h)
        qn = torch.cat([qn[:, :1], r], 1)
        an = kick(qn)
        un = torch.cat([u[:, :1], w + h / 2 * an], 1)
        qn = drift(qn, un, h / 2)
        x, v = torch.where(live()[:, None, None], torch.stack(back(qn, un)), torch.stack((x, v)))
        q, u, a = qn, un, an
        after(x, (k + 1) * h)
    return x, v


def _advance(kind, integ, m, x, v, dt, t_end, stops=True):
    """(pos, vel, time, status) of equal-n systems after one call."""
    s = len(x)
    t = torch.zeros(s, dtype=x.dtype, device=x.device)
    st = torch.zeros(s, dtype=torch.int32, device=x.device)

    def after(x, tk):
        nonlocal t, st
        run = st == 0
        t = torch.where(run, tk, t)
        if stops:
            st = torch.where(run, _stopped(m, x), st)

    live = lambda: st == 0
    keep = lambda new, old, ok: torch.where(ok[:, None, None], new, old)
    steps = round(t_end / dt)
    if integ in (S.MVS_DH, S.MVS_JACOBI):
        x, v = _mvs(m, x, v, dt, steps, integ == S.MVS_JACOBI, live, after)
    elif integ == S.HERMITE4:
        for k in range(steps):
            a, j = _accjerk(m, x, v)
            xn, vn = _hermite_step(m, x, v, a, j, dt)
            x, v = keep(xn, x, live()), keep(vn, v, live())
            after(x, (k + 1) * dt)
    elif integ == S.RKCK:
        for k in range(steps):
            xn, vn, _ = _rkck_step(m, x, v, dt)
            x, v = keep(xn, x, live()), keep(vn, v, live())
            after(x, (k + 1) * dt)
    else:
        h = torch.full_like(t, abs(dt))
        going = live()
        while bool(going.any()):
            rem = t_end - t
            if integ == S.HERMITE4_ADAPTIVE:
                a, j = _accjerk(m, x, v)
                h = dt / ((j * j).sum(-1) / (a * a).sum(-1)).sum(-1).sqrt()
            last = h >= rem
            hs = torch.where(last, rem, h)[:, None, None]
            if integ == S.HERMITE4_ADAPTIVE:
                xn, vn = _hermite_step(m, x, v, a, j, hs)
                ok = going
            else:
                xn, vn, err = _rkck_step(m, x, v, hs)
                err = err / EPS
                ok = going & (err <= 1)
                f = 0.9 * err ** -0.2
                h = hs[:, 0, 0] * torch.where(err <= 1, f.clamp(0.2, 5.0), f.clamp(min=0.2))
            x, v = keep(xn, x, ok), keep(vn, v, ok)
            t = torch.where(ok, torch.where(last, torch.full_like(t, t_end), t + hs[:, 0, 0]), t)
            st = torch.where(ok, _stopped(m, x), st)
            going = going & (st == 0) & ~(ok & last)
    st = torch.where(st == 0, 1, st)
    t = torch.where(st == 1, t_end, t)
    return x, v, t, st


def _by_count(ics, advance):
    """Runs advance(m, x, v) for each body count and puts the rows back in the ensemble's order."""
    nb = np.asarray(ics["n_body"])
    first = np.concatenate([[0], np.cumsum(nb)])
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    put = lambda a: torch.as_tensor(np.asarray(a), dtype=torch.float64, device=dev)
    mass, pos, vel = put(ics["mass"]), put(ics["pos"]), put(ics["vel"])
    out = {"pos": torch.empty_like(pos), "vel": torch.empty_like(vel), "time": torch.zeros(len(nb), dtype=torch.float64, device=dev),
           "status": torch.zeros(len(nb), dtype=torch.int32, device=dev)}
    for n in np.unique(nb):
        which = np.nonzero(nb == n)[0]
        rows = torch.as_tensor(first[which][:, None] + np.arange(n)[None, :], device=dev)
        x, v, t, st = advance(mass[rows], pos[rows], vel[rows])
        out["pos"][rows], out["vel"][rows] = x, v
        at = torch.as_tensor(which, device=dev)
        out["time"][at], out["status"][at] = t, st
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind == "serve":
        out = {}
        for k, (ics, t_end, integ) in enumerate(_requests(case, seed)):
            dt = DT if integ == S.HERMITE4 else DT_MVS
            got = _by_count(ics, lambda m, x, v: _advance(kind, integ, m, x, v, dt, t_end))
            out["r%02d" % k] = torch.cat([got["pos"].ravel(), got["vel"].ravel(), got["time"]]).cpu().numpy()
        return out
    ics = _ensemble(case, seed)
    integ, dt, t_end = _plan(case)
    if kind == "rv":
        x, v, m = (torch.as_tensor(ics[k], dtype=torch.float64).reshape(case["systems"], 3, -1) for k in ("pos", "vel", "mass"))
        m, rv = m[..., 0], []
        for _ in range(12):
            x, v, _, _ = _advance(kind, integ, m, x, v, dt, case["steps"] * dt, stops=False)
            rv.append(v[:, 0] @ torch.tensor(LOS, dtype=torch.float64))
        return {"rv": torch.stack(rv).numpy()}
    out = _by_count(ics, lambda m, x, v: _advance(kind, integ, m, x, v, dt, t_end))
    out["status"] = None
    return out
