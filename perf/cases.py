"""Workloads of the test-particle map, each through the package's public entry points.

Every kind of call that a program makes of this package has a case: one-shot
runs of a particle set (create, advance, read), short calls on a context that
is kept, the eccentric and fixed-iteration variants, runs with element
sampling, batches of systems, the differentiable map with its adjoint and with
the growth indicator's gradient, and the device-level partition.  Sizes run
from about a thousand particles (latency) to the million-particle belt.

``exact`` restates the map in plain float64 torch / numpy.
"""
import math

import numpy as np
import torch

import glisse_inputs as gi
import paper_2011_03484_gb300 as G

G0 = 4.0 * math.pi * math.pi
DT = 0.5
DEVICE = "cuda"

# orbits: (a range in AU, e range, sigma_i in degrees), as the package's own workloads draw them
BELTS = {
    "inner": ((21.0, 28.0), (0.0, 0.05), 1.0),   # between Uranus and Neptune, cold
    "scatter": ((20.0, 29.0), (0.0, 0.1), 2.0),  # the same region, removals throughout
    "outer": ((40.0, 50.0), (0.0, 0.4), 5.0),    # resonant belt beyond Neptune
    "eccentric": ((20.0, 29.0), (0.0, 0.9), 2.0),  # planet-crossing, mixed solve costs
}


def listed():
    return [
        # a program that steps and looks: a kept context, few steps a call
        {"name": "call_1000x16", "kind": "call", "belt": "inner", "n": 1000, "steps": 16},
        # a small study from start to end
        {"name": "run_1024x1000", "kind": "run", "belt": "inner", "n": 1024, "steps": 1000},
        # ordinary runs: odd size, more than one planet chunk
        {"name": "run_20011x1500", "kind": "run", "belt": "outer", "n": 20011, "steps": 1500},
        {"name": "run_131072x2048", "kind": "run", "belt": "scatter", "n": 131072, "steps": 2048},
        # the largest set
        {"name": "run_1048576x1024", "kind": "run", "belt": "outer", "n": 1048576, "steps": 1024},
        # planet-crossing orbits up to e = 0.9
        {"name": "run_ecc_65537x512", "kind": "run", "belt": "eccentric", "n": 65537, "steps": 512},
        # the published fixed-iteration solver, an option of the same call
        {"name": "fixed_30000x256", "kind": "fixed", "belt": "scatter", "n": 30000, "steps": 256},
        # elements logged for resonance studies
        {"name": "sampled_32768x1024", "kind": "sampled", "belt": "outer", "n": 32768, "steps": 1024, "every": 128},
        # many systems in one context, 2 to 8 planets each
        {"name": "batch_24x512", "kind": "batch", "systems": 24, "n_max": 65536, "steps": 512},
        # gradients of final states: forward with the per-step record, then the adjoint
        {"name": "adjoint_32768x512", "kind": "adjoint", "belt": "inner", "n": 32768, "steps": 512, "every": 0},
        # stability indicator and its gradient, from checkpoints
        {"name": "growth_8209x256", "kind": "growth", "belt": "inner", "n": 8209, "steps": 256, "every": 64},
        # device-level stable partition of a caller's own arrays
        {"name": "partition_3000017", "kind": "partition", "n": 3000017, "keep": 0.9},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["call", "run", "run", "run", "run", "fixed", "sampled", "batch", "adjoint", "growth",
                       "partition"])
    belt = rng.choice(sorted(BELTS))
    if kind == "call":
        return {"kind": kind, "belt": belt, "n": _log_int(rng, 200, 200000), "steps": _log_int(rng, 1, 64)}
    if kind == "run":
        n = _log_int(rng, 500, 1000000)
        return {"kind": kind, "belt": belt, "n": n, "steps": _log_int(rng, 64, min(4096, 1024 * 1048576 // n // 2))}
    if kind == "fixed":
        return {"kind": kind, "belt": "scatter", "n": _log_int(rng, 500, 100000), "steps": _log_int(rng, 32, 512)}
    if kind == "sampled":
        every = rng.choice([64, 100, 128, 200])
        return {"kind": kind, "belt": rng.choice(["inner", "outer", "scatter"]), "n": _log_int(rng, 1000, 60000),
                "steps": every * rng.randint(2, 8), "every": every}
    if kind == "batch":
        return {"kind": kind, "systems": _log_int(rng, 2, 64), "n_max": _log_int(rng, 1000, 65536),
                "steps": _log_int(rng, 64, 512)}
    if kind == "adjoint":
        return {"kind": kind, "belt": rng.choice(["inner", "outer", "scatter"]), "n": _log_int(rng, 500, 65536),
                "steps": _log_int(rng, 32, 512), "every": rng.choice([0, 0, 50, 256])}
    if kind == "growth":
        return {"kind": kind, "belt": rng.choice(["inner", "outer"]), "n": _log_int(rng, 500, 16384),
                "steps": _log_int(rng, 32, 256), "every": rng.choice([64, 256, -2])}
    return {"kind": kind, "n": _log_int(rng, 5000, 4000000), "keep": round(rng.uniform(0.3, 1.0), 3)}


# ---- inputs ----------------------------------------------------------------
def _system(case, seed):
    rng = np.random.Generator(np.random.PCG64([seed, 20110]))
    planets = gi.planet_system(rng)
    a, e, sig = BELTS[case["belt"]]
    return planets, gi.particle_belt(rng, case["n"], a, e, sig)


def _batch_sizes(case):
    return [int(round(n)) for n in np.geomspace(512, case["n_max"], case["systems"])]


def _batch_inputs(case, seed):
    one = [gi.make_batched(seed=[seed, s], n_systems=1, n_min=n, n_max=n) for s, n in enumerate(_batch_sizes(case))]
    return {k: np.concatenate([b[k] for b in one]) for k in one[0]}


def _pinned(shape, dtype):
    return torch.empty(shape, dtype=dtype, pin_memory=True).numpy()


def _out_buffers(n):
    return {"state": _pinned((n, 6), torch.float64), "alive": _pinned((n,), torch.uint8),
            "removal_step": _pinned((n,), torch.int64), "removal_reason": _pinned((n,), torch.int32)}


def _unit(x):
    return x / x.norm(dim=1, keepdim=True)


def _diff_inputs(case, seed):
    planets, parts = _system(case, seed)
    gen = torch.Generator().manual_seed(seed)
    g = torch.randn(case["n"], 6, dtype=torch.float64, generator=gen)
    return planets, torch.from_numpy(parts).to(DEVICE), g.to(DEVICE)


def _partition_inputs(case, seed):
    gen = torch.Generator(device=DEVICE).manual_seed(seed)
    n = case["n"]
    src = torch.randn(6, n, dtype=torch.float64, device=DEVICE, generator=gen)
    keep = (torch.rand(n, device=DEVICE, generator=gen) < case["keep"]).to(torch.uint8)
    return src, torch.arange(n, dtype=torch.int32, device=DEVICE), keep


def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case}
    if kind in ("run", "fixed", "sampled", "call"):
        planets, parts = _system(case, seed)
        host = _pinned(parts.shape, torch.float64)
        host[:] = parts
        st.update(planets=planets, particles=host, out=_out_buffers(case["n"]))
        if kind == "call":
            st["sim"] = G.Simulation(1.0, planets, host, DT)
    elif kind == "batch":
        b = _batch_inputs(case, seed)
        st.update(batch=b, out=_out_buffers(len(b["particles"])))
    elif kind in ("adjoint", "growth"):
        planets, s0, g = _diff_inputs(case, seed)
        st.update(s0=s0, g=g, map=G.DiffMap(1.0, planets, case["n"], DT, case["steps"],
                                            checkpoint_every=case["every"]))
        if kind == "growth":
            st["t0"] = _unit(g).unsqueeze(0).contiguous()
            st["gg"] = g[:, 0].contiguous()
    else:
        src, ids, keep = _partition_inputs(case, seed)
        st.update(src=src, ids=ids, keep=keep, dst=torch.zeros_like(src), dst_id=torch.full_like(ids, -1),
                  count=torch.zeros(1, dtype=torch.int64, device=DEVICE))
    return st


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "call":
        st["sim"].advance(case["steps"])
        return st["sim"].read(st["out"])
    if kind in ("run", "fixed", "sampled"):
        opt = {"kepler_mode": G.GLISSE_KEPLER_PAPER_FIXED} if kind == "fixed" else {}
        sim = G.Simulation(1.0, st["planets"], st["particles"], DT, **opt)
        if kind == "sampled":
            sim.set_sampling(case["every"], max_samples=case["steps"] // case["every"], res_planet=3, res_p=3, res_q=2)
        sim.advance(case["steps"])
        got = sim.read(st["out"])
        if kind == "sampled":
            got["elements"] = sim.elements()[0]
            got["count"] = sim.libration()["count"]
        sim.close()
        return got
    if kind == "batch":
        b = st["batch"]
        sim = G.BatchSimulation(b["star_mass"], b["n_planets"], b["planets"], b["n_particles"], b["particles"], b["dt"])
        sim.advance(case["steps"])
        got = sim.read(st["out"])
        sim.close()
        return got
    if kind == "adjoint":
        s1, _, _, rstep, reason = st["map"].forward(st["s0"])
        return {"state": s1, "gradient": st["map"].backward(st["g"]), "removal_step": rstep, "removal_reason": reason}
    if kind == "growth":
        s1, t1, growth, rstep, reason = st["map"].forward(st["s0"], st["t0"])
        gs, gt = st["map"].backward_growth(st["g"], st["gg"], t1[0])
        return {"state": s1, "tangent": t1, "growth": growth, "gradient": gs, "gradient_seed": gt,
                "removal_step": rstep, "removal_reason": reason}
    G.glisse_partition_device(case["n"], case["n"], st["keep"].data_ptr(), st["src"].data_ptr(), st["ids"].data_ptr(),
                              st["dst"].data_ptr(), st["dst_id"].data_ptr(), st["count"].data_ptr(),
                              torch.cuda.current_stream().cuda_stream)
    return {"dst": st["dst"], "dst_id": st["dst_id"], "count": st["count"]}


# ---- what a pass cannot do without ------------------------------------------
def _map_flops(npl):
    # drift and h0 term 86, each planet's kick 25 (a fused multiply-add counts two)
    return 86.0 + 25.0 * npl


def work(case):
    kind = case["kind"]
    if kind == "partition":
        kept = case["keep"] * case["n"]
        return {"bytes": case["n"] + 2 * 52 * kept, "flops": 0}
    if kind == "batch":
        n = sum(_batch_sizes(case))  # two to eight planets, five on average
        return {"bytes": n * (48 + 61), "flops": n * case["steps"] * _map_flops(5)}
    n, steps = case["n"], case["steps"]
    flops = n * steps * _map_flops(4)
    io = n * (48 + 61)
    if kind == "sampled":
        return {"bytes": io + 48 * n * (steps // case["every"]) + 4 * n, "flops": flops}
    if kind == "adjoint":  # the map and its transposed Jacobians, about two maps
        return {"bytes": n * 48 * 4, "flops": 3 * flops}
    if kind == "growth":  # the map with a tangent, and the sweep of the map extended by it
        return {"bytes": n * 48 * 7, "flops": 9 * flops}
    return {"bytes": io, "flops": flops}


# Relative errors of the start's outputs against `exact` are 4e-16 (16 steps) to 1e-12 where particles stay clear of
# the planets.  On planet-crossing orbits a few particles that pass close to a planet multiply a rounding difference
# and set the norm: 4e-12 to 3e-9 between particle sets, and more where a pass is closer still.
TOLERANCE = {
    "call": {"rel": 1e-11, "max": 1e-8, "differ": 0.001},
    "run": {"rel": 1e-10, "max": 1e-6, "differ": 0.001},
    "fixed": {"rel": 1e-10, "max": 1e-6, "differ": 0.001},
    "sampled": {"rel": 1e-9, "max": 1e-5, "differ": 0.001},
    "batch": {"rel": 1e-9, "max": 1e-5, "differ": 0.001},
    "adjoint": {"rel": 1e-9, "max": 1e-5, "differ": 0.001},
    "growth": {"rel": 1e-9, "max": 1e-5, "differ": 0.001},
}
CROSSING = {"rel": 1e-7, "max": 1e-3, "differ": 0.001}


def tolerance(case):
    if case["kind"] in ("run", "sampled") and case["belt"] in ("scatter", "eccentric"):
        return CROSSING
    return TOLERANCE.get(case["kind"], "exact")


# ---- the map in plain float64 -----------------------------------------------
def _stumpff(z):
    """c0..c3 of an array (numpy or torch): quarter until |z| < 0.5, series, duplication."""
    big = float(abs(z.detach() if torch.is_tensor(z) else z).max()) if z.shape[-1] else 0.0
    k = 0
    while big > 0.5 and k < 40:
        big *= 0.25
        k += 1
    z = z * 0.25**k
    c2 = c3 = 0.0
    for n in range(9, -1, -1):
        c2 = c2 * -z + 1.0 / math.factorial(2 * n + 2)
        c3 = c3 * -z + 1.0 / math.factorial(2 * n + 3)
    c0, c1 = 1.0 - z * c2, 1.0 - z * c3
    for _ in range(k):
        c0, c1, c2, c3 = 2.0 * c0 * c0 - 1.0, c0 * c1, 0.5 * c1 * c1, 0.25 * (c3 + c1 * c2)
    return c0, c1, c2, c3


def _drift(mu, dt, x, v, newton=0):
    """Two-body motion of the columns of x, v [..., 3, n]: Laguerre's iteration on the universal Kepler
    equation, then `newton` Newton steps (which carry the derivatives when autograd records them)."""
    r0 = (x * x).sum(-2) ** 0.5
    u = (x * v).sum(-2)
    beta = 2.0 * mu / r0 - (v * v).sum(-2)
    s = dt / r0 * (1.0 - 0.5 * dt * u / (r0 * r0))
    tensor = torch.is_tensor(x)
    q = [t.detach() if tensor else t for t in (r0, u, beta, s)]
    if tensor and torch.autograd.forward_ad._current_level >= 0:
        q = [torch.autograd.forward_ad.unpack_dual(t).primal.detach() for t in q]
    qr, qu, qb, s = q
    for it in range(30):
        c0, c1, c2, c3 = _stumpff(qb * s * s)
        f = qr * s * c1 + qu * s * s * c2 + mu * s * s * s * c3 - dt
        f1 = qr * c0 + qu * s * c1 + mu * s * s * c2
        f2 = qu * c0 + (mu - qb * qr) * s * c1
        root = abs(16.0 * f1 * f1 - 20.0 * f * f2) ** 0.5
        ds = -5.0 * f / (f1 + root)
        s = s + ds
        if it >= 1 and not bool((abs(ds) > 1e-9 * abs(s)).any()):
            break
    for _ in range(newton):
        c0, c1, c2, c3 = _stumpff(beta * s * s)
        s = s - (r0 * s * c1 + u * s * s * c2 + mu * s * s * s * c3 - dt) / (r0 * c0 + u * s * c1 + mu * s * s * c2)
    c0, c1, c2, c3 = _stumpff(beta * s * s)
    g1, g2, g3 = s * c1, s * s * c2, s * s * s * c3
    r = r0 * c0 + u * g1 + mu * g2
    f, g = (1.0 - mu * g2 / r0), dt - mu * g3
    fd, gd = -mu * g1 / (r * r0), 1.0 - mu * g2 / r
    one = (Ellipsis, None, slice(None))
    return f[one] * x + g[one] * v, fd[one] * x + gd[one] * v


def _planets(m, pos, vel, dt, steps, keep_vel=False):
    """Wisdom-Holman map in Jacobi coordinates for systems [S] of planets [P] (star mass 1): heliocentric
    positions [steps + 1][S][3][P] (and velocities)."""
    S, P = m.shape
    eta = np.concatenate([np.ones((S, 1)), 1.0 + np.cumsum(m, axis=1)], axis=1)
    lower = np.tril(np.ones((P, P)), -1)  # [i][k], k < i
    q, w = np.empty_like(pos), np.empty_like(vel)
    for i in range(P):
        q[:, :, i] = pos[:, :, i] - (m[:, None, :i] * pos[:, :, :i]).sum(-1) / eta[:, i, None]
        w[:, :, i] = vel[:, :, i] - (m[:, None, :i] * vel[:, :, :i]).sum(-1) / eta[:, i, None]
    back = lower[None] * (m / eta[:, 1:])[:, None, :]  # r_i = q_i + sum_{k<i} m_k / eta_k q_k
    mu = G0 * eta[:, 1:] / eta[:, :-1]
    h = np.asarray(dt, dtype=np.float64).reshape(S, 1)

    def helio(a):
        return a + np.einsum("sik,sdk->sdi", back, a)

    def accel(q, r):
        d = r[:, :, :, None] - r[:, :, None, :]
        d2 = (d * d).sum(1) + np.eye(P)
        gh = G0 * r / ((r * r).sum(1) ** 1.5)[:, None, :]
        gh = gh + G0 * (m[:, None, None, :] * d * (d2**-1.5)[:, None, :, :]).sum(-1)
        suffix = np.einsum("sik,sdi->sdk", np.broadcast_to(lower, (S, P, P)), m[:, None, :] * gh)
        grad = gh + suffix / eta[:, None, 1:] - G0 * q / ((q * q).sum(1) ** 1.5)[:, None, :]
        return -(eta[:, 1:] / eta[:, :-1])[:, None, :] * grad

    r = helio(q)
    a = accel(q, r)
    log, logv = [r], [helio(w)]
    for _ in range(steps):
        w = w + 0.5 * h[:, :, None] * a
        q, w = _drift(mu, h, q, w)
        r = helio(q)
        a = accel(q, r)
        w = w + 0.5 * h[:, :, None] * a
        log.append(r)
        if keep_vel:
            logv.append(helio(w))
    return np.stack(log), (np.stack(logv) if keep_vel else None)


def _hill(m, pos, vel):
    r = np.sqrt((pos**2).sum(-2))
    a = 1.0 / (2.0 / r - (vel**2).sum(-2) / (G0 * (1.0 + m)))
    return a * np.cbrt(m / 3.0)


class _Map:
    """Particles [3, n] against planet positions log [steps + 1][3][P] (one system) or, with `sysid`,
    [steps + 1][S][3][P]."""

    def __init__(self, log, gm, rc, dt, sysid=None):
        self.log = torch.from_numpy(np.ascontiguousarray(log)).to(DEVICE)
        self.gm = torch.from_numpy(np.ascontiguousarray(gm)).to(DEVICE)
        self.rc2 = torch.from_numpy(np.ascontiguousarray(rc * rc)).to(DEVICE)
        self.dt, self.sysid = dt, sysid
        h0 = -(self.gm[..., None, :] * self.log / ((self.log**2).sum(-2, keepdim=True) ** 1.5)).sum(-1)
        self.h0 = h0
        if sysid is not None:
            self.gm_p, self.rc2_p = self.gm[sysid].T[:, :], self.rc2[sysid].T[:, :]  # [P, n]
        else:
            self.gm_p, self.rc2_p = self.gm[:, None], self.rc2[:, None]

    def at(self, k):
        if self.sysid is None:
            return self.log[k].T[:, :, None], self.h0[k][:, None]  # [P, 3, 1], [3, 1]
        return self.log[k][self.sysid].permute(2, 1, 0), self.h0[k][self.sysid].T  # [P, 3, n], [3, n]

    def geometry(self, x, k):
        p, h0 = self.at(k)
        d = x[None] - p
        return d, (d * d).sum(1), h0

    def hit(self, x, d2):
        """0 or the removal reason: the lowest planet, before escape."""
        near = d2 < self.rc2_p
        first = near.to(torch.int8).argmax(0).to(torch.int32) + 1
        r2 = (x * x).sum(0)
        return torch.where(near.any(0), first, torch.where(r2 > 1e6, -1, 0).to(torch.int32))

    def kick(self, d, d2, h0, tau):
        return tau * (h0 - ((self.gm_p / (d2 * d2.sqrt()))[:, None] * d).sum(0))

    def run(self, x, v, steps, newton=0, at_step=None):
        n = x.shape[1]
        step = torch.full((n,), -1, dtype=torch.int64, device=x.device)
        d, d2, h0 = self.geometry(x, 0)
        reason = self.hit(x.detach(), d2.detach())
        step = torch.where(reason != 0, 0, step)
        live = reason == 0
        for k in range(steps):
            xd, vd = _drift(G0, self.dt, x, v + self.kick(d, d2, h0, 0.5 * self.dt), newton)
            d, d2, h0 = self.geometry(xd, k + 1)
            h = torch.where(live, self.hit(xd.detach(), d2.detach()), 0)
            vk = vd + self.kick(d, d2, h0, 0.5 * self.dt)
            gone = live & (h != 0)
            x = torch.where(live, xd, x)
            v = torch.where(gone, vd, torch.where(live, vk, v))
            step = torch.where(gone, k + 1, step)
            reason = torch.where(gone, h, reason)
            live = live & ~gone
            if not bool(live.all()):  # removed particles stay where they are
                d, d2, h0 = self.geometry(x, k + 1)
            if at_step is not None:
                at_step(k + 1, x, v, live)
        return x, v, step, reason


def _result(x, v, step, reason):
    return {"state": torch.cat([x, v]).T.contiguous(), "alive": step < 0, "removal_step": step,
            "removal_reason": reason}


def _elements(mu, s):
    """a, e, i, node, peri, M of rows s [n, 6] about mu (bound orbits; others NaN)."""
    r, v = s[:, :3], s[:, 3:]
    rn = r.norm(dim=1)
    h = torch.linalg.cross(r, v)
    hn = h.norm(dim=1)
    ev = torch.linalg.cross(v, h) / mu - r / rn[:, None]
    e = ev.norm(dim=1)
    a = 1.0 / (2.0 / rn - (v * v).sum(1) / mu)
    inc = torch.atan2((h[:, 0] ** 2 + h[:, 1] ** 2).sqrt(), h[:, 2])
    node = torch.atan2(h[:, 0], -h[:, 1])
    p = torch.stack([node.cos(), node.sin(), torch.zeros_like(node)], dim=1)
    q = torch.linalg.cross(h / hn[:, None], p)
    peri = torch.atan2((ev * q).sum(1), (ev * p).sum(1))
    f = torch.atan2((r * q).sum(1), (r * p).sum(1)) - peri
    E = torch.atan2(((1 - e) * (1 + e)).sqrt() * f.sin(), e + f.cos())
    tau = 2.0 * math.pi
    return torch.stack([a, e, inc, node % tau, peri % tau, (E - e * E.sin()) % tau], dim=1)


def _helio(planets):
    return planets[:, 0], planets[None, :, 1:4].transpose(0, 2, 1), planets[None, :, 4:7].transpose(0, 2, 1)


def _one_system(planets, steps, keep_vel=False):
    m, pos, vel = _helio(planets)
    log, logv = _planets(m[None], pos, vel, DT, steps, keep_vel)
    return _Map(log[:, 0], G0 * m, _hill(m, pos[0], vel[0]), DT), log[:, 0], None if logv is None else logv[:, 0]


def exact(case, seed):
    kind = case["kind"]
    if kind == "partition":
        src, ids, keep = _partition_inputs(case, seed)
        at = keep.nonzero()[:, 0]
        dst, dst_id = torch.zeros_like(src), torch.full_like(ids, -1)
        dst[:, : len(at)] = src[:, at]
        dst_id[: len(at)] = ids[at]
        return {"dst": dst, "dst_id": dst_id, "count": torch.tensor([len(at)])}
    if kind == "batch":
        return _exact_batch(case, seed)
    if kind in ("adjoint", "growth"):
        return _exact_diff(case, seed)
    planets, parts = _system(case, seed)
    p = torch.from_numpy(parts).to(DEVICE)
    m, log, logv = _one_system(planets, case["steps"], kind == "sampled")
    kept = []
    mt = 1.0 + planets[:, 0].sum()

    def sample(k, x, v, live):
        if k % case["every"]:
            return
        off = torch.from_numpy(np.concatenate([(planets[:, 0] * a[k]).sum(-1) / mt for a in (log, logv)])).to(DEVICE)
        el = _elements(G0 * mt, torch.cat([x, v]).T - off)
        kept.append(torch.where(live[:, None], el, float("nan")))

    got = _result(*m.run(p[:, :3].T.contiguous(), p[:, 3:].T.contiguous(), case["steps"],
                         at_step=sample if kind == "sampled" else None))
    if kind == "sampled":
        got["elements"] = torch.stack(kept)
        got["count"] = (~torch.isnan(got["elements"][:, :, 5])).sum(0).to(torch.int32)
    return got


def _exact_batch(case, seed):
    b = _batch_inputs(case, seed)
    S, P = case["systems"], 8
    m = np.zeros((S, P))
    # places without a planet hold a massless body on a far circular orbit
    pos, vel = np.zeros((S, 3, P)), np.zeros((S, 3, P))
    for j in range(P):
        pos[:, 0, j] = 1e4 * (j + 1)
        vel[:, 1, j] = math.sqrt(G0 / (1e4 * (j + 1)))
    rc = np.zeros((S, P))
    off = 0
    for s in range(S):
        k = int(b["n_planets"][s])
        pl = b["planets"][off:off + k]
        off += k
        m[s, :k], pos[s, :, :k], vel[s, :, :k] = pl[:, 0], pl[:, 1:4].T, pl[:, 4:7].T
        rc[s, :k] = _hill(pl[:, 0], pl[:, 1:4].T, pl[:, 4:7].T)
    log, _ = _planets(m, pos, vel, b["dt"], case["steps"])
    sysid = torch.from_numpy(np.repeat(np.arange(S), b["n_particles"])).to(DEVICE)
    dt = torch.from_numpy(np.repeat(b["dt"], b["n_particles"])).to(DEVICE)
    p = torch.from_numpy(b["particles"]).to(DEVICE)
    return _result(*_Map(log, G0 * m, rc, dt, sysid).run(p[:, :3].T.contiguous(), p[:, 3:].T.contiguous(),
                                                        case["steps"]))


def _exact_diff(case, seed):
    planets, s0, g = _diff_inputs(case, seed)
    m = _one_system(planets, case["steps"])[0]
    s0 = s0.requires_grad_(True)
    if case["kind"] == "adjoint":
        got = m.run(s0[:, :3].T, s0[:, 3:].T, case["steps"], newton=1)
        s1 = torch.cat(got[:2]).T
        (grad,) = torch.autograd.grad(s1, s0, g)
        return {"state": s1.detach(), "gradient": grad, "removal_step": got[2], "removal_reason": got[3]}
    deep = case["steps"] <= 40  # the gradient of the growth: a graph of the tangent's own graph, time and memory
    t0 = _unit(g).requires_grad_(deep)
    s0.requires_grad_(deep)
    with torch.set_grad_enabled(deep), torch.autograd.forward_ad.dual_level():
        d = torch.autograd.forward_ad.make_dual(s0, t0)
        got = m.run(d[:, :3].T, d[:, 3:].T, case["steps"], newton=2)
        s1, t1 = torch.autograd.forward_ad.unpack_dual(torch.cat(got[:2]).T)
        growth = 0.5 * torch.log((t1 * t1).sum(1) / (t0 * t0).sum(1))
        gs = gt = None
        if deep:
            gs, gt = torch.autograd.grad((s1 * g).sum() + (growth * g[:, 0]).sum(), (s0, t0))
    return {"state": s1.detach(), "tangent": t1.detach()[None], "growth": growth.detach(), "gradient": gs,
            "gradient_seed": gt, "removal_step": got[2], "removal_reason": got[3]}
