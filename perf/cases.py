"""Workloads of the kinetic Monte Carlo library, each one pass through its public calls.

A pass is one of three programs:

``advance``  a simulation that lives on: ``step(k)``, ``sync()``, and the state gathered into
             the caller's device buffer (``state_device``), as an in-situ analysis reads it.
``job``      a whole run: a simulation made from the caller's arrays or init descriptor, stepped,
             its state and step records (and profiles) read, and closed, as a queue of runs does.
``group``    an ensemble that lives on: one group of boxes and tubes stepped together, every
             member's state gathered.

The gases are the ones of ``kmc_inputs``: the equilibrium box, the piston tube, the paper's
equal-speed gases in three dimensions and in the plane, the spherical blast and the binary
mixture, at its densities, diameters and time steps.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import kmc_inputs as ki
import paper_1310_3437_gb300 as kmc


# --------------------------------------------------------------------------- #
# cases

def listed():
    return [
        # interactive use and coupling to a host code: one step at a time, launches count
        case("box_4k_single_step", "advance", "box", 4096, steps=1),
        # the 4096-particle box in binary64, the binding's default precision
        case("box_4k_fp64", "advance", "box", 4096, steps=10, fp64=True),
        # one request of a serving stream: host arrays in, 100 steps, state and records out
        case("request_tube_50k", "job", "tube", 50021, steps=100, source="host", u_p=2.0),
        # a box of the serving stream, between observations
        case("box_262k", "advance", "box", 262139, steps=8),
        # an ensemble of independent runs (even: boxes with many particles per cell; odd: tubes)
        case("ensemble_30", "group", "ensemble", 0, steps=4, members=30, first=1000),
        # the shock tube of the profiles, start to observation, from arrays on the device
        case("tube_1M_job", "job", "tube", 1 << 20, steps=100, source="device", u_p=2.0, every=20),
        # the same tube in binary64
        case("tube_1M_fp64", "advance", "tube", 1 << 20, steps=2, u_p=2.0, fp64=True),
        # a mixture between absorbing walls (evaporation), all options of a particle kind
        case("mixture_100k_absorbing", "job", "mixture", 100003, steps=50, source="device",
             absorb=True),
        # dense hot ball in a cold gas: most of the work in few cells
        case("blast_2M", "job", "blast", 1 << 21, steps=10, source="init"),
        # the paper's hybrid study: particles in the plane
        case("plane_10M", "advance", "plane", 10_000_003, steps=4),
        # the headline tube
        case("tube_16M", "advance", "tube", 1 << 24, steps=4, u_p=2.0),
        # the paper's timing study: 10^8 particles in three dimensions
        case("gas_100M", "advance", "gas", 10 ** 8, steps=2),
    ]


def case(name, program, gas, n, steps, fp64=False, **more):
    return dict({"name": name, "program": program, "gas": gas, "n": n, "steps": steps,
                 "fp64": fp64}, **more)


def draw(rng):
    """One more case of the same programs and ranges."""
    kind = rng.choice(["box", "box", "box64", "request", "ensemble", "tube_job", "tube", "tube64",
                       "mixture", "blast", "plane", "gas"])

    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    if kind == "box":
        c = case("", "advance", "box", size(1 << 11, 1 << 21), rng.randint(1, 8))
    elif kind == "box64":
        c = case("", "advance", "box", size(1 << 11, 1 << 19), rng.randint(1, 10), True)
    elif kind == "request":
        c = case("", "job", "tube", size(1 << 14, 1 << 18), rng.randint(60, 140), source="host",
                 u_p=rng.uniform(1.0, 3.0))
    elif kind == "ensemble":
        c = case("", "group", "ensemble", 0, rng.randint(1, 6), members=rng.randint(6, 30),
                 first=1000 + 2 * rng.randint(1, 100))
    elif kind == "tube_job":
        c = case("", "job", "tube", size(1 << 17, 1 << 20), rng.randint(40, 100), source="device",
                 u_p=rng.uniform(1.0, 3.0), every=20)
    elif kind == "tube":
        c = case("", "advance", "tube", size(1 << 19, 1 << 24), rng.randint(1, 8),
                 u_p=rng.uniform(1.0, 3.0))
    elif kind == "tube64":
        c = case("", "advance", "tube", size(1 << 16, 1 << 20), rng.randint(1, 3), True,
                 u_p=rng.uniform(1.0, 3.0))
    elif kind == "mixture":
        c = case("", "job", "mixture", size(1 << 13, 1 << 19), rng.randint(30, 60),
                 source="device", absorb=rng.random() < 0.5)
    elif kind == "blast":
        c = case("", "job", "blast", size(1 << 17, 1 << 21), rng.randint(6, 10), source="init")
    elif kind == "plane":
        c = case("", "advance", "plane", size(1 << 20, 40_000_000), rng.randint(1, 4))
    else:
        c = case("", "advance", "gas", size(1 << 20, 60_000_000), rng.randint(1, 3))
    del c["name"]
    return c


# --------------------------------------------------------------------------- #
# the gases

def setup_of(c, seed):
    """The physical set-up of a case (kmc_inputs.Setup); the seed keys its scatter draws."""
    n, gas = c["n"], c["gas"]
    if gas == "box":  # the serving stream's box: the 4096-particle box's density and d0
        return ki.equilibrium_setup(n=n, seed=seed, L=(n / 4096.0) ** (1.0 / 3.0))
    if gas == "tube":
        every = c.get("every", 0)
        return ki.piston_setup(n=n, seed=seed, u_p=c["u_p"], profile_every=every,
                               profile_bins=256 if every else 0)
    if gas == "mixture":
        s = ki.mixture_setup(n=n, seed=seed, L=(n / 6000.0) ** (1.0 / 3.0))
        return s.with_(bc=(ki.ABSORB, ki.PERIODIC, ki.PERIODIC)) if c.get("absorb") else s
    if gas == "blast":
        return ki.blast_setup(n=n, seed=seed)
    if gas == "plane":  # mean free path 0.001, time step a tenth of it
        return ki.equal_speed_setup(n=n, seed=seed, planar=True, dt=1e-4,
                                    d0=1.0 / (2.0 * math.sqrt(2.0) * n * 0.001))
    if gas == "gas":  # mean free path 0.01, time step a tenth of it
        return ki.equal_speed_setup(n=n, seed=seed, planar=False, dt=1e-3,
                                    d0=ki.d0_for_mean_free_path(float(n), 0.01))
    raise ValueError(gas)


def member_setups(c, seed):
    """The members of an ensemble: the sizes and pistons are the case's, the draws the seed's."""
    out = ki.ensemble_setups(c["members"], seed0=c["first"])
    return [s.with_(seed=seed * 1000 + k) for k, s in enumerate(out)]


def arrays_of(setup, seed):
    """x, y, z, vx, vy, vz on the GPU: uniform positions, normal velocities (of a mixture's
    species at temperature 1)."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    n = setup.n

    def uniform(hi):
        u = torch.rand(n, generator=g, device="cuda", dtype=torch.float64) * hi
        return torch.clamp_(u, max=math.nextafter(hi, 0.0))

    out = [uniform(float(b)) for b in setup.box]
    out += [torch.randn(n, generator=g, device="cuda", dtype=torch.float64) for _ in range(3)]
    if setup.species is not None:
        m = torch.tensor(setup.masses, dtype=torch.float64, device="cuda")
        scale = torch.sqrt(1.0 / m)[torch.from_numpy(setup.species).long().cuda()]
        out[3:] = [v * scale for v in out[3:]]
    return out


# --------------------------------------------------------------------------- #
# what a program has in hand, and a pass

WARM = 20  # steps after which an equal-speed gas is near its equilibrium


def prepare(case, seed):
    c = dict(case)
    state = {"case": c, "stream": torch.cuda.Stream()}
    precision = kmc.KMC_FP64 if c["fp64"] else kmc.KMC_GUARDED_FP32
    if c["program"] == "group":
        setups = member_setups(c, seed)
        params = [kmc.params_from_setup(s, precision=precision) for s in setups]
        arrays = [arrays_of(s, s.seed) for s in setups]
        state["stream"].wait_stream(torch.cuda.current_stream())
        sims = [kmc.Simulation(p, a, stream=state["stream"].cuda_stream)
                for p, a in zip(params, arrays)]
        state["sims"] = sims
        state["group"] = kmc.Group(sims, stream=state["stream"].cuda_stream)
        state["out"] = [out_buffer(s.n) for s in setups]
        return state
    setup = setup_of(c, seed)
    state["setup"] = setup
    state["params"] = kmc.params_from_setup(setup, precision=precision)
    if setup.species is not None:
        state["mixture"] = (torch.from_numpy(setup.species).cuda(), setup.masses, setup.radii)
    source = c.get("source", "init" if c["gas"] in ("plane", "gas") else "device")
    if source == "init":
        state["init"] = ki.init_spec(setup)
    else:
        state["arrays"] = arrays_of(setup, seed)
        if source == "host":
            state["arrays"] = [a.cpu().numpy() for a in state["arrays"]]
    if c["program"] == "advance":
        state["sim"] = make(state)
        if c["gas"] in ("plane", "gas"):
            state["sim"].step(WARM).sync()
        state.pop("arrays", None)
    if source != "host":
        state["out"] = out_buffer(setup.n)
    return state


def make(state):
    state["stream"].wait_stream(torch.cuda.current_stream())  # the arrays are ready
    return kmc.Simulation(state["params"], state.get("arrays"), init=state.get("init"),
                          mixture=state.get("mixture"), stream=state["stream"].cuda_stream)


def out_buffer(n):
    return torch.zeros(52 * n, dtype=torch.uint8, device="cuda")


def views(buf):
    n = buf.numel() // 52
    return buf[: 48 * n].view(torch.float64).view(6, n), buf[48 * n:].view(torch.int32)


def run(state):
    c = state["case"]
    if c["program"] == "group":
        for sim in state["sims"]:
            state["group"].budget(sim, c["steps"])
        state["group"].step(c["steps"])
        state["group"].sync()
        for sim, buf in zip(state["sims"], state["out"]):
            sim.state_device(buf)
        torch.cuda.current_stream().wait_stream(state["stream"])
        return [views(buf) for buf in state["out"]]
    if c["program"] == "advance":
        state["sim"].step(c["steps"]).sync()
        state["sim"].state_device(state["out"])
        torch.cuda.current_stream().wait_stream(state["stream"])
        return list(views(state["out"]))
    sim = make(state)
    sim.step(c["steps"]).sync()
    if c["source"] == "host":
        columns, last = sim.state()
        out = [np.stack(columns), last.view(np.int32)]
    else:
        sim.state_device(state["out"])
        torch.cuda.current_stream().wait_stream(state["stream"])
        out = list(views(state["out"]))
    records = sim.counts()
    out.append(np.array([[r["collisions"], r["edges"], r["absorbed"], r["live"]] for r in records],
                        dtype=np.int64))
    if c.get("every"):
        out.append(sim.profiles())
    sim.close()
    return out


# --------------------------------------------------------------------------- #
# what a pass cannot do without

def near(setup):
    """Partners a particle of mean speed can reach in one step, each pair once: the density
    times half a sphere of radius d0 + 2 <v> dt (half a disk in the plane)."""
    speed = setup.extra.get("speed", 1.6)
    if setup.name.startswith("spherical_blast"):
        speed = 3.0
    r = setup.d0 + 2.0 * speed * setup.dt
    if setup.planar:
        return 0.5 * setup.n / (setup.box[0] * setup.box[1]) * math.pi * r * r
    return 0.5 * setup.n / math.prod(setup.box) * 4.0 / 3.0 * math.pi * r ** 3


def work(case):
    """Per step every particle's state (six binary64 and the last partner) is read and written
    once and its reachable partners are tested (18 operations); a pass reads its input arrays
    and writes the state it returns once."""
    setups = member_setups(case, 1) if case["program"] == "group" else [setup_of(case, 1)]
    total = {"bytes": 0.0, "flops": 0.0}
    for s in setups:
        total["bytes"] += s.n * (104.0 * case["steps"] + 52.0 + (48.0 if case["program"] == "job" else 0.0))
        total["flops"] += s.n * case["steps"] * (12.0 + 18.0 * near(s))
    return total


# --------------------------------------------------------------------------- #
# the same pass in plain torch, binary64

MOST_PAIRS = 2e10  # pairs examined per exact(): some seconds


def exact(case, seed):
    c = dict(case)
    if c["gas"] in ("blast", "plane", "gas"):
        return None  # drawn on the device, or steps that follow a long warm-up
    setups = member_setups(c, seed) if c["program"] == "group" else [setup_of(c, seed)]
    pairs = sum(s.n * 14.0 * s.n / math.prod(s.box) * (s.d0 + 11.0 * s.dt) ** 3 for s in setups)
    if pairs * c["steps"] > MOST_PAIRS:
        return None
    members = []
    for s in setups:
        state = arrays_of(s, s.seed)
        last = torch.full((s.n,), -1, dtype=torch.int64, device="cuda")
        records, profiles = [], []
        for step in range(c["steps"]):
            records.append(reference_step(s, state, last, step))
            if s.profile_every and (step + 1) % s.profile_every == 0:
                profiles.append(reference_profile(s, state, last))
        member = [torch.stack(state), last.to(torch.int32)]
        if c["program"] == "job":
            member.append(np.array(records, dtype=np.int64))
            if c.get("every"):
                member.append(torch.stack(profiles))
        members.append(member)
    return members if c["program"] == "group" else members[0]


def reference_step(s, state, last, step):
    """One step in place; returns (collisions, candidate pairs, absorbed, live)."""
    i, j, d2, t = reference_candidates(s, state, last, step)
    a, b, ta = reference_matches(s.n, i, j, d2, t, s.max_rounds)
    moved = torch.zeros(s.n, dtype=torch.bool, device="cuda")
    if a.numel():
        moved[a] = moved[b] = True
        va, vb = [v[a] for v in state[3:]], [v[b] for v in state[3:]]
        if s.species is None:
            fa = fb = 0.5
            V = [(p + q) * 0.5 for p, q in zip(va, vb)]
        else:
            m = torch.tensor(s.masses, dtype=torch.float64, device="cuda")
            m = m[torch.from_numpy(s.species).long().cuda()]
            ma, mb = m[a], m[b]
            V = [(ma * p + mb * q) / (ma + mb) for p, q in zip(va, vb)]
            fa, fb = mb / (ma + mb), ma / (ma + mb)
        g = [p - q for p, q in zip(va, vb)]
        G = torch.sqrt((g[0] * g[0] + g[1] * g[1]) + g[2] * g[2])
        ga, gb = fa * G, fb * G
        normal = reference_directions(s, a, step)
        rest = s.dt - ta
        for k in range(3):
            na, nb = V[k] + ga * normal[k], V[k] - gb * normal[k]
            xa, xb = state[k][a], state[k][b]
            state[k][a] = (xa + va[k] * ta) + na * rest
            state[k][b] = (xb + vb[k] * ta) + nb * rest
            state[3 + k][a] = na
            state[3 + k][b] = nb
    inside = last != -2
    free = inside & ~moved
    for k in range(3):
        state[k].copy_(torch.where(free, state[k] + state[3 + k] * s.dt, state[k]))
    gone = torch.zeros_like(inside)
    for k in range(3):
        if s.bc[k] == ki.ABSORB:
            gone |= inside & ((state[k] < 0.0) | (state[k] > s.box[k]))
    stay = inside & ~gone
    for k in range(3):
        reference_walls(s, k, state, stay, step)
    last[a] = torch.where(gone[a], last[a], b)
    last[b] = torch.where(gone[b], last[b], a)
    last[gone] = -2
    return int(a.numel()), int(i.numel()), int(gone.sum()), int(stay.sum())


def reference_walls(s, k, state, stay, step):
    x, v, L = state[k], state[3 + k], s.box[k]
    if s.bc[k] == ki.PERIODIC:
        y = torch.where(x >= L, x - L, x)
        z = torch.where(y < 0.0, y + L, y)
        z = torch.where((y < 0.0) & (z == L), torch.zeros_like(z), z)
        x.copy_(torch.where(stay, z, x))
    elif s.bc[k] == ki.REFLECT:
        X, u = L, 0.0
        if k == 0:
            u = s.piston_u
            X = (s.piston_x0 or L) - u * (float(step + 1) * s.dt)
        low = stay & (x < 0.0)
        x.copy_(torch.where(low, -x, x))
        v.copy_(torch.where(low, -v, v))
        high = stay & (x > X)
        x.copy_(torch.where(high, (X + X) - x, x))
        v.copy_(torch.where(high, -v - (u + u), v))


def reference_candidates(s, state, last, step):
    """Candidate pairs (i, j), their squared distance and time of closest approach.  Cells are
    at least the reach d0 + 2 max|v| dt wide; an axis with fewer than three is one cell."""
    inside = torch.nonzero(last != -2).flatten()
    pos, vel = [x[inside] for x in state[:3]], [v[inside] for v in state[3:]]
    top = float(torch.sqrt(vel[0] ** 2 + vel[1] ** 2 + vel[2] ** 2).max())
    reach = (s.d0 + 2.0 * top * s.dt) * 1.0001
    nc, cell = [], []
    for k in range(3):
        ext = float(pos[k].max()) * (1.0 + 1e-9) if s.bc[k] != ki.PERIODIC else s.box[k]
        q = min(int(ext / reach), 400)
        nc.append(q if q >= 3 else 1)
        cell.append(torch.clamp((pos[k] * (nc[k] / ext)).long(), 0, nc[k] - 1))
    key = (cell[2] * nc[1] + cell[1]) * nc[0] + cell[0]
    key, order = torch.sort(key)
    inside = inside[order]
    pos, vel, cell = [x[order] for x in pos], [v[order] for v in vel], [q[order] for q in cell]
    count = torch.bincount(key, minlength=math.prod(nc))
    start = torch.cumsum(count, 0) - count
    here = torch.arange(inside.numel(), device="cuda")
    radius = None
    if s.species is not None:
        radius = torch.tensor(s.radii, dtype=torch.float64, device="cuda")
        radius = radius[torch.from_numpy(s.species).long().cuda()][inside]
    found = []
    for dz in range(-1, 2):
        for dy in range(-1, 2):
            for dx in range(-1, 2):
                d = (dx, dy, dz)
                if (dz, dy, dx) < (0, 0, 0) or any(d[k] and nc[k] == 1 for k in range(3)):
                    continue
                valid = torch.ones_like(here, dtype=torch.bool)
                to = []
                for k in range(3):
                    q = cell[k] + d[k]
                    if s.bc[k] == ki.PERIODIC:
                        q = q % nc[k]
                    else:
                        valid &= (q >= 0) & (q < nc[k])
                        q = q.clamp(0, nc[k] - 1)
                    to.append(q)
                other = (to[2] * nc[1] + to[1]) * nc[0] + to[0]
                first, many = start[other], torch.where(valid, count[other], 0)
                if d == (0, 0, 0):
                    many = first + many - here - 1
                    first = here + 1
                found += reference_tests(s, pos, vel, inside, last, radius, here, first, many)
    if not found:
        none = torch.zeros(0, dtype=torch.int64, device="cuda")
        return none, none, none.double(), none.double()
    return [torch.cat(f) for f in zip(*found)]


def reference_tests(s, pos, vel, ids, last, radius, here, first, many):
    """The candidates among particle p and `many[p]` particles from `first[p]` on, some at a time."""
    ends = torch.cumsum(many, 0)
    total = int(ends[-1]) if ends.numel() else 0
    out, chunk = [], 1 << 25
    for at in range(0, total, chunk):
        flat = torch.arange(at, min(total, at + chunk), device="cuda")
        p = torch.searchsorted(ends, flat, right=True)
        q = first[p] + (flat - (ends[p] - many[p]))
        r2 = torch.zeros(flat.numel(), dtype=torch.float64, device="cuda")
        g2 = torch.zeros_like(r2)
        for k in range(3):
            r = image(s, k, pos[k][q] - pos[k][p])
            g = vel[k][q] - vel[k][p]
            r2 += r * r
            g2 += g * g
        keep = r2 <= (s.d0 * s.d0 + s.dt * s.dt * g2) * (1.0 + 1e-9)  # |r|^2 = t^2 |v|^2 + d^2
        p, q = p[keep], q[keep]
        r = [image(s, k, pos[k][q] - pos[k][p]) for k in range(3)]
        v = [vel[k][q] - vel[k][p] for k in range(3)]
        vv = (v[0] * v[0] + v[1] * v[1]) + v[2] * v[2]
        rv = (r[0] * v[0] + r[1] * v[1]) + r[2] * v[2]
        t = -rv / vv
        w = [r[1] * v[2] - r[2] * v[1], r[2] * v[0] - r[0] * v[2], r[0] * v[1] - r[1] * v[0]]
        d2 = ((w[0] * w[0] + w[1] * w[1]) + w[2] * w[2]) / vv
        contact = s.d0 * s.d0
        if radius is not None:
            contact = (radius[p] + radius[q]) * (radius[p] + radius[q])
        i, j = ids[p], ids[q]
        ok = (vv != 0.0) & (t >= 0.0) & (t < s.dt) & (d2 < contact)
        ok &= ~((last[i] == j) & (last[j] == i))
        out.append((i[ok], j[ok], d2[ok], t[ok]))
    return out


def image(s, k, r):
    if s.bc[k] != ki.PERIODIC:
        return r
    L, h = s.box[k], s.box[k] * 0.5
    return torch.where(r > h, r - L, torch.where(r < -h, r + L, r))


def reference_matches(n, i, j, d2, t, rounds):
    """Pairs that chose each other, round by round: (smaller id, larger id, time)."""
    free = torch.ones(n, dtype=torch.bool, device="cuda")
    a, b, ta = [i[:0]], [i[:0]], [t[:0]]
    for _ in range(rounds):
        live = free[i] & free[j]
        i, j, d2, t = i[live], j[live], d2[live], t[live]
        who, other = torch.cat([i, j]), torch.cat([j, i])
        kd, kt = torch.cat([d2, d2]), torch.cat([t, t])
        order = torch.arange(who.numel(), device="cuda")
        for k in (other, kt, kd, who):  # stable sorts, least significant key first
            order = order[torch.sort(k[order], stable=True)[1]]
        lead = who[order]
        head = torch.ones_like(lead, dtype=torch.bool)
        head[1:] = lead[1:] != lead[:-1]
        pick = torch.full((n,), -1, dtype=torch.int64, device="cuda")
        when = torch.zeros(n, dtype=torch.float64, device="cuda")
        pick[lead[head]] = other[order][head]
        when[lead[head]] = kt[order][head]
        p = lead[head]
        p = p[(pick[pick[p]] == p) & (p < pick[p])]
        a.append(p)
        b.append(pick[p])
        ta.append(when[p])
        free[p] = free[pick[p]] = False
    return torch.cat(a), torch.cat(b), torch.cat(ta)


def reference_directions(s, ids, step):
    """Unit vectors by Marsaglia's method from Philox4x32-10, counter (id, step, k, 0)."""
    mask = 0xFFFFFFFF
    out = [torch.zeros(ids.numel(), dtype=torch.float64, device="cuda") for _ in range(3)]
    todo = torch.arange(ids.numel(), device="cuda")
    for k in range(64):
        if not todo.numel():
            break
        c = [ids[todo], torch.full_like(todo, step), torch.full_like(todo, k), torch.zeros_like(todo)]
        k0, k1 = s.seed & mask, (s.seed >> 32) & mask
        for _ in range(10):
            p0, p1 = wide(c[0], 0xD2511F53), wide(c[2], 0xCD9E8D57)
            c = [p1[0] ^ c[1] ^ k0, p1[1], p0[0] ^ c[3] ^ k1, p0[1]]
            k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
        taken = torch.zeros_like(todo, dtype=torch.bool)
        for h in (0, 2):
            u1, u2 = c[h].double() * 2.0 ** -31 - 1.0, c[h + 1].double() * 2.0 ** -31 - 1.0
            q = u1 * u1 + u2 * u2
            ok = (q > 0.0) & (q < 1.0) & ~taken
            root = torch.sqrt(1.0 - q)
            n = [(u1 + u1) * root, (u2 + u2) * root, 1.0 - (q + q)]
            for e in range(3):
                out[e][todo[ok]] = n[e][ok]
            taken |= ok
        todo = todo[~taken]
    return out


def wide(a, m):
    """High and low words of the product of 32-bit words held in int64."""
    lo, hi = a & 0xFFFF, a >> 16
    low = lo * m                       # below 2^48
    high = hi * m + (low >> 16)        # below 2^49
    return high >> 16, ((high & 0xFFFF) << 16) | (low & 0xFFFF)


def reference_profile(s, state, last):
    bins = s.profile_bins
    f = state[0] * (bins / s.profile_range)
    ok = (last != -2) & (state[0] >= 0.0) & (f < bins)
    at = f[ok].long()
    rows = [torch.ones_like(f[ok])] + [v[ok] for v in state[3:]] + [v[ok] * v[ok] for v in state[3:]]
    out = torch.zeros(7, bins, dtype=torch.float64, device="cuda")
    for k, r in enumerate(rows):
        out[k].index_add_(0, at, r)
    return out.t().contiguous()
