"""Cases that time the DPD fluid step through the package's public entry points.

A case is one call pattern of a user's program: forces on a state that the
program holds, one step with a statistics read-back, a run of several steps
with the state read back, a batch of uneven boxes, a set of served requests.
Sizes, densities and parameters are those of the repository's own workloads
(the L = 8 check box, the density sweep, the paper's L = 64 benchmark, the
L = 128 box, the binary mixture, the box mix and the request stream).

``exact`` restates the method in float64 torch: Groot-Warren pair forces with
the Philox-4x32-10 pair noise of Salmon et al. (SC'11), velocity-Verlet with
the velocity predicted at the half step.

Positions read back after several steps are returned unwrapped (the image
nearest to the loaded position, as a diffusion analysis keeps them): a particle
that lies on a box face to the last bit may be read at either face.
"""

from __future__ import annotations

import math

import numpy as np
import torch

from paper_1911_04712_gb300 import batch as B
from paper_1911_04712_gb300 import dpd as D
from paper_1911_04712_gb300 import serve as S
from paper_1911_04712_gb300.workloads import box_mix, request_stream

FULL, HALF = 0, 1


def _box(name, Lx, Ly, Lz, rho, steps, stencil, a=25.0, gamma=4.5, kT=1.0, dt=0.005, noise=0,
         species=1, force="none", f=0.0, stats=False, unwrap=True):
    return {"name": name, "kind": "box", "Lx": Lx, "Ly": Ly, "Lz": Lz, "rho": rho, "steps": steps,
            "stencil": stencil, "a": a, "gamma": gamma, "kT": kT, "dt": dt, "noise": noise,
            "species": species, "force": force, "f": f, "stats": stats, "unwrap": unwrap}


def listed():
    return [
        # forces for a program that holds the state itself (no allocation in the call)
        {"name": "forces_L8", "kind": "forces", "Lx": 8.0, "Ly": 8.0, "Lz": 8.0, "rho": 3.0,
         "a": 25.0, "gamma": 4.5, "kT": 1.0, "dt": 0.005, "noise_step": 7},
        # the smallest box, monitored after every step
        _box("box_L8_step_stats", 8.0, 8.0, 8.0, 3.0, 1, FULL, stats=True, unwrap=False),
        # a small box run for a while between read-outs (default stencil)
        _box("box_L12_50_steps", 12.0, 12.0, 12.0, 3.0, 50, FULL, unwrap=False),
        # the largest boxes of a parameter sweep, run alone
        _box("box_L24_half", 24.0, 24.0, 24.0, 4.0, 20, HALF, a=40.0, gamma=6.0),
        # a channel of uneven, non-integer edges with the paper's Gaussian noise
        _box("box_ragged_gauss", 41.3, 27.7, 33.9, 3.0, 20, FULL, noise=1, force="poiseuille",
             f=0.05),
        # the density sweep's dense end, constant body force (default stencil)
        _box("box_L48_rho10", 48.0, 48.0, 48.0, 10.0, 10, FULL, a=7.5, force="constant", f=0.05),
        # a binary mixture with a cut-off for each pair of species
        _box("mixture_L64_half", 64.0, 64.0, 64.0, 3.0, 10, HALF, species=2),
        # the paper's weak-scaling box: L = 64, rho = 8, periodic Poiseuille force
        _box("paper_L64_rho8_half", 64.0, 64.0, 64.0, 8.0, 10, HALF, a=50.0, gamma=20.0, dt=0.002,
             force="poiseuille", f=0.05),
        # the default, bitwise reproducible stencil on a large box
        _box("box_L96_full", 96.0, 96.0, 96.0, 3.0, 10, FULL),
        # the benchmark's box: 6.3 million particles
        _box("box_L128_half", 128.0, 128.0, 128.0, 3.0, 20, HALF),
        # 512 uneven boxes stepped together, statistics of each, a few followed closely
        {"name": "batch_mix512_half", "kind": "batch", "boxes": 512, "mix": 0, "steps": 20,
         "stencil": HALF, "follow": 8},
        # a burst of served requests (default stencil), each from its own state
        {"name": "served_16", "kind": "served", "requests": 16, "mix": 0, "steps": 64,
         "stencil": FULL},
    ]


def draw(rng):
    kind = rng.choices(["box", "forces", "batch", "served"], [60, 14, 14, 12])[0]
    rnd = lambda lo, hi: round(rng.uniform(lo, hi), 2)  # noqa: E731
    log = lambda lo, hi: math.exp(rng.uniform(math.log(lo), math.log(hi)))  # noqa: E731
    if kind == "forces":
        rho = rng.choice([3.0, 4.0, 5.0])
        edges = [round(log(4, (32000 / rho) ** (1 / 3) / 1.08), 1) for _ in range(3)]
        return {"kind": kind, "Lx": edges[0], "Ly": edges[1], "Lz": edges[2], "rho": rho,
                "a": rnd(10, 80), "gamma": rnd(2, 8), "kT": rnd(0.5, 2), "dt": 0.005,
                "noise_step": rng.randrange(1000)}
    if kind == "batch":
        return {"kind": kind, "boxes": int(log(8, 512)), "mix": rng.randrange(1, 1000),
                "steps": rng.randrange(5, 21), "stencil": rng.choice([FULL, HALF, HALF]),
                "follow": 4}
    if kind == "served":
        return {"kind": kind, "requests": rng.randrange(4, 25), "mix": rng.randrange(1, 1000),
                "steps": rng.randrange(40, 81), "stencil": rng.choice([FULL, HALF])}
    rho = rng.choice([3.0, 3.0, 4.0, 5.0, 8.0, 10.0])
    n = log(1000, 5.5e6)  # spread over the particle counts
    edge = (n / rho) ** (1 / 3)
    cube = rng.random() < 0.5
    edges = [max(4.0, float(round(edge)) if cube else round(edge * rng.uniform(0.9, 1.1), 1))
             for _ in range(3)]
    n = rho * edges[0] * edges[1] * edges[2]
    steps = rng.randrange(1, 21) if n > 2e5 else rng.randrange(1, 51)
    noise, species = rng.choices([(0, 1), (1, 1), (0, 2)], [70, 15, 15])[0]
    force = rng.choice(["none", "none", "constant", "poiseuille"])
    c = _box("", *edges, rho, steps, rng.choice([FULL, HALF]), a=rnd(10, 60), gamma=rnd(2, 20),
             kT=rnd(0.5, 1.5), dt=rng.choice([0.002, 0.005, 0.005]), noise=noise, species=species,
             force=force, f=0.0 if force == "none" else 0.05, stats=rng.random() < 0.3,
             unwrap=n > 8000)
    del c["name"]
    return c


# ------------------------------------------------------------------ inputs
def _edges(c):
    return (c["Lx"], c["Ly"], c["Lz"])


def _state(L, n, kT, seed):
    """Uniform positions and Maxwellian velocities with zero mean (float32, CUDA)."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    L = torch.tensor(L, dtype=torch.float32, device="cuda")
    x = torch.rand((n, 3), generator=g, device="cuda") * L
    x = torch.where(x >= L, torch.zeros_like(x), x)
    v = torch.randn((n, 3), generator=g, device="cuda") * math.sqrt(kT)
    return x, v - v.mean(0)


def _count(c):
    return int(round(c["rho"] * c["Lx"] * c["Ly"] * c["Lz"]))


# the bench's binary mixture: own repulsion and cut-off between unlike species
MIX_A = np.array([[25.0, 40.0], [40.0, 25.0]])
MIX_G = np.array([[4.5, 4.5], [4.5, 4.5]])
MIX_RC = np.array([[1.0, 0.9], [0.9, 1.0]])


def _batch_specs(c):
    return box_mix(c["boxes"], master_seed=c["mix"], steps=0)


def _followed(c):
    k = c["follow"]
    return sorted({(2 * i + 1) * c["boxes"] // (2 * k) for i in range(k)})


def _request_specs(c):
    return request_stream(c["requests"], master_seed=c["mix"])


def _seeded(seed, k):
    return (int(seed) * 1009 + 7919 * k) % (1 << 31)


def prepare(case, seed):
    c = dict(case)
    if c["kind"] in ("box", "forces"):
        L, n = _edges(c), _count(c)
        x, v = _state(L, n, c["kT"], _seeded(seed, 0))
        st = {"case": c, "x": x, "v": v, "seed": int(seed)}
        if c["kind"] == "forces":
            return st
        box = D.Box(L, a=c["a"], gamma=c["gamma"], kT=c["kT"], dt=c["dt"], seed=int(seed),
                    stencil=c["stencil"], noise=c["noise"],
                    body_force=c["f"] if c["force"] == "constant" else None,
                    poiseuille_f=c["f"] if c["force"] == "poiseuille" else None)
        if c["species"] > 1:
            box.set_species(MIX_A, MIX_G, MIX_RC)
            box.set_state(x, v, species=(torch.arange(n, device="cuda") % 2).to(torch.int32))
        else:
            box.set_state(x, v)
        return st | {"box": box, "L": torch.tensor(L, dtype=torch.float32, device="cuda")}
    if c["kind"] == "batch":
        specs = _batch_specs(c)
        states = [_state((s.L,) * 3, s.n, s.kT, _seeded(seed, k)) for k, s in enumerate(specs)]
        b = B.Batch([B.make_desc(s.L, s.n, a=s.a, gamma=s.gamma, kT=s.kT, dt=s.dt, seed=s.seed)
                     for s in specs], stencil=c["stencil"])
        for k, (x, v) in enumerate(states):
            b.set_state(k, x, v)
        follow = {k: (states[k][0].cpu().numpy(), np.float32(specs[k].L)) for k in _followed(c)}
        b.step(0)
        return {"case": c, "batch": b, "follow": follow}
    specs = _request_specs(c)
    q = S.Queue(int(120e9), chunk_steps=100, sample_every=20, nbins=16, stencil=c["stencil"])
    runs = []
    for k, s in enumerate(specs):
        x, v = _state((s.L,) * 3, s.n, s.kT, _seeded(seed, k))
        req = S.make_request(s.L, n=s.n, a=s.a, gamma=s.gamma, kT=s.kT, dt=s.dt, seed=s.seed,
                             steps=c["steps"])
        runs.append((req, x.cpu().numpy(), v.cpu().numpy(), s))
    return {"case": c, "queue": q, "runs": runs}


# --------------------------------------------------------------------- run
def _unwrapped(x, x0, L, rnd):
    d = x - x0
    d -= rnd(d / L) * L
    d += x0
    return d


THERMO = ("kinetic", "kT", "virial", "pressure")


def run(state):
    c = state["case"]
    if c["kind"] == "forces":
        return D.forces_noalloc(state["x"], state["v"], _edges(c), a=c["a"], gamma=c["gamma"],
                                kT=c["kT"], dt=c["dt"], seed=state["seed"], step=c["noise_step"])
    if c["kind"] == "box":
        box, out = state["box"], {}
        box.step(c["steps"])
        if c["stats"]:
            s = box.stats()
            out = {k: s[k] for k in THERMO}
        x, out["vel"] = box.get_state(device=True)
        out["pos"] = _unwrapped(x, state["x"], state["L"], torch.round) if c["unwrap"] else x
        return out
    if c["kind"] == "batch":
        b = state["batch"]
        b.step(c["steps"])
        s = b.stats()
        out = {k: np.array([q[k] for q in s]) for k in THERMO}
        for k, (x0, L) in state["follow"].items():
            x, v = b.get_state(k)
            out["box%d" % k] = {"pos": _unwrapped(x, x0, L, np.round), "vel": v}
        return out
    q = state["queue"]
    tickets = [q.submit_state(req, x, v, keep_final=True) for req, x, v, _ in state["runs"]]
    q.wait_all()
    done = [q.result(t) for t in tickets]
    out = {k: np.array([r[k] for r in done]) for k in ("samples", "kT_mean", "pressure_mean")}
    for k, (t, (_, x0, _, s)) in enumerate(zip(tickets, state["runs"])):
        x, v = q.final_state(t, s.n)
        out["run%d" % k] = {"pos": _unwrapped(x, x0, np.float32(s.L), np.round), "vel": v}
    return out


# -------------------------------------------------------------------- work
# One candidate of the 27-cell stencil is a squared distance and a compare (9),
# a pair within rc the force of Eqs. 2-5 (30) and a Philox-4x32-10 word (10
# rounds of two products and four xors); each counted once per pair.  A step
# reads and writes positions and velocities.
def _ops(n, rho):
    return n * (13.5 * rho * 9 + 2.0 * math.pi / 3.0 * rho * (30 + 60))


def work(case):
    c = case
    if c["kind"] == "forces":
        n = _count(c)
        return {"bytes": 36.0 * n, "flops": _ops(n, c["rho"])}
    if c["kind"] == "box":
        sizes = [(_count(c), c["rho"])]
    elif c["kind"] == "batch":
        sizes = [(s.n, s.rho) for s in _batch_specs(c)]
    else:
        sizes = [(s.n, s.rho) for s in _request_specs(c)]
    k = c["steps"]
    return {"bytes": sum(n for n, _ in sizes) * 48.0 * k,
            "flops": sum(_ops(n, rho) for n, rho in sizes) * k}


# ------------------------------------------------------------ 64-bit values
M0, M1, W0, W1 = 0xD2511F53, 0xCD9E8D57, 0x9E3779B9, 0xBB67AE85
LOW = 0xFFFFFFFF


def _words(lo, hi, step, seed):
    """Words 0 and 1 of Philox-4x32-10 on (lo, hi, step, 0) with key `seed` (int64 tensors)."""
    def product(m, c):  # 32 x 32 -> (high, low), without overflow of int64
        p0, p1 = (m & 0xFFFF) * c, (m >> 16) * c
        s = p1 + (p0 >> 16)
        return s >> 16, ((s & 0xFFFF) << 16) | (p0 & 0xFFFF)

    k0, k1 = seed & LOW, (seed >> 32) & LOW
    c0, c1 = lo, hi
    c2, c3 = torch.full_like(lo, step & LOW), torch.full_like(lo, (step >> 32) & LOW)
    for r in range(10):
        if r:
            k0, k1 = (k0 + W0) & LOW, (k1 + W1) & LOW
        h0, l0 = product(M0, c0)
        h1, l1 = product(M1, c2)
        c0, c1, c2, c3 = h1 ^ c1 ^ k0, l1, h0 ^ c3 ^ k1, l0
    return c0, c1


def _forces64(x, v, L, p, step):
    """Forces (n, 3) and the virial sum_{i<j} r_ij . F^C_ij of Eqs. 2-5 at one step."""
    n, dev = len(x), x.device
    Lt = torch.tensor(L, dtype=torch.float64, device=dev)
    y = x - torch.floor(x / Lt) * Lt
    nc = [int(math.floor(e)) for e in L]
    nct = torch.tensor(nc, device=dev)
    cell = torch.minimum((y / Lt * nct).long(), nct - 1)
    key = (cell[:, 2] * nc[1] + cell[:, 1]) * nc[0] + cell[:, 0]
    order = torch.argsort(key)
    cell, y, v = cell[order], y[order], v[order]
    count = torch.bincount(key, minlength=nc[0] * nc[1] * nc[2])
    start = torch.cumsum(count, 0) - count
    slot = torch.arange(n, device=dev)
    F = torch.zeros((n, 3), dtype=torch.float64, device=dev)
    vir = torch.zeros((), dtype=torch.float64, device=dev)
    spec = (order % 2) if p["species"] > 1 else None
    offsets = [(dx, dy, dz) for dz in (0, 1) for dy in (-1, 0, 1) for dx in (-1, 0, 1)
               if (dz, dy, dx) >= (0, 0, 0)]
    for off in offsets:
        nb = (cell + torch.tensor(off, device=dev)) % nct
        nb = (nb[:, 2] * nc[1] + nb[:, 1]) * nc[0] + nb[:, 0]
        first, m = start[nb], count[nb]
        if off == (0, 0, 0):  # the own cell: later slots only
            m = first + m - slot - 1
            first = slot + 1
        i = torch.repeat_interleave(slot, m)
        j = torch.arange(len(i), device=dev) - torch.repeat_interleave(torch.cumsum(m, 0) - m, m)
        j += first[i]
        d = y[i] - y[j]
        d -= torch.round(d / Lt) * Lt
        r2 = (d * d).sum(1)
        keep = ((r2 < 1.0) & (r2 > 0.0)).nonzero()[:, 0]
        i, j, d, r = i[keep], j[keep], d[keep], torch.sqrt(r2[keep])
        a, gam, rc = p["a"], p["gamma"], 1.0
        if spec is not None:
            tab = [torch.tensor(t, device=dev)[spec[i], spec[j]] for t in (MIX_A, MIX_G, MIX_RC)]
            a, gam, rc = tab
        w = torch.clamp(1.0 - r / rc, min=0.0)
        ids = (torch.minimum(order[i], order[j]), torch.maximum(order[i], order[j]))
        u0, u1 = _words(*ids, step, p["seed"])
        U0 = ((u0 >> 8).double() + 0.5) / 2.0 ** 24
        if p["noise"]:
            U1 = ((u1 >> 8).double() + 0.5) / 2.0 ** 24
            xi = torch.sqrt(-2.0 * torch.log(U0)) * torch.cos(2.0 * math.pi * U1)
        else:
            xi = math.sqrt(3.0) * (2.0 * U0 - 1.0)
        e = d / r[:, None]
        ev = (e * (v[i] - v[j])).sum(1)
        sigma = torch.sqrt(2.0 * torch.as_tensor(gam, dtype=torch.float64, device=dev) * p["kT"])
        fc = a * w
        f = (fc - gam * w * w * ev + sigma * w * xi / math.sqrt(p["dt"]))[:, None] * e
        F.index_add_(0, i, f)
        F.index_add_(0, j, -f)
        vir += (fc * r).sum()
    if p["force"] != "none":
        f = torch.full((n,), float(p["f"]), dtype=torch.float64, device=dev)
        if p["force"] == "poiseuille":
            f = torch.where(y[:, 0] <= 0.5 * L[0], -f, f)
        F[:, 2] += f
    out = torch.empty_like(F)
    out[order] = F
    return out, vir


def _run64(x, v, L, p, steps):
    """Unwrapped positions, full-step velocities and thermodynamics after `steps` steps."""
    x, v, h = x.double(), v.double(), 0.5 * p["dt"]
    F, vir = _forces64(x, v, L, p, 0)
    samples = []
    for k in range(1, steps + 1):
        v = v + h * F
        x = x + p["dt"] * v
        F, vir = _forces64(x, v, L, p, k)
        v = v + h * F
        n, V = len(x), L[0] * L[1] * L[2]
        kin = 0.5 * (v * v).sum()
        kT = 2.0 * kin / (3.0 * (n - 1))
        samples.append((kin, kT, vir, n * kT / V + vir / (3.0 * V)))
    return x, v, samples


def _pars(a, gamma, kT, dt, seed, noise=0, species=1, force="none", f=0.0):
    return {"a": a, "gamma": gamma, "kT": kT, "dt": dt, "seed": int(seed), "noise": noise,
            "species": species, "force": force, "f": f}


def exact(case, seed):
    c = dict(case)
    if c["kind"] in ("box", "forces"):
        L, n = _edges(c), _count(c)
        x, v = _state(L, n, c["kT"], _seeded(seed, 0))
        if c["kind"] == "forces":
            p = _pars(c["a"], c["gamma"], c["kT"], c["dt"], seed)
            return _forces64(x.double(), v.double(), L, p, c["noise_step"])[0]
        if n * c["steps"] * c["rho"] > 3.2e8:
            return None
        p = _pars(c["a"], c["gamma"], c["kT"], c["dt"], seed, c["noise"], c["species"], c["force"],
                  c["f"])
        xs, vs, samples = _run64(x, v, L, p, c["steps"])
        out = {"vel": vs, "pos": xs if c["unwrap"] else xs - torch.floor(
            xs / torch.tensor(L, device=xs.device)) * torch.tensor(L, device=xs.device)}
        if c["stats"]:
            out |= {k: float(q) for k, q in zip(THERMO, samples[-1])}
        return out
    if c["kind"] == "batch":
        specs, out = _batch_specs(c), {k: None for k in THERMO}
        for k in _followed(c):
            s = specs[k]
            x, v = _state((s.L,) * 3, s.n, s.kT, _seeded(seed, k))
            p = _pars(s.a, s.gamma, s.kT, s.dt, s.seed)
            xs, vs, _ = _run64(x, v, (s.L,) * 3, p, c["steps"])
            out["box%d" % k] = {"pos": xs, "vel": vs}
        return out
    out, means = {"samples": None}, []
    for k, s in enumerate(_request_specs(c)):
        if c["requests"] * c["steps"] > 1400:  # the float64 runs would take too long
            return None
        x, v = _state((s.L,) * 3, s.n, s.kT, _seeded(seed, k))
        p = _pars(s.a, s.gamma, s.kT, s.dt, s.seed)
        xs, vs, samples = _run64(x, v, (s.L,) * 3, p, c["steps"])
        taken = [q for m, q in enumerate(samples, 1) if m > c["steps"] // 2 and m % 20 == 0]
        means.append([sum(float(q[f]) for q in taken) / len(taken) for f in (1, 3)])
        out["run%d" % k] = {"pos": xs, "vel": vs}
    return out | {"kT_mean": np.array([m[0] for m in means]),
                  "pressure_mean": np.array([m[1] for m in means])}
