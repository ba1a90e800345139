"""Performance cases: what users of the MD library have it do, through its public calls.

Every case is one pass of a program that holds a handle (md.System) or device buffers:

  md       sim.step(n), then the samples, the per-step energies and the state are read back: the
           production loop of every study here (paper Sec. 3-5), in the three precision modes, for the
           monatomic fluid and the Kob-Andersen mixture, plain or smoothed (Sec. 4), one system or an
           ensemble of replicas, free (NVE) or with a heat bath or rescaling between stretches (Sec. 2.3)
  corr     the same loop with a time-correlation sample after every stretch (Sec. 2.5)
  forces   a configuration from the host in, forces, energies and totals out
  noalloc  forces of device arrays by the call that needs no handle and no workspace

Inputs are liquids: a small periodic box is melted and brought to the case's temperature here, in plain
torch (dense, deterministic), repeated to the size wanted, thinned at random to the exact particle count,
and given fresh Maxwell-Boltzmann velocities, all from the seed.  A pass covers at most about 0.3 units of
reduced time, so that rounding differences have not grown by the fluid's chaos when two passes are compared.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_0912_3824_gb300 import md, synth

DEV = "cuda"


# --------------------------------------------------------------------------------------------------
# the cases
# --------------------------------------------------------------------------------------------------
def _md(name, pot, n, density, temperature, dt, steps, precision, **more):
    c = {"name": name, "kind": "md", "pot": pot, "n": n, "density": density, "temperature": temperature,
         "dt": dt, "steps": steps, "precision": precision, "skin": 0.3, "smooth": 0.0, "replicas": 1,
         "bath": "none", "sample": 20}
    c.update(more)
    return c


def listed():
    return [
        # the textbook argon-like fluid at its smallest: a call is launches and latency
        _md("lj864_mixed", "lj", 864, 0.8442, 0.722, 0.005, 40, "mixed"),
        # glass-former at the size of exploratory runs, default parameters
        _md("ka16384_mixed", "ka", 16384, 1.2, 0.7, 0.001, 200, "mixed"),
        # the headline system: 65,536 particles of the mixture, at the skin that tuning finds for it
        _md("ka65536_mixed", "ka", 65536, 1.2, 0.5, 0.001, 250, "mixed", skin=0.2, sample=50),
        # an odd size beyond one wave of blocks
        _md("lj250047_mixed", "lj", 250047, 0.8442, 1.0, 0.002, 100, "mixed"),
        # the largest of the size sweep: lists far larger than the L2
        _md("lj1048576_mixed", "lj", 1048576, 0.8442, 1.0, 0.002, 100, "mixed"),
        # dilute supercritical fluid in single precision: few neighbours, wide skin (the Sec. 3 measurement)
        _md("lj87808_sparse_fp32", "lj", 87808, 0.4, 1.5, 0.001, 200, "fp32", skin=0.5),
        # the double-precision runs that energy drift is judged against
        _md("ka16384_fp64", "ka", 16384, 1.2, 0.7, 0.001, 60, "fp64"),
        # the smoothed potential of the stability study
        _md("lj10000_smooth_mixed", "lj", 10000, 0.75, 1.12, 0.001, 200, "mixed", smooth=0.005),
        # an ensemble of independent systems of uneven size in one handle, kept at temperature
        _md("ka_replicas64_mixed", "ka", 0, 1.2, 0.7, 0.001, 60, "mixed", replicas=64, bath="rescale"),
        # equilibration with the heat bath and tagged-particle correlations along the way
        {"name": "ka20011_corr_mixed", "kind": "corr", "pot": "ka", "n": 20011, "density": 1.2, "temperature": 0.7,
         "dt": 0.001, "stride": 10, "samples": 30, "blocks": 2, "length": 5, "nq": 16, "precision": "mixed",
         "skin": 0.3, "bath": "andersen"},
        # forces of configurations that come from outside: binning, list build, force, back to the host
        {"name": "ka50000_forces_mixed", "kind": "forces", "pot": "ka", "n": 50000, "density": 1.2,
         "temperature": 0.7, "precision": "mixed", "skin": 0.3, "smooth": 0.0},
        # forces on the device from a program that may allocate nothing
        {"name": "ka6000_noalloc_mixed", "kind": "noalloc", "pot": "ka", "n": 6000, "density": 1.2,
         "temperature": 0.7, "precision": "mixed"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["md"] * 6 + ["replicas", "corr", "forces", "noalloc"])
    pot = rng.choice(["lj", "ka"])
    precision = rng.choice(["mixed", "mixed", "mixed", "fp32", "fp64"])
    ka = pot == "ka"
    density = 1.2 if ka else round(rng.choice([rng.uniform(0.2, 0.6), rng.uniform(0.7, 0.9)]), 4)
    temperature = round(rng.uniform(0.5, 1.5) if ka else rng.uniform(0.8, 1.5) if density > 0.65 else
                        rng.uniform(1.4, 2.0), 3)
    dt = 0.001 if ka else rng.choice([0.001, 0.002, 0.004])
    skin = rng.choice([0.2, 0.3, 0.3, 0.4])
    most = 65536 if precision == "fp64" else 350000
    if kind == "noalloc":
        return {"kind": "noalloc", "pot": pot, "n": _log_int(rng, 200, 12000), "density": density,
                "temperature": temperature, "precision": precision}
    if kind == "forces":
        return {"kind": "forces", "pot": pot, "n": _log_int(rng, 500, 200000 if precision != "fp64" else 50000),
                "density": density, "temperature": temperature, "precision": precision, "skin": skin,
                "smooth": rng.choice([0.0, 0.0, 0.005])}
    if kind == "corr":
        return {"kind": "corr", "pot": pot, "n": _log_int(rng, 600, 60000), "density": density,
                "temperature": temperature, "dt": dt, "stride": rng.choice([5, 10, 15]), "samples": 15,
                "blocks": 2, "length": rng.choice([4, 6, 7]), "nq": rng.choice([1, 8, 16, 31]),
                "precision": "mixed" if precision == "fp64" else precision, "skin": skin,
                "bath": rng.choice(["none", "andersen"])}
    replicas = rng.choice([3, 9, 40]) if kind == "replicas" else 1
    n = 0 if replicas > 1 else _log_int(rng, 500, most)
    steps = max(20, int(round(0.2 / dt)))
    if precision == "fp64":
        steps = min(steps, 60)
    if replicas > 9:
        steps = min(steps, 80)
    c = _md("", pot, n, density, temperature, dt, steps, precision, skin=skin,
            smooth=rng.choice([0.0, 0.0, 0.0, 0.005]), replicas=replicas,
            bath=rng.choice(["none", "none", "rescale", "andersen"]), sample=rng.choice([7, 20, 50]))
    del c["name"]
    return c


# --------------------------------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------------------------------
def _params(case):
    return (synth.ka_params if case["pot"] == "ka" else synth.lj_params)(smooth=case.get("smooth", 0.0))


def _tables(p):
    """Per-pair constants [2, 2] on the device, in double."""
    eps, sig, rc = (torch.tensor(p[k], dtype=torch.float64, device=DEV) for k in ("eps", "sigma", "rcut"))
    s6 = (sig / rc) ** 6
    return eps, sig * sig, rc, 4.0 * eps * (s6 * s6 - s6), sig


def _melt(pot, n, box, temperature, seed):
    """Liquid positions [n, 3] and species [n] in a periodic box, from dense pair sums (deterministic)."""
    p = synth.ka_params() if pot == "ka" else synth.lj_params()
    s = synth.perturb(synth.make_system(n, n / box ** 3, max(temperature, 0.1), seed, p), 0.1, seed + 1)
    x = torch.from_numpy(s.pos).to(DEV)
    v = torch.from_numpy(s.vel).to(DEV)
    sp = torch.from_numpy(s.species.astype(np.int64)).to(DEV)
    eps, sig2, rc, _, _ = _tables(p)
    ab = sp[:, None] * 2 + sp[None, :]
    e48, s2, r2c = 48.0 * eps.reshape(-1)[ab], sig2.reshape(-1)[ab], (rc * rc).reshape(-1)[ab]
    s2.fill_diagonal_(0.0)                                    # no self interaction

    def force():
        d = x[:, None, :] - x[None, :, :]
        d -= box * torch.round(d / box)
        r2 = (d * d).sum(-1)
        u = (s2 / r2.clamp_min(0.5)) ** 3                     # softened core: the start is a crystal with holes
        f = torch.where(r2 < r2c, e48 * u * (u - 0.5) / r2.clamp_min(0.5), 0.0)
        return (f[:, :, None] * d).sum(1)

    dt, f = 0.003, force()
    for k in range(420):
        v += 0.5 * dt * f
        x += dt * v
        f = force()
        v += 0.5 * dt * f
        t = temperature if k >= 200 else 3.0 + 2.0 * temperature
        v *= torch.sqrt(t * (3 * n - 3) / (v * v).sum())
    return torch.remainder(x, box).cpu().numpy(), s.species


def _liquid(case, n, seed):
    """n particles of the case's fluid at its density: (box, species, pos)."""
    box = (n / case["density"]) ** (1.0 / 3.0)
    m = max(1, min(int(box / 6.0), int(round((n / 500.0) ** (1.0 / 3.0)))))
    n0 = -(-n // m ** 3)
    tile = box / m
    x, sp = _melt(case["pot"], n0, tile, case["temperature"], seed)
    g = np.stack(np.meshgrid(*(np.arange(m),) * 3, indexing="ij"), -1).reshape(-1, 3)
    pos = (x[None, :, :] + tile * g[:, None, :]).reshape(-1, 3)
    species = np.tile(sp, m ** 3)
    keep = np.sort(np.random.RandomState(seed % 2 ** 31).permutation(len(pos))[:n])
    return box, species[keep].astype(np.int32), pos[keep]


def _velocities(n, temperature, mass, seed):
    r = np.random.RandomState((seed + 77) % 2 ** 31)
    v = r.standard_normal((n, 3))
    v -= v.mean(axis=0)
    return v * math.sqrt(temperature * (3 * n - 3) / float((v * v).sum()))


def _kinds(case):
    """How many different sizes an ensemble has."""
    return max(3, min(16, case["replicas"] // 4))


def _input(case, seed):
    """(n per replica, box per replica, species, pos, vel) in the order the handle gets them."""
    if case.get("replicas", 1) == 1:
        box, sp, x = _liquid(case, case["n"], seed)
        v = _velocities(case["n"], case["temperature"], 1.0, seed)
        return [case["n"]], [box], sp, x, v
    # an ensemble: a few uneven sizes, each a melted box that its replicas take turned, shifted and with
    # velocities of their own
    r = np.random.RandomState((seed + 5) % 2 ** 31)
    kinds = _kinds(case)
    made = [_liquid(case, n, seed + 11 * k) for k, n in enumerate(synth.ensemble_sizes(kinds))]
    n, boxes, sp, xs, vs = [], [], [], [], []
    for k in range(case["replicas"]):
        box, s, x = made[k % kinds]
        x = np.mod(x[:, r.permutation(3)] + r.random_sample(3) * box, box)
        n.append(len(x))
        boxes.append(box)
        sp.append(s)
        xs.append(np.where(x >= box, 0.0, x))
        vs.append(_velocities(len(x), case["temperature"], 1.0, seed + 1000 + k))
    return n, boxes, np.concatenate(sp), np.concatenate(xs), np.concatenate(vs)


def prepare(case, seed):
    n, box, sp, x, v = _input(case, seed)
    prec = md.PRECISIONS[case["precision"]]
    s = {"case": case, "seed": seed}
    if case["kind"] == "noalloc":
        s["p"] = md.make_params(_params(case), 0.001, precision=prec)
        s["box"] = box[0]
        s["species"] = torch.from_numpy(sp).to(DEV)
        s["pos"] = torch.from_numpy(x).to(DEV)
        return s
    p = md.make_params(_params(case), case.get("dt", 0.001), skin=case["skin"], precision=prec,
                       sample_interval=case.get("sample", 20))
    s["sim"] = md.System(p, n, box, sp, x, v)
    s["edge"] = box[0] if len(box) == 1 else np.repeat(np.asarray(box), n)[:, None]
    s["event"] = 0
    if case["kind"] == "forces":
        s["pos"], s["vel"] = np.mod(x + 0.02, box[0]), v
        return s
    if case["kind"] == "corr":
        q = synth.shell_wavevectors(box[0], 7.25, case["nq"], seed % 1000)
        s["corr"] = md.Correlator(s["sim"], case["blocks"], case["length"], q)
    s["sim"].observables()                                     # drop the sample and energy of the creation
    s["sim"].epot_series()
    return s


# --------------------------------------------------------------------------------------------------
# one pass
# --------------------------------------------------------------------------------------------------
def _stretches(case):
    """MD steps between the calls of the bath (NVE: one stretch)."""
    if case["bath"] == "none":
        return [case["steps"]]
    k = case["steps"] // 3
    return [k, k, case["steps"] - 2 * k]


def _bath(state):
    """What keeps the temperature, before a stretch."""
    case, sim = state["case"], state["sim"]
    if case["bath"] == "rescale":
        sim.rescale(case["temperature"])
    elif case["bath"] == "andersen":
        sim.andersen(case["temperature"], state["seed"] & 0xFFFF, state["event"])
        state["event"] += 1


def _read(state):
    sim = state["sim"]
    obs = sim.observables()
    steps, e = sim.epot_series()
    pos, vel, img = sim.get_state()
    return {"obs": [np.ascontiguousarray(obs[k]) for k in ("step", "e_pot", "e_kin", "virial", "w")],
            "steps": steps, "e_pot": e, "unwrapped": pos + state["edge"] * img, "vel": vel}


def run(state):
    case = state["case"]
    if case["kind"] == "noalloc":
        n = case["n"]
        f = torch.empty(n, 3, dtype=torch.float64, device=DEV)
        e = torch.empty(n, dtype=torch.float64, device=DEV)
        t = torch.empty(8, dtype=torch.float64, device=DEV)
        md.md_forces_noalloc(state["p"], n, state["box"], state["species"].data_ptr(), state["pos"].data_ptr(),
                             f.data_ptr(), e.data_ptr(), t.data_ptr(), torch.cuda.current_stream().cuda_stream)
        return {"f": f, "e": e, "totals": t}
    sim = state["sim"]
    if case["kind"] == "forces":
        sim.set_state(state["pos"], state["vel"])
        f, e, tot = sim.forces()
        return {"f": f, "e": e, "totals": [np.ascontiguousarray(tot[k]) for k in ("e_pot", "e_kin", "virial", "w")]}
    if case["kind"] == "corr":
        _bath(state)
        for _ in range(case["samples"]):
            state["corr"].sample()
            sim.step(case["stride"])
        lags, msd, fs, origins = state["corr"].result()
        out = _read(state)
        out["corr"] = [lags, msd, fs, origins]
        return out
    for k in _stretches(case):
        _bath(state)
        sim.step(k)
    return _read(state)


# --------------------------------------------------------------------------------------------------
# the work of a pass, and how close another correct implementation comes
# --------------------------------------------------------------------------------------------------
def _count(case):
    """(particles, mean number of partners within the cutoff)."""
    n, k = case["n"], case.get("replicas", 1)
    if k > 1:
        sizes = synth.ensemble_sizes(_kinds(case))
        n = sum(sizes[i % len(sizes)] for i in range(k))
    p = _params(case)
    mix = (0.8, 0.2) if case["pot"] == "ka" else (1.0, 0.0)
    rc3 = sum(mix[a] * mix[b] * p["rcut"][a][b] ** 3 for a in range(2) for b in range(2))
    return n, 4.0 / 3.0 * math.pi * rc3 * case["density"]


def work(case):
    n, nb = _count(case)
    wide = 8 if case["precision"] != "fp32" else 4               # bytes of a state word
    if case["kind"] == "noalloc":
        return {"bytes": n * (28 + 32), "flops": n * (n - 1) * 15.0 + n * nb * 38.0}
    if case["kind"] == "forces":
        return {"bytes": n * (48 + 32), "flops": n * nb * (15.0 + 38.0)}
    steps = case["steps"] if case["kind"] == "md" else case["stride"] * case["samples"]
    flops = steps * n * (nb * 38.0 + 60.0)
    nbytes = n * (12.0 * wide + 60.0)                             # the state in, and out to the host
    if case["kind"] == "corr":
        m = sum(max(0, (case["samples"] - 1) // case["length"] ** b + 2 - case["length"]) for b in range(case["blocks"]))
        flops += m * (case["length"] - 1) * n * (8.0 + case["nq"] * 8.0)
        nbytes += case["samples"] * n * 24.0
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    """Four times what the same passes give with their force sums in other orders (1, 2 and 8 lanes per
    particle), the second pass on a state included: mixed 9e-7 (largest single value 9e-5), single 6e-6
    (3e-4), double 7e-15 (3e-13); forces alone 6e-8 mixed, 1e-6 from 64 bits.  On top, in the modes whose pair
    distances are single precision, a pair that rounding moves across the cutoff, where the force jumps by up
    to 0.073: one step's kick is 0.073 dt, seen in the norm as 0.1 dt / sqrt(N T)."""
    p = case["precision"]
    if case["kind"] in ("forces", "noalloc"):
        # a pair on the other side of the cutoff: 0.073 against forces of about 30 sqrt(N) in the norm
        return {"rel": 1e-12, "max": 1e-10} if p == "fp64" else \
            {"rel": (4e-6 if p == "mixed" else 4e-5) + 0.01 / math.sqrt(case["n"]), "max": 0.01}
    if p == "fp64":
        return {"rel": 1e-12, "max": 1e-10}
    flip = 0.2 * case["dt"] / math.sqrt(_count(case)[0])
    return {"rel": (4e-6 if p == "mixed" else 4e-5) + flip, "max": (4e-4 if p == "mixed" else 2e-3) + 0.4 * case["dt"]}


# --------------------------------------------------------------------------------------------------
# the same in 64 bits, in plain torch
# --------------------------------------------------------------------------------------------------
def _near(x, box, reach):
    """Pairs (i < j) of one periodic box closer than `reach`: dense for small boxes, by cells otherwise."""
    n = x.shape[0]
    nc = int(box / reach)
    found = []
    if nc < 4:
        rows = max(1, 40_000_000 // n)
        for a in range(0, n, rows):
            d = x[a:a + rows, None, :] - x[None, :, :]
            d -= box * torch.round(d / box)
            i, j = torch.nonzero((d * d).sum(-1) < reach * reach, as_tuple=True)
            i = i + a
            found.append(torch.stack([i, j])[:, i < j])
        return torch.cat(found, 1)
    c = (x * (nc / box)).long().clamp_(0, nc - 1)
    cell = (c[:, 0] * nc + c[:, 1]) * nc + c[:, 2]
    order = torch.argsort(cell)
    count = torch.bincount(cell, minlength=nc ** 3)
    first = torch.cumsum(count, 0) - count
    cap = int(count.max())
    slot = torch.arange(n, device=x.device) - first[cell[order]]
    table = torch.full((nc ** 3, cap), -1, dtype=torch.long, device=x.device)
    table[cell[order], slot] = order
    every = torch.arange(nc ** 3, device=x.device)
    cx, cy, cz = every // (nc * nc), every // nc % nc, every % nc
    rows = max(1, 30_000_000 // (cap * cap))
    for k in range(27):
        other = ((cx + k // 9 - 1) % nc * nc + (cy + k // 3 % 3 - 1) % nc) * nc + (cz + k % 3 - 1) % nc
        for a in range(0, nc ** 3, rows):
            ti, tj = table[a:a + rows], table[other[a:a + rows]]
            d = x[ti.clamp_min(0)][:, :, None, :] - x[tj.clamp_min(0)][:, None, :, :]
            d -= box * torch.round(d / box)
            hit = ((d * d).sum(-1) < reach * reach) & (ti[:, :, None] >= 0) & (ti[:, :, None] < tj[:, None, :])
            r, u, w = torch.nonzero(hit, as_tuple=True)
            found.append(torch.stack([ti[r, u], tj[r, w]]))
    return torch.cat(found, 1)


class _Plain:
    """Velocity Verlet of all replicas together, unwrapped positions, double precision."""

    def __init__(self, case, seed, dt):
        self.n, self.box, sp, x, v = _input(case, seed)
        if case["kind"] == "forces":
            x = np.mod(x + 0.02, self.box[0])
        self.x, self.v = torch.from_numpy(x).to(DEV), torch.from_numpy(v).to(DEV)
        self.sp = torch.from_numpy(sp.astype(np.int64)).to(DEV)
        self.L = torch.from_numpy(np.repeat(np.asarray(self.box), self.n)).to(DEV)
        self.rep = torch.from_numpy(np.repeat(np.arange(len(self.n)), self.n)).to(DEV)
        self.p, self.dt = _params(case), dt
        self.eps, self.sig2, self.rc, self.shift, self.sig = _tables(self.p)
        self.reach = synth.max_rcut(self.p) + min(0.6, min(self.box) / 2 - synth.max_rcut(self.p) - 1e-9)
        self.built = None
        self.forces()

    def forces(self):
        skin = self.reach - synth.max_rcut(self.p)
        if self.built is None or float((self.x - self.built).square().sum(-1).max()) > (0.49 * skin) ** 2:
            self.built, at, pairs = self.x.clone(), 0, []
            for n, box in zip(self.n, self.box):
                pairs.append(_near(torch.remainder(self.x[at:at + n], box), box, self.reach) + at)
                at += n
            self.i, self.j = torch.cat(pairs, 1)
            self.ab = self.sp[self.i] * 2 + self.sp[self.j]
        self.f = torch.zeros_like(self.x)
        self.e = torch.zeros_like(self.x[:, 0])
        self.w = torch.zeros(len(self.n), 6, dtype=torch.float64, device=DEV)
        for a in range(0, len(self.i), 1 << 25):
            self._add(self.i[a:a + (1 << 25)], self.j[a:a + (1 << 25)], self.ab[a:a + (1 << 25)])

    def _add(self, i, j, ab):
        box = self.L[i][:, None]
        d = self.x[i] - self.x[j]
        d -= box * torch.round(d / box)
        r2 = d.square().sum(-1)
        at = torch.nonzero(r2 < self.rc.reshape(-1)[ab].square())[:, 0]
        i, j, ab, d, r2 = i[at], j[at], ab[at], d[at], r2[at]
        u = (self.sig2.reshape(-1)[ab] / r2) ** 3
        eps = self.eps.reshape(-1)[ab]
        f = 48.0 * eps * u * (u - 0.5) / r2
        v = 4.0 * eps * (u * u - u) - self.shift.reshape(-1)[ab]
        h = self.p["smooth"]
        if h > 0:
            r = r2.sqrt()
            hs = h * self.sig.reshape(-1)[ab]
            y = (r - self.rc.reshape(-1)[ab]) / hs
            g = y ** 4 / (1.0 + y ** 4)
            f, v = f * g - v * (4.0 * y ** 3 / (1.0 + y ** 4) ** 2) / (hs * r), v * g
        fd = f[:, None] * d
        self.f.index_add_(0, i, fd)
        self.f.index_add_(0, j, -fd)
        self.e.index_add_(0, i, 0.5 * v)
        self.e.index_add_(0, j, 0.5 * v)
        t = torch.stack([fd[:, 0] * d[:, 0], fd[:, 1] * d[:, 1], fd[:, 2] * d[:, 2], fd[:, 0] * d[:, 1],
                         fd[:, 0] * d[:, 2], fd[:, 1] * d[:, 2]], 1)
        self.w.index_add_(0, self.rep[i], t)

    def per_replica(self, y):
        return torch.zeros(len(self.n), dtype=torch.float64, device=DEV).index_add_(0, self.rep, y)

    def kinetic(self):
        return self.per_replica(0.5 * self.v.square().sum(-1))

    def step(self):
        self.v += 0.5 * self.dt * self.f
        self.x += self.dt * self.v
        self.forces()
        self.v += 0.5 * self.dt * self.f

    def to_temperature(self, t):
        n = torch.tensor(self.n, dtype=torch.float64, device=DEV)
        self.v *= torch.sqrt(t * (3 * n - 3) / (2 * self.kinetic()))[self.rep][:, None]

    def heat_bath(self, t, seed, event):
        """Maxwell-Boltzmann velocities from the rand48 sequence, centre of mass at rest, at temperature t."""
        n, mask = int(sum(self.n)), (1 << 48) - 1
        A, C, x = 0x5DEECE66D, 0xB, (seed << 16) | 0x330E
        a, c, ra, rc, k = A, C, 1, 0, 4 * event * n + 1
        while k:
            if k & 1:
                ra, rc = a * ra & mask, (a * rc + c) & mask
            a, c, k = a * a & mask, (a * c + c) & mask, k >> 1
        seq, a, c = np.array([(ra * x + rc) & mask], dtype=np.uint64), A, C
        while len(seq) < 4 * n:
            seq = np.concatenate([seq, (seq * np.uint64(a) + np.uint64(c)) & np.uint64(mask)])
            a, c = a * a & mask, (a * c + c) & mask
        u = torch.from_numpy(seq[:4 * n].astype(np.float64) * 2.0 ** -48).to(DEV).reshape(4, n)
        r1, r2 = torch.sqrt(-2.0 * torch.log(1.0 - u[0])), torch.sqrt(-2.0 * torch.log(1.0 - u[2]))
        two_pi = 2.0 * math.pi
        self.v = torch.stack([r1 * torch.cos(two_pi * u[1]), r1 * torch.sin(two_pi * u[1]),
                              r2 * torch.cos(two_pi * u[3])], 1)
        m = torch.tensor(self.n, dtype=torch.float64, device=DEV)
        mean = torch.stack([self.per_replica(self.v[:, k]) for k in range(3)], 1) / m[:, None]
        self.v -= mean[self.rep]
        self.to_temperature(t)


def exact(case, seed):
    if case["kind"] in ("forces", "noalloc"):
        s = _Plain(case, seed, 0.001)
        w = s.w.cpu().numpy()
        if case["kind"] == "noalloc":
            tot = np.concatenate([[float(s.e.sum()), w[0, :3].sum()], w[0]])
            return {"f": s.f, "e": s.e, "totals": tot}
        return {"f": s.f, "e": s.e, "totals": [s.per_replica(s.e), s.kinetic(), w[:, :3].sum(1), w]}
    s = _Plain(case, seed, case["dt"])
    every = case.get("sample", 20)
    samples, energies, snaps = [], [], []

    def advance(k):
        for _ in range(k):
            s.step()
            energies.append(s.per_replica(s.e))
            if len(energies) % every == 0:
                samples.append((np.full(len(s.n), len(energies)), energies[-1].cpu().numpy(),
                                s.kinetic().cpu().numpy(), s.w[:, :3].sum(1).cpu().numpy(), s.w.cpu().numpy()))

    def bath(event):
        if case["bath"] == "rescale":
            s.to_temperature(case["temperature"])
        elif case["bath"] == "andersen":
            s.heat_bath(case["temperature"], seed & 0xFFFF, event)

    if case["kind"] == "md":
        for event, k in enumerate(_stretches(case)):
            bath(event)
            advance(k)
    else:
        bath(0)
        for _ in range(case["samples"]):
            snaps.append(s.x.clone())
            advance(case["stride"])
    obs = [np.stack([x[k] for x in samples]) for k in range(5)]
    out = {"obs": obs, "steps": np.arange(1, len(energies) + 1), "e_pot": torch.stack(energies), "unwrapped": s.x,
           "vel": s.v}
    if case["kind"] == "corr":
        q = torch.from_numpy(synth.shell_wavevectors(s.box[0], 7.25, case["nq"], seed % 1000)).to(DEV)
        k, l = case["blocks"], case["length"]
        msd, fs = np.full((k, l - 1, 2), np.nan), np.full((k, l - 1, 2), np.nan)
        lags, origins = np.zeros((k, l - 1), np.int64), np.zeros((k, l - 1), np.int64)
        for b in range(k):
            held = snaps[::l ** b]
            for j in range(1, l):
                lags[b, j - 1] = j * l ** b
                origins[b, j - 1] = max(0, len(held) - l + 1)
                got = []
                for o in range(origins[b, j - 1]):
                    d = held[o + j] - held[o]
                    one, many = d.square().sum(1), torch.cos(d @ q.T).mean(1)
                    got.append([[float(y[s.sp == a].mean()) if bool((s.sp == a).any()) else math.nan for a in (0, 1)]
                                for y in (one, many)])
                if got:
                    msd[b, j - 1], fs[b, j - 1] = np.mean([g[0] for g in got], 0), np.mean([g[1] for g in got], 0)
        out["corr"] = [lags, msd, fs, origins]
    return out
