"""Workloads of the library as its users run them, through the public binding.

A case is a dict with the kind of call, the system (FCC-equivalent tiles of a melted box,
the number of particles taken out of it, the model and its options) and the length of the
call.  Kinds:

  md       steps, then the energies and the unwrapped frame (a production run's output
           interval)
  monitor  one step and one observation per call, several times, then the frame
  batch    steps of many replicas of uneven size, then every replica's frame
  forces   a host configuration in, its forces and per-particle energies out
  gr       the radial distribution functions, energy and virial of a state
  relax    a host configuration in, steepest descent, the relaxed frame out

Inputs are liquids: a small box melted with plain torch arithmetic in 64 bits, tiled, then
shifted, displaced and given Maxwell-Boltzmann velocities from the seed.  Mixed precision
does its arithmetic in FP32, so its frames and forces are returned in single precision
(the precision a trajectory file keeps); the FP64 form's in double.
"""
import math

import numpy as np
import torch

from paper_1105_5613_gb300 import bbmd

RHO = 1.2
EPS = ((1.0, 1.5), (1.5, 0.5))
SIG = ((1.0, 0.8), (0.8, 0.88))
FRAC_B = 0.2


def _case(kind, name=None, **kw):
    c = {"kind": kind, "model": "lj", "m": 10, "tx": 1, "ty": 1, "tz": 1, "removed": 0,
         "precision": "mixed", "search": "list", "thermostat": "nve", "T": 2.0, "skin": 0.3,
         "dt": 0.005, "steps": 1}
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest system of the parity runs and of a first trial: latency and launches
        _case("md", "md_4k", steps=50),
        # a program that looks at the state after every step (the benchmark's end-to-end
        # loop), on a ragged particle count
        _case("monitor", "monitor_32k", tx=2, ty=2, tz=2, removed=43, thermostat="nh", steps=10),
        # the ordinary size: the supercooling ramp at the sample size of the CPU baseline
        _case("md", "md_256k", tx=4, ty=4, tz=4, thermostat="nh", steps=50),
        # the other pair model: soft spheres with the shifted force
        _case("md", "soft_256k", model="soft", tx=4, ty=4, tz=4, removed=77, thermostat="nh", T=0.8,
              steps=50),
        # a large box that is neither cubic nor full: ragged cells and blocks on every axis
        _case("md", "md_2m_slab", tx=12, ty=8, tz=5, removed=1713, steps=20),
        # the headline quench, 16 384 000 particles at its skin
        _case("md", "quench_16m", tx=16, ty=16, tz=16, thermostat="nh", skin=0.4, steps=40),
        # the search without a stored list (what systems too large for lists run)
        _case("md", "cell_4m", tx=10, ty=10, tz=10, search="cell", T=0.6, steps=20),
        # the FP64 form
        _case("md", "fp64_108k", tx=3, ty=3, tz=3, precision="fp64", thermostat="nh", steps=10),
        # the replica set: one mixture per temperature, 2048 to 32768 particles each
        _case("batch", "replicas_64", m=6, thermostat="nh", replicas=64, steps=50),
        # a configuration evaluated once: state up, forces and energies down
        _case("forces", "forces_256k", tx=4, ty=4, tz=4, removed=11),
        # the analysis call of the structure studies
        _case("gr", "gr_108k", tx=3, ty=3, tz=3, nbins=500, rmax=5.0),
        # setting up a replica: steepest descent from a badly overlapping start
        _case("relax", "relax_16k", m=8, tx=2, ty=2, tz=2, removed=5, steps=20),
    ]


def _tiles(rng, m, lo, hi):
    """Tile counts of a box of lo to hi particles (spread over the logarithm), sides within
    a factor of about two."""
    n = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    per = 4 * m ** 3
    side = (n / per) ** (1.0 / 3.0)
    t = [max(1, int(round(side * 2.0 ** rng.uniform(-0.5, 0.5)))) for _ in range(3)]
    while per * t[0] * t[1] * t[2] > hi and max(t) > 1:
        t[t.index(max(t))] -= 1
    return {"m": m, "tx": t[0], "ty": t[1], "tz": t[2],
            "removed": rng.randrange(0, max(2, per * t[0] * t[1] * t[2] // 200))}


def draw(rng):
    kind = rng.choice(["md", "md", "md", "monitor", "cell", "fp64", "batch", "forces", "gr", "relax"])
    m = rng.choice([6, 7, 8, 9, 10])
    th = rng.choice(["nve", "nh"])
    opt = {"model": rng.choice(["lj", "lj", "lj_fs", "soft"]), "thermostat": th,
           "T": round(rng.uniform(0.6, 2.0), 2), "dt": rng.choice([0.005, 0.005, 0.002]),
           "skin": rng.choice([0.3, 0.4])}
    if kind == "md":
        return _case("md", steps=rng.randrange(5, 51), **{**opt, **_tiles(rng, m, 2000, 6_000_000)})
    if kind == "monitor":
        return _case("monitor", steps=rng.randrange(4, 21), **{**opt, **_tiles(rng, m, 2000, 500_000)})
    if kind == "cell":
        return _case("md", search="cell", steps=rng.randrange(4, 21),
                     **{**opt, "skin": 0.3, **_tiles(rng, m, 2000, 4_000_000)})
    if kind == "fp64":
        return _case("md", precision="fp64", steps=rng.randrange(4, 21), **{**opt, **_tiles(rng, m, 2000, 200_000)})
    if kind == "batch":
        return _case("batch", replicas=rng.randrange(3, 65), steps=rng.randrange(10, 61), **{**opt, "m": 6})
    if kind == "forces":
        return _case("forces", **{**opt, "precision": rng.choice(["mixed", "mixed", "fp64"]),
                                  **_tiles(rng, m, 2000, 500_000)})
    if kind == "gr":
        return _case("gr", nbins=rng.choice([200, 333, 500, 1000]), rmax=rng.choice([3.0, 4.0, 5.0]),
                     **{**opt, **_tiles(rng, m, 2000, 300_000)})
    return _case("relax", steps=rng.randrange(5, 41), **{**opt, **_tiles(rng, m, 2000, 100_000)})


# ------------------------------------------------------------------------- the model ----

class _Model:
    """Pair tables of a case in 64 bits (Eqs. lj0, sc0, mod0)."""

    def __init__(self, name):
        self.soft = name == "soft"
        self.force_shift = name in ("soft", "lj_fs")
        self.rc = tuple(tuple(2.5 * s for s in row) for row in SIG)
        self.rc_max = max(max(r) for r in self.rc)

    def table(self, what):
        """Tables [4] indexed by 2 a + b."""
        out = []
        for a in range(2):
            for b in range(2):
                e, s, rc = EPS[a][b], SIG[a][b], self.rc[a][b]
                s6 = (s / rc) ** 6
                cut = 4.0 * e * (s6 * s6 if self.soft else s6 * s6 - s6)
                dcut = -(48.0 * e * s6 * s6 if self.soft else 48.0 * e * s6 * s6 - 24.0 * e * s6) / rc
                out.append({"rc": rc, "sig": s, "eps": e, "vcut": cut,
                            "dcut": dcut if self.force_shift else 0.0}[what])
        return torch.tensor(out, dtype=torch.float64, device="cuda")

    def pair(self, k, r2):
        """(f, V) of pairs of kind k at r2 < rc2: force on i is -f (x_j - x_i)."""
        e, s2 = self.table("eps")[k], self.table("sig")[k].square()
        dc, rc = self.table("dcut")[k], self.table("rc")[k]
        ir2 = 1.0 / r2
        s6 = (s2 * ir2) ** 3
        r = r2.sqrt()
        f = 48.0 * e * ir2 * s6 * (s6 if self.soft else s6 - 0.5) + dc / r
        V = 4.0 * e * (s6 * s6 if self.soft else s6 * s6 - s6) - self.table("vcut")[k] - (r - rc) * dc
        return f, V

    def params(self, case):
        p = bbmd.ka_params(
            potential=bbmd.POT_SOFT if self.soft else bbmd.POT_LJ,
            shift=bbmd.SHIFT_FORCE if self.force_shift else bbmd.SHIFT_ENERGY,
            precision=bbmd.PREC_FP64 if case["precision"] == "fp64" else bbmd.PREC_MIXED,
            nbr_mode=bbmd.NBR_CELL if case["search"] == "cell" else bbmd.NBR_VERLET,
            skin=case["skin"])
        for a in range(2):
            for b in range(2):
                p.rcut[a][b] = self.rc[a][b]
        return p


def _pairs(pos, box, reach):
    """Half pair list (i, j) within reach (at least; a few more) of one periodic system."""
    n = pos.shape[0]
    nc = torch.floor(box / reach).long()
    if int(nc.min()) < 3:
        i = []
        j = []
        step = max(1, (1 << 26) // n)
        for a in range(0, n, step):
            d = pos[a:a + step, None] - pos[None]
            d -= box * torch.round(d / box)
            ii, jj = torch.nonzero(d.square().sum(-1) < reach * reach, as_tuple=True)
            keep = jj > ii + a
            i.append((ii + a)[keep])
            j.append(jj[keep])
        return torch.cat(i), torch.cat(j)
    c3 = torch.minimum((pos / (box / nc)).long(), nc - 1)
    key = (c3[:, 2] * nc[1] + c3[:, 1]) * nc[0] + c3[:, 0]
    order = torch.argsort(key)
    ncell = int(nc.prod())
    count = torch.bincount(key, minlength=ncell)
    first = torch.cumsum(count, 0) - count
    cap = int(count.max())
    table = torch.full((ncell, cap), -1, dtype=torch.long, device=pos.device)
    ks = key[order]
    table[ks, torch.arange(n, device=pos.device) - first[ks]] = order
    off = torch.tensor([(x, y, z) for z in (-1, 0, 1) for y in (-1, 0, 1) for x in (-1, 0, 1)],
                       device=pos.device)
    p32, b32 = pos.float(), box.float()
    i = []
    j = []
    step = max(1, (1 << 26) // (27 * cap))
    for a in range(0, n, step):
        q = torch.remainder(c3[a:a + step, None] + off, nc)
        cand = table[(q[..., 2] * nc[1] + q[..., 1]) * nc[0] + q[..., 0]].reshape(q.shape[0], -1)
        me = torch.arange(a, a + q.shape[0], device=pos.device)[:, None]
        d = p32[cand.clamp_min(0)] - p32[me]
        d -= b32 * torch.round(d / b32)
        hit = (cand > me) & (d.square().sum(-1) < reach * reach * 1.0005)
        ii, jj = torch.nonzero(hit, as_tuple=True)
        i.append(ii + a)
        j.append(cand[ii, jj])
    return torch.cat(i), torch.cat(j)


class _Exact:
    """Systems side by side in 64 bits: sysid[i] tells the system of a particle."""

    def __init__(self, model, systems):
        self.model = model
        self.x = torch.cat([s["pos"] for s in systems])
        self.v = torch.cat([s["vel"] for s in systems])
        self.sp = torch.cat([s["sp"] for s in systems]).long()
        self.ns = [s["pos"].shape[0] for s in systems]
        self.boxes = torch.stack([s["box"] for s in systems])
        self.sysid = torch.repeat_interleave(torch.arange(len(systems), device="cuda"),
                                             torch.tensor(self.ns, device="cuda"))
        self.left = -1.0

    def _list(self):
        side = float(self.boxes.min())
        reach = self.model.rc_max + 0.7
        if side / reach < 3.0 and side / 3.0 >= self.model.rc_max + 0.3:
            reach = 0.999 * side / 3.0
        self.left = reach - self.model.rc_max
        i, j, a = [], [], 0
        for n, box in zip(self.ns, self.boxes):
            w = torch.remainder(self.x[a:a + n], box)
            ii, jj = _pairs(w, box, reach)
            i.append(ii + a)
            j.append(jj + a)
            a += n
        self.i, self.j = torch.cat(i), torch.cat(j)

    def closed(self, dist):
        """Some pair has closed by up to dist since the last call."""
        self.left -= dist

    def forces(self, energies=False):
        if self.left <= 0.0:
            self._list()
        F = torch.zeros_like(self.x)
        u = torch.zeros(self.x.shape[0], dtype=torch.float64, device="cuda")
        W = 0.0
        rc2 = self.model.table("rc").square()
        for a in range(0, self.i.numel(), 1 << 26):
            i, j = self.i[a:a + (1 << 26)], self.j[a:a + (1 << 26)]
            d = self.x[j] - self.x[i]
            L = self.boxes[self.sysid[i]]
            d -= L * torch.round(d / L)
            r2 = d.square().sum(-1)
            k = self.sp[i] * 2 + self.sp[j]
            keep = r2 < rc2[k]
            i, j, d, r2, k = i[keep], j[keep], d[keep], r2[keep], k[keep]
            f, V = self.model.pair(k, r2)
            fd = f[:, None] * d
            F.index_add_(0, i, -fd)
            F.index_add_(0, j, fd)
            if energies:
                u.index_add_(0, i, 0.5 * V)
                u.index_add_(0, j, 0.5 * V)
                W += float((f * r2).sum())
        return (F, u, W) if energies else F

    def kinetic(self):
        k = torch.zeros(len(self.ns), dtype=torch.float64, device="cuda")
        return k.index_add_(0, self.sysid, 0.5 * self.v.square().sum(-1))

    def run(self, steps, dt, targets):
        """Velocity Verlet; targets: None, or per step the Nose-Hoover target of each system
        (tau = 0.5).  Returns the kinetic energies after each step."""
        g = 3.0 * torch.tensor(self.ns, dtype=torch.float64, device="cuda") - 3.0
        xi = torch.zeros_like(g)

        def half(T):
            nonlocal xi
            K, Q = self.kinetic(), g * T * 0.25
            xi = xi + 0.25 * dt * (2.0 * K - g * T) / Q
            s = torch.exp(-xi * 0.5 * dt)
            self.v = self.v * s[self.sysid][:, None]
            xi = xi + 0.25 * dt * (2.0 * K * s * s - g * T) / Q

        F, ke = self.forces(), []
        for k in range(steps):
            if targets is not None:
                half(targets[k])
            self.v = self.v + 0.5 * dt * F
            self.x = self.x + dt * self.v
            self.closed(2.0 * dt * float(self.v.norm(dim=-1).max()))
            F = self.forces()
            self.v = self.v + 0.5 * dt * F
            if targets is not None:
                half(targets[k])
            ke.append(self.kinetic())
        return ke


# ------------------------------------------------------------------------- the inputs ----

_melted = {}


def _melt(m, model_name, T):
    """A periodic box of 4 m^3 particles melted from the FCC lattice with velocities
    rescaled to T, in 64 bits (made once per process)."""
    T = 2.0 if T >= 1.2 else 1.0
    key = (m, model_name, T)
    if key not in _melted:
        g = torch.Generator(device="cuda").manual_seed(7919 + m)
        model = _Model(model_name)
        a = (4.0 / RHO) ** (1.0 / 3.0)
        cell = torch.stack(torch.meshgrid(*[torch.arange(m, device="cuda")] * 3, indexing="ij"), -1)
        basis = torch.tensor([[0, 0, 0], [0.5, 0.5, 0], [0.5, 0, 0.5], [0, 0.5, 0.5]],
                             dtype=torch.float64, device="cuda")
        pos = ((cell.reshape(-1, 1, 3).double() + basis + 0.25) * a).reshape(-1, 3)
        n = pos.shape[0]
        sp = torch.zeros(n, dtype=torch.uint8, device="cuda")
        sp[torch.randperm(n, generator=g, device="cuda")[:int(FRAC_B * n)]] = 1
        vel = torch.randn(n, 3, generator=g, device="cuda", dtype=torch.float64)
        e = _Exact(model, [{"pos": pos, "vel": vel, "sp": sp,
                            "box": torch.full((3,), m * a, dtype=torch.float64, device="cuda")}])
        for k in range(30):
            e.v = e.v * (3.0 * n * (T if k > 12 else 2.0) / (e.v.square().sum())).sqrt()
            e.run(8, 0.004, None)
        _melted[key] = (torch.remainder(e.x, m * a), sp, m * a)
    return _melted[key]


def _system(case, seed, noise=0.02):
    """Positions, velocities, species and box of one system, on the GPU."""
    base, sp, side = _melt(case["m"], case["model"], case["T"])
    g = torch.Generator(device="cuda").manual_seed(int(seed) * 2654435761 % (1 << 61))
    t = [case["tx"], case["ty"], case["tz"]]
    tiles = torch.stack(torch.meshgrid(*[torch.arange(k, device="cuda") for k in t], indexing="ij"), -1)
    pos = (tiles.reshape(-1, 1, 3).double() * side + base).reshape(-1, 3)
    sp = sp.repeat(t[0] * t[1] * t[2])
    n = pos.shape[0] - case["removed"]
    if case["removed"]:
        keep = torch.randperm(pos.shape[0], generator=g, device="cuda")[:n].sort().values
        pos, sp = pos[keep], sp[keep]
    box = torch.tensor([side * k for k in t], dtype=torch.float64, device="cuda")
    pos += torch.rand(3, generator=g, device="cuda", dtype=torch.float64) * box
    pos += noise * torch.randn(n, 3, generator=g, device="cuda", dtype=torch.float64)
    pos = torch.remainder(pos, box)
    pos = torch.where(pos < box, pos, torch.zeros_like(pos))
    vel = torch.randn(n, 3, generator=g, device="cuda", dtype=torch.float64)
    vel -= vel.mean(0)
    vel *= (case["T"] * (3 * n - 3) / vel.square().sum()).sqrt()
    return {"pos": pos, "vel": vel, "sp": sp, "box": box}


def _replicas(case, seed):
    """Replicas of 2048 to 32768 particles, spread as the replica set spreads them."""
    r = np.random.default_rng(case["replicas"])
    out = []
    for k in range(case["replicas"]):
        n = 2048 + int(r.integers(0, 30721))
        m, tx, ty, tz = max((s for s in ((8, 1, 1, 1), (9, 1, 1, 1), (10, 1, 1, 1), (6, 2, 2, 2), (6, 2, 2, 3),
                                         (6, 2, 3, 3), (6, 3, 3, 3), (6, 3, 3, 4))
                             if 4 * s[0] ** 3 * s[1] * s[2] * s[3] <= n), key=lambda s: s[0] ** 3 * s[1] * s[2] * s[3])
        out.append(_system({**case, "m": m, "tx": tx, "ty": ty, "tz": tz,
                            "removed": int(r.integers(0, 20))}, int(seed) * 1009 + k))
    return out


def _inputs(case, seed):
    if case["kind"] == "batch":
        return _replicas(case, seed)
    return [_system(case, seed, noise=0.1 if case["kind"] == "relax" else 0.02)]


def _temperatures(case):
    """T of each replica: evenly spaced, as a temperature ladder."""
    return np.linspace(0.4, 2.0, case["replicas"])


class _Frame:
    """Pinned buffers of n particles for get_state, and the unwrapped frame made of them."""

    def __init__(self, n, double):
        pin = lambda dt: torch.zeros(n, 3, dtype=dt, pin_memory=True)  # noqa: E731
        self.pos, self.vel, self.img = pin(torch.float64), pin(torch.float64), pin(torch.int32)
        self.x = torch.zeros(n, 3, dtype=torch.float64)
        self.double = double
        if not double:
            self.x32, self.v32 = torch.zeros(n, 3), torch.zeros(n, 3)

    def views(self, a, b):
        return self.pos[a:b].numpy(), self.vel[a:b].numpy(), self.img[a:b].numpy()

    def unwrap(self, a, b, box):
        torch.mul(self.img[a:b], box, out=self.x[a:b])
        self.x[a:b].add_(self.pos[a:b])

    def out(self):
        if self.double:
            return {"frame": self.x, "velocities": self.vel}
        return {"frame": self.x32.copy_(self.x), "velocities": self.v32.copy_(self.vel)}


def prepare(case, seed):
    model = _Model(case["model"])
    systems = _inputs(case, seed)
    host = [{k: v.cpu() for k, v in s.items()} for s in systems]
    st = {"case": case, "boxes": [h["box"] for h in host], "ns": [h["pos"].shape[0] for h in host]}
    if case["kind"] == "batch":
        st["sim"] = bbmd.Batch(model.params(case), st["ns"], np.stack([h["box"].numpy() for h in host]),
                               [h["sp"].numpy() for h in host], [h["pos"].numpy() for h in host],
                               [h["vel"].numpy() for h in host])
    else:
        h = host[0]
        st["sim"] = bbmd.Sim(model.params(case), st["ns"][0], h["box"].numpy(), h["sp"].numpy(),
                             h["pos"].numpy(), h["vel"].numpy())
        if case["kind"] in ("forces", "relax"):  # what comes from the host on each call
            st["pos"], st["vel"] = (h[k].pin_memory() for k in ("pos", "vel"))
    if case["kind"] not in ("forces", "gr"):
        st["frame"] = _Frame(sum(st["ns"]), case["precision"] == "fp64")
    th = {"nve": None, "nh": (bbmd.THERMO_NH, case["T"], 0.98 * case["T"], 0.5)}[case["thermostat"]]
    if case["kind"] == "batch" and th is not None:
        th = [(bbmd.THERMO_NH, float(T), float(T), 0.5) for T in _temperatures(case)]
    st["thermostat"] = th
    return st


# --------------------------------------------------------------------------- the calls ----

def _whole(st, sim):
    f = st["frame"]
    sim.get_state(out=f.views(0, sim.n))
    f.unwrap(0, sim.n, st["boxes"][0])
    return f.out()


def run(st):
    c, sim = st["case"], st["sim"]
    if c["kind"] == "md":
        sim.step(c["steps"], c["dt"], st["thermostat"])
        o = sim.observe(bbmd.OBS_ENERGY)
        return {"ke": o["ke"], "pe": o["pe"], **_whole(st, sim)}
    if c["kind"] == "monitor":
        ke = []
        for _ in range(c["steps"]):
            sim.step(1, c["dt"], st["thermostat"])
            ke.append(sim.observe(bbmd.OBS_MOMENTUM)["ke"])
        return {"ke": np.array(ke, dtype=np.float32), **_whole(st, sim)}
    if c["kind"] == "batch":
        sim.step(c["steps"], c["dt"], st["thermostat"])
        f, a, ke = st["frame"], 0, []
        for r, (n, box) in enumerate(zip(st["ns"], st["boxes"])):
            rep = sim.replica(r)
            ke.append(rep.observe(bbmd.OBS_MOMENTUM)["ke"])
            rep.get_state(out=f.views(a, a + n))
            f.unwrap(a, a + n, box)
            a += n
        return {"ke": np.array(ke, dtype=np.float32), **f.out()}
    if c["kind"] == "forces":
        sim.set_state(st["pos"].numpy(), st["vel"].numpy())
        F, u = sim.get_forces(energies=True)
        F = torch.from_numpy(F)
        return {"F": F if c["precision"] == "fp64" else F.float(), "u": u}
    if c["kind"] == "gr":
        o = sim.observe(bbmd.OBS_GR | bbmd.OBS_ENERGY | bbmd.OBS_VIRIAL, nbins=c["nbins"], rmax=c["rmax"])
        return {"counts": o["gr_counts"].astype(np.int64), "gr": o["gr"], "pe": o["pe"], "virial": o["virial"]}
    sim.set_state(st["pos"].numpy(), st["vel"].numpy())
    sim.minimize(c["steps"], 1e-3, 0.05)
    return {"pe": sim.observe(bbmd.OBS_ENERGY)["pe"], **_whole(st, sim)}


# -------------------------------------------------------------------- work and values ----

def _count(case):
    if case["kind"] == "batch":
        return case["replicas"] * 15000
    return 4 * case["m"] ** 3 * case["tx"] * case["ty"] * case["tz"] - case["removed"]


def work(case):
    n, model = _count(case), _Model(case["model"])
    b = FRAC_B
    w = ((1 - b) ** 2, b * (1 - b), b * (1 - b), b * b)
    half = sum(wk * 4.0 / 3.0 * math.pi * rc ** 3 for wk, rc in zip(w, sum(model.rc, ()))) * RHO / 2.0
    evaluations = {"forces": 1, "gr": 1}.get(case["kind"], case["steps"])
    flops = 25.0 * half * n * evaluations  # interacting half pairs, 25 flops each
    bytes_ = 48.0 * n  # positions and velocities
    if case["kind"] == "forces":
        bytes_ += 32.0 * n
    elif case["kind"] == "gr":
        flops = 9.0 * n * 4.0 / 3.0 * math.pi * case["rmax"] ** 3 * RHO / 2.0
    else:
        bytes_ += 60.0 * n  # the state back
    return {"bytes": bytes_, "flops": flops}


def exact(case, seed):
    n, model = _count(case), _Model(case["model"])
    if n * case["steps"] > 9e7 or (case["kind"] == "gr" and n > 3e5):
        return None
    e = _Exact(model, _inputs(case, seed))
    if case["kind"] == "gr":
        return _exact_gr(case, e)
    if case["kind"] == "forces":
        F, u, _ = e.forces(energies=True)
        return {"F": F, "u": u}
    if case["kind"] == "relax":
        for _ in range(case["steps"]):
            F = e.forces()
            fm = float(F.norm(dim=-1).max())
            h = min(1e-3, 0.05 / fm)
            e.x = e.x + h * F
            e.closed(2.0 * h * fm)
        pe = float(e.forces(energies=True)[1].sum())
        return {"pe": pe, "frame": e.x, "velocities": e.v}
    k = case["steps"]
    targets = None
    if case["thermostat"] == "nh":
        if case["kind"] == "batch":
            T = torch.tensor(_temperatures(case), dtype=torch.float64, device="cuda")
            targets = [T] * k
        elif case["kind"] == "monitor":
            targets = [torch.tensor([case["T"]], dtype=torch.float64, device="cuda")] * k
        else:
            targets = [torch.tensor([case["T"] * (1.0 - 0.02 * s / k)], dtype=torch.float64, device="cuda")
                       for s in range(k)]
    ke = e.run(k, case["dt"], targets)
    if case["kind"] == "monitor":
        return {"ke": torch.cat(ke), "frame": e.x, "velocities": e.v}
    if case["kind"] == "batch":
        return {"ke": ke[-1], "frame": e.x, "velocities": e.v}
    pe = float(e.forces(energies=True)[1].sum())
    return {"ke": float(ke[-1][0]), "pe": pe, "frame": e.x, "velocities": e.v}


def _exact_gr(case, e):
    nb, rmax = case["nbins"], case["rmax"]
    box = e.boxes[0]
    i, j = _pairs(torch.remainder(e.x, box), box, rmax)
    d = e.x[j] - e.x[i]
    d -= box * torch.round(d / box)
    r = d.square().sum(-1).sqrt()
    q = torch.floor(r / (rmax / nb)).long()
    ok = q < nb
    i, j, q = i[ok], j[ok], q[ok]
    a, b = e.sp[i], e.sp[j]
    counts = (torch.bincount((a * 2 + b) * nb + q, minlength=4 * nb)
              + torch.bincount((b * 2 + a) * nb + q, minlength=4 * nb)).reshape(2, 2, nb)
    N = torch.bincount(e.sp, minlength=2).double()
    edge = torch.arange(nb + 1, dtype=torch.float64, device="cuda") * (rmax / nb)
    shell = 4.0 * math.pi / 3.0 * (edge[1:] ** 3 - edge[:-1] ** 3)
    den = (N[:, None] * (N[None] - torch.eye(2, device="cuda", dtype=torch.float64)))[..., None] * shell
    gr = torch.where(den > 0, float(box.prod()) * counts / den, torch.zeros_like(den))
    _, u, W = e.forces(energies=True)
    return {"counts": None, "gr": gr, "pe": float(u.sum()), "virial": W}
