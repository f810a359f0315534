"""Timed workloads of the united-atom polyethylene MD engine, through its public entry points.

Seven kinds of work a user gives the engine:
  md         a piece of a trajectory: md_step(n), then the frame (positions, velocities, image
             counters), with or without the energy read-out
  replicas   independent melts of uneven size at their own temperatures, stepped together
  molecules  a trajectory of a general molecule type (md_desc.topology)
  forces     forces and energies of given positions: md_set_state, md_forces, md_energy
  adjoint    gradients of trajectory means with respect to the force field
  analysis   radial distribution function and chain observables of a configuration
  binning    md_bin_static into the caller's arrays

Melts are seeded: chains grown at 0.77 g/cm^3 (chaingen) and brought to 500 K by a short Langevin
run written here in torch, one periodic tile per (chains, sites); larger melts repeat the tile, and
the seed gives the axes, reflections, shift, order of the chains and the velocities.
"""
import math

import numpy as np
import torch

import chaingen
import paper_1001_3764_gb300 as md

KB = md.KB
DT = 0.001          # ps, the engine's default step
RC, SKIN = 1.0, 0.1   # nm, the engine's defaults
PAIR_FLOPS = 69.2 * 20.0   # unique pairs within the cutoff per atom in a melt x operations of one
BONDED_FLOPS = 250.0       # one bond, angle and dihedral per atom
TILES = (20, 27, 37, 54, 80, 125)   # chains per tile of the replicas


# ---------------------------------------------------------------- which cases

def listed():
    return [
        # the smallest system of the engine's configurations, run a little at a time with every
        # frame read on the host: launches and latency are all there is
        dict(name="nve_1500", kind="md", base=10, tile=1, sites=150, precision="mixed", ensemble="nve", T=500.0,
             steps=20, frame="host", energy=False),
        # the paper-scale melt being quenched, plain FP32 with the weak-coupling thermostat
        dict(name="quench_150k_plain", kind="md", base=125, tile=2, sites=150, precision="plain", ensemble="vrescale",
             T=300.0, steps=10, frame="device", energy=False),
        # the benchmark melt: 10,000 chains, mixed precision, NVE
        dict(name="nve_1500k_mixed", kind="md", base=80, tile=5, sites=150, precision="mixed", ensemble="nve", T=500.0,
             steps=10, frame="device", energy=False),
        # the paper's ensemble (Leap-Frog, Nose-Hoover) and its longer chains; 25 steps are two
        # list cycles and a remainder
        dict(name="nvt_35k_300mers", kind="md", base=117, tile=1, sites=300, precision="mixed", ensemble="nose_hoover",
             T=450.0, steps=25, frame="device", energy=False),
        # half a million sites with thermodynamic output after every list cycle
        dict(name="nve_506k_energy", kind="md", base=125, tile=3, sites=150, precision="mixed", ensemble="nve", T=500.0,
             steps=10, frame="device", energy=True),
        # uneven replicas quenched at their own temperatures in the same launches
        dict(name="replicas_64", kind="replicas", count=64, sites=150, steps=12, skin=0.12, rebin=12),
        # branched molecules through the bond-graph topology
        dict(name="branched_36k", kind="molecules", k=9, mixed_types=False, steps=10),
        # positions from another program (a Monte Carlo move, a force matching set): set, forces, energies
        dict(name="forces_65k", kind="forces", base=54, tile=2, sites=150, precision="mixed", pair_exact=False),
        # force-field gradients of a trajectory, the 7,500-site system of the configurations
        dict(name="adjoint_7500", kind="adjoint", base=50, sites=150, steps=100, checkpoint=50, lj_form=0),
        # structure of a saved configuration of the paper-scale melt
        dict(name="analysis_150k", kind="analysis", base=125, tile=2, sites=150, precision="mixed", r_max=1.0, bins=200),
        # cell binning for a caller that owns all device memory
        dict(name="binning_778k", kind="binning", atoms=777_777, cells=25),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _melt_size(rng, most):
    """(base, tile, sites) of a melt of about 1,500 .. most sites, log-uniform."""
    sites = 150 if rng.random() < 0.5 else _log_int(rng, 7, 511)
    n = math.exp(rng.uniform(math.log(1500), math.log(most)))
    tile = max(1, math.ceil((n / 19000.0) ** (1.0 / 3.0) - 1e-9))
    base = max(math.ceil(1500 / sites), int(n / tile ** 3 / sites))
    return base, tile, sites


def draw(rng):
    kind = rng.choice(["md", "md", "md", "md", "replicas", "molecules", "forces", "adjoint", "analysis", "binning"])
    if kind == "replicas":
        skin, rebin = rng.choice([(0.08, 6), (0.1, 10), (0.12, 12)])
        return dict(kind=kind, count=rng.randint(2, 64), sites=150, steps=rng.randint(4, 12), skin=skin, rebin=rebin)
    if kind == "molecules":
        return dict(kind=kind, k=rng.randint(4, 24), mixed_types=rng.random() < 0.5, steps=rng.randint(5, 15))
    if kind == "adjoint":
        steps = _log_int(rng, 10, 100)
        return dict(kind=kind, base=rng.randint(10, 50), sites=rng.choice([rng.randint(120, 150), 150]), steps=steps,
                    checkpoint=rng.randint(5, 50), lj_form=rng.randint(0, 1))
    if kind == "binning":
        return dict(kind=kind, atoms=_log_int(rng, 1000, 1 << 20), cells=rng.randint(3, 50))
    if kind == "forces":
        base, tile, sites = _melt_size(rng, 600_000)
        return dict(kind=kind, base=base, tile=tile, sites=sites, precision=rng.choice(["mixed", "mixed", "plain"]),
                    pair_exact=rng.random() < 0.3)
    if kind == "analysis":
        base, tile, sites = _melt_size(rng, 150_000)
        return dict(kind=kind, base=base, tile=tile, sites=sites, precision=rng.choice(["mixed", "plain"]),
                    r_max=round(rng.uniform(0.6, 1.0), 3), bins=rng.randint(50, 500))
    base, tile, sites = _melt_size(rng, 1_400_000)
    big = base * tile ** 3 * sites > 200_000
    return dict(kind=kind, base=base, tile=tile, sites=sites, precision=rng.choice(["mixed", "mixed", "plain"]),
                ensemble=rng.choice(["nve", "nve", "vrescale", "nose_hoover"]), T=round(rng.uniform(300.0, 500.0), 1),
                steps=rng.randint(3, 10) if big else rng.randint(3, 40), frame=rng.choice(["device", "host"]) if not big
                else "device", energy=rng.random() < 0.4)


# ---------------------------------------------------------------- inputs

def _near(x, L, sites, radius, most):
    """Neighbour matrix [N, most] of one tile (FP32, nearest first), 1-2 and 1-3 neighbours left out."""
    n = x.shape[0]
    idx = torch.arange(n, device=x.device)
    chain, site = idx // sites, idx % sites
    out = []
    for b in range(0, n, 2048):
        d = x[b:b + 2048, None, :] - x[None, :, :]
        d -= L * torch.round(d / L)
        r2 = (d * d).sum(2)
        same = (chain[b:b + 2048, None] == chain[None]) & ((site[b:b + 2048, None] - site[None]).abs() <= 2)
        r2.masked_fill_(same, 1e9)
        out.append(torch.topk(r2, min(most, n), dim=1, largest=False).indices)
    return torch.cat(out)


def _bonded_energy(x, params):
    """Energy of bonds, angles and dihedrals of chains x[chains, sites, 3] (continuous)."""
    b = x[:, 1:] - x[:, :-1]
    r = b.square().sum(2).sqrt()
    e = 0.5 * params["kb"] * (r - params["b0"]).square().sum()
    u, w = -b[:, :-1], b[:, 1:]
    th = torch.atan2(torch.linalg.cross(u, w).square().sum(2).sqrt(), (u * w).sum(2))
    e = e + 0.5 * params["ka"] * (th - params["theta0"]).square().sum()
    if x.shape[1] > 3:
        m, n = torch.linalg.cross(b[:, :-2], b[:, 1:-1]), torch.linalg.cross(b[:, 1:-1], b[:, 2:])
        phi = torch.atan2(r[:, 1:-1] * (b[:, :-2] * n).sum(2), (m * n).sum(2))
        e = e + params["kphi"] * (1.0 + torch.cos(params["n_mult"] * phi - params["phis"])).sum()
    return e


def _relax(x, L, sites, steps=280):
    """0.28 ps of Langevin dynamics at 500 K (friction 20 / ps, FP32, forces capped while contacts open).
    Every sum has a fixed order, so the result is the same on every run."""
    p = md.default_params()
    dev = torch.device("cuda")
    x = torch.tensor(x, dtype=torch.float32, device=dev)
    gen = torch.Generator(device=dev).manual_seed(1001)
    mass, T = p["mass"][0], 500.0
    c = math.exp(-20.0 * DT)
    noise = math.sqrt((1.0 - c * c) * KB * T / mass)
    v = math.sqrt(KB * T / mass) * torch.randn(x.shape, generator=gen, device=dev)
    eps, s2 = p["eps"][0], p["sigma"][0] ** 2
    for k in range(steps):
        if k % 14 == 0:
            nbr = _near(x, L, sites, 0.9, 112)
        d = x[:, None, :] - x[nbr]
        d -= L * torch.round(d / L)
        r2 = (d * d).sum(2)
        ir2 = torch.where(r2 < 0.64, 1.0 / r2.clamp_min(0.01), torch.zeros_like(r2))
        s6 = (s2 * ir2) ** 3
        f = ((24.0 * eps * (2.0 * s6 * s6 - s6) * ir2)[:, :, None] * d).sum(1)
        xg = x.reshape(-1, sites, 3).detach().requires_grad_(True)
        f = f - torch.autograd.grad(_bonded_energy(xg, p), xg)[0].reshape(-1, 3)
        norm = f.square().sum(1, keepdim=True).sqrt()
        f = f * (4000.0 / norm.clamp_min(4000.0))
        v = c * (v + DT / mass * f) + noise * torch.randn(x.shape, generator=gen, device=dev)
        x = x + DT * v
    return x.double().cpu().numpy()


_tiles = {}


def _tile(chains, sites):
    """(continuous positions [N, 3], side) of a relaxed tile; the same in every process."""
    if (chains, sites) not in _tiles:
        L = round(chaingen.box_length(chains, sites) * 2 ** 14) / 2 ** 14   # its multiples stay exact in FP32
        m = chaingen.melt(chains, sites, seed=97, T=500.0, L=L)
        _tiles[chains, sites] = _relax(chaingen.unwrapped(m), L, sites), L
    return _tiles[chains, sites]


def _masses(types):
    return np.asarray(md.default_params()["mass"])[types]


def _maxwell(rng, masses, T):
    v = rng.standard_normal((len(masses), 3)) * np.sqrt(KB * T / masses)[:, None]
    return v - (masses[:, None] * v).sum(0) / masses.sum()


def _melt(base, tile, sites, seed, T):
    rng = np.random.default_rng(seed)
    x, L0 = _tile(base, sites)
    L = L0 * tile
    x = x.reshape(base, sites, 3)
    if tile > 1:
        k = np.arange(tile) * L0
        o = np.stack(np.meshgrid(k, k, k, indexing="ij"), -1).reshape(-1, 1, 1, 3)
        x = (o + x[None]).reshape(-1, sites, 3)
    x = x[rng.permutation(len(x))].reshape(-1, 3)[:, rng.permutation(3)]
    x = x * rng.choice([-1.0, 1.0], 3) + rng.uniform(0.0, L, 3)
    x = np.mod(x, L)
    x[x >= L] = 0.0
    types = np.zeros(sites, np.int64)
    types[[0, -1]] = 1
    n = base * tile ** 3
    v = _maxwell(rng, np.tile(_masses(types), n), T)
    return dict(pos=np.ascontiguousarray(x), vel=v, L=L, n_chains=n, sites=sites, T=T)


def _molecule(mixed_types):
    """A branched 12-atom molecule: (bonds, types, coordinates); atoms with one bond are C_33."""
    bonds = [(k, k + 1) for k in range(7)] + [(2, 8), (4, 9), (6, 10), (10, 11)]
    deg = np.bincount(np.array(bonds).ravel(), minlength=12)
    types = (deg == 1).astype(np.int32)
    if mixed_types:
        types[3] = 1
    b, th = 0.153, math.acos(-1.0 / 3.0)
    x = [np.array([k * b * math.sin(th / 2), (k % 2) * b * math.cos(th / 2), 0.0]) for k in range(8)]
    x += [x[2] + [0, 0, b], x[4] - [0, 0, b], x[6] + [0, 0, b]]
    tip = np.array([0.5, 0.3, 0.8124])
    x.append(x[10] + b * tip / np.linalg.norm(tip))
    x = np.array(x)
    return np.array(bonds, np.int32), types, x - x.mean(0)


def _molecules(k, mixed_types, seed):
    """4 k^3 molecules along x on a 21/16 x 21/32 x 21/32 nm lattice, turned a little about their axis."""
    rng = np.random.default_rng(seed)
    bonds, types, x0 = _molecule(mixed_types)
    a = 21.0 / 16.0
    gx, gy, gz = np.meshgrid(np.arange(k), np.arange(2 * k), np.arange(2 * k), indexing="ij")
    o = np.stack([gx * a, gy * a / 2, gz * a / 2], -1).reshape(-1, 3) + 0.2
    o = o + rng.uniform(-0.02, 0.02, o.shape)
    t = rng.uniform(-0.25, 0.25, len(o))
    x = np.empty((len(o), 12, 3))
    x[:, :, 0] = x0[:, 0]
    x[:, :, 1] = np.cos(t)[:, None] * x0[:, 1] - np.sin(t)[:, None] * x0[:, 2]
    x[:, :, 2] = np.sin(t)[:, None] * x0[:, 1] + np.cos(t)[:, None] * x0[:, 2]
    x = np.mod(x + o[:, None, :], k * a).reshape(-1, 3)
    x[x >= k * a] = 0.0
    v = _maxwell(rng, np.tile(_masses(types), len(o)), 300.0)
    return dict(pos=x, vel=v, L=k * a, n_chains=len(o), sites=12, T=300.0), (bonds, types)


def _replica_sizes(count, seed):
    """(chains of a tile, tiles per side, temperature) of each replica: 20 .. 296 chains, 250 .. 500 K."""
    rng = np.random.default_rng(seed)
    return [(int(rng.choice(TILES[:3] if k == 2 else TILES)), k, float(rng.uniform(250.0, 500.0)))
            for k in (int(rng.integers(1, 3)) for _ in range(count))]


def _replica_melts(case, seed):
    return [_melt(b, k, case["sites"], seed * 1000 + r, T)
            for r, (b, k, T) in enumerate(_replica_sizes(case["count"], case["count"]))]


def _precision(case):
    return md.MD_PLAIN_FP32 if case.get("precision") == "plain" else md.MD_MIXED


ENSEMBLES = {"nve": md.MD_NVE, "vrescale": md.MD_VRESCALE, "nose_hoover": md.MD_NOSE_HOOVER}


def prepare(case, seed):
    kind = case["kind"]
    dev = torch.device("cuda")
    if kind == "binning":
        g = torch.Generator(device=dev).manual_seed(seed)
        n, M, L = case["atoms"], case["cells"], (case["atoms"] / 33.0) ** (1.0 / 3.0)
        return dict(case=case, L=L, pos=L * torch.rand(3, n, dtype=torch.float64, generator=g, device=dev),
                    cell_of=torch.empty(n, dtype=torch.int32, device=dev),
                    cell_start=torch.empty(M ** 3 + 1, dtype=torch.int32, device=dev),
                    perm=torch.empty(n, dtype=torch.int32, device=dev), stream=torch.cuda.current_stream().cuda_stream)
    if kind == "adjoint":
        m = _melt(case["base"], 1, case["sites"], seed, 500.0)
        return dict(case=case, adj=md.Adjoint(m, n_steps=case["steps"], checkpoint_every=case["checkpoint"],
                                              lj_form=case["lj_form"]))
    if kind == "replicas":
        melts = _replica_melts(case, seed)
        s = md.System(melts, precision=md.MD_MIXED, thermostat=md.MD_VRESCALE, T_target=[m["T"] for m in melts],
                      tau_t=0.1, skin=case["skin"], rebin_every=case["rebin"])
    elif kind == "molecules":
        m, topology = _molecules(case["k"], case["mixed_types"], seed)
        s = md.System(m, topology=topology)
    else:
        m = _melt(case["base"], case["tile"], case["sites"], seed, case.get("T", 500.0))
        kw = {}
        if kind == "md" and case["ensemble"] != "nve":
            kw = dict(thermostat=ENSEMBLES[case["ensemble"]], T_target=case["T"], tau_t=0.1)
        s = md.System(m, precision=_precision(case), lj_pair_exact=bool(case.get("pair_exact")), **kw)
    state = dict(case=case, system=s, stream=torch.cuda.current_stream())
    if kind != "analysis":
        n = s.n_atoms
        state.update(x=torch.empty(n, 3, dtype=torch.float64, device=dev),
                     v=torch.empty(n, 3, dtype=torch.float64, device=dev),
                     img=torch.empty(n, 3, dtype=torch.int32, device=dev))
    if kind == "forces":
        state["pos"], state["vel"] = (torch.tensor(a, device=dev) for a in (m["pos"], m["vel"]))
    return state


# ---------------------------------------------------------------- one pass

def _ok(code, s):
    if code != md.MD_OK:
        raise md.MDError(code, md.md_last_error(s.h))


def _energies(s):
    """Energies of all replicas, one list per quantity."""
    e = s.energy()
    return {k: np.array([q[k] for q in e], np.float64) for k in ("lj", "lj_shifted", "bond", "angle", "dihedral",
                                                                 "kinetic", "temperature", "total", "virial",
                                                                 "pressure")}


def _frame(state):
    """Positions, velocities and image counters in the caller's device arrays (the C ABI takes either kind)."""
    s = state["system"]
    _ok(md.load().md_get_state(s.h, state["x"].data_ptr(), state["v"].data_ptr(), state["img"].data_ptr()), s)
    return dict(x=state["x"], v=state["v"], img=state["img"])


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "binning":
        md.md_bin_static(state["pos"].data_ptr(), case["atoms"], state["L"], case["cells"], state["cell_of"].data_ptr(),
                         state["cell_start"].data_ptr(), state["perm"].data_ptr(), state["stream"])
        return dict(cell_of=state["cell_of"], cell_start=state["cell_start"], perm=state["perm"])
    if kind == "adjoint":
        adj = state["adj"]
        obs = adj.forward()
        return dict(obs=obs, grad=adj.backward((1.0, 0.5)))
    s = state["system"]
    if kind == "forces":
        _ok(md.load().md_set_state(s.h, state["pos"].data_ptr(), state["vel"].data_ptr()), s)
        _ok(md.load().md_forces(s.h, state["x"].data_ptr()), s)
        return dict(forces=state["x"], energy=_energies(s))
    if kind == "analysis":
        _, g, counts = s.rdf(case["r_max"], case["bins"])
        o = s.observables()
        return dict(g=g, counts=counts, r_ee=o["r_ee"], rg2=o["rg2"], trans=o["trans_fraction"])
    s.step(case["steps"])
    if case.get("frame") == "host":
        x, v, img = s.state()
        out = dict(x=x, v=v, img=img)
    else:
        out = _frame(state)
    if case.get("energy"):
        out["energy"] = _energies(s)
    return out


def work(case):
    kind = case["kind"]
    if kind == "binning":   # positions in; cell, order and starts out
        n = case["atoms"]
        return dict(bytes=n * (24 + 4 + 4) + 4 * case["cells"] ** 3, flops=6 * n)
    if kind == "replicas":
        n = case["sites"] * sum(b * k ** 3 for b, k, _ in _replica_sizes(case["count"], case["count"]))
    elif kind == "molecules":
        n = 48 * case["k"] ** 3
    else:
        n = case["base"] * case.get("tile", 1) ** 3 * case["sites"]
    if kind == "adjoint":   # a forward run, its recomputation, and the tangent evaluations (value and derivative)
        k = case["steps"]
        return dict(bytes=4 * k * n * 96, flops=4 * k * n * (PAIR_FLOPS + BONDED_FLOPS))
    if kind == "analysis":  # every pair within r_max once
        return dict(bytes=n * 48 + 8 * case["bins"], flops=n * 69.2 * case["r_max"] ** 3 * 12)
    state = 48 if case.get("precision") == "plain" else 96   # x, v read and written once per step
    if kind == "forces":
        return dict(bytes=n * (48 + 24), flops=2 * n * (PAIR_FLOPS + BONDED_FLOPS))
    steps = case["steps"] + (1 if case.get("energy") else 0)
    return dict(bytes=n * (state * case["steps"] + 60), flops=steps * n * (PAIR_FLOPS + BONDED_FLOPS))


# ---------------------------------------------------------------- the same in 64 bits, plainly

class _Plain:
    """One melt or molecular system in FP64 torch: pair list by cells, forces, energies, steps."""

    def __init__(self, m, bonds=None, types=None, lj_form=0):
        dev = torch.device("cuda")
        self.p = md.default_params()
        self.L, self.n, S = m["L"], len(m["pos"]), m["sites"]
        self.sites, self.lj_form = S, lj_form
        if bonds is None:
            bonds = [(k, k + 1) for k in range(S - 1)]
            types = [1] + [0] * (S - 2) + [1]
        nb = [[] for _ in range(S)]
        for a, b in bonds:
            nb[a].append(int(b))
            nb[b].append(int(a))
        ang = [(a, b, c) for b in range(S) for a in nb[b] for c in nb[b] if a < c]
        dih = [(a, b, c, d) for b in range(S) for c in nb[b] if b < c for a in nb[b] if a != c for d in nb[c]
               if d not in (a, b)]
        first = torch.arange(0, self.n, S, device=dev)[:, None, None]

        def all_of(t, w):
            return (first + torch.tensor(np.array(t).reshape(-1, w), device=dev)[None]).reshape(-1, w)
        self.bonds, self.angles, self.dih = all_of(bonds, 2), all_of(ang, 3), all_of(dih, 4)
        excl = np.eye(S, dtype=bool)
        for a, b in bonds:
            excl[a, b] = excl[b, a] = True
        for a, b, c in ang:
            excl[a, c] = excl[c, a] = True
        self.excl = torch.tensor(excl, device=dev)
        self.type = torch.tensor(np.array(types, np.int64), device=dev).repeat(self.n // S)
        self.mass = torch.tensor(np.array(self.p["mass"]), device=dev)[self.type][:, None]
        self.theta = torch.tensor([*self.p["eps"], *self.p["sigma"], self.p["kphi"]], dtype=torch.float64, device=dev)
        self.x, self.v = (torch.tensor(m[k], dtype=torch.float64, device=dev) for k in ("pos", "vel"))

    def image(self, d):
        return d - self.L * torch.round(d / self.L)

    def pairs(self, x, radius):
        """Every non-excluded pair i < j by position nearer than radius."""
        M = int(self.L // radius)
        if M < 3:
            raise ValueError("box too small")
        w = torch.remainder(x, self.L)
        c3 = (w * (M / self.L)).long().clamp_(0, M - 1)
        cell = (c3[:, 2] * M + c3[:, 1]) * M + c3[:, 0]
        order = torch.argsort(cell, stable=True)
        count = torch.bincount(cell, minlength=M ** 3)
        start = torch.cumsum(count, 0) - count
        K = int(count.max())
        slot = torch.arange(self.n, device=x.device) - start[cell[order]]
        table = torch.full((M ** 3, K), -1, dtype=torch.int64, device=x.device)
        table[cell[order], slot] = order
        ids = torch.arange(M ** 3, device=x.device)
        cx, cy, cz = ids % M, ids // M % M, ids // (M * M)
        forward = [(0, 0, 0)] + [(a, b, 1) for a in (-1, 0, 1) for b in (-1, 0, 1)] + [(a, 1, 0) for a in (-1, 0, 1)]
        found, chunk = [], max(1, 24_000_000 // (K * K))
        for ox, oy, oz in forward + [(1, 0, 0)]:
            other = (((cz + oz) % M) * M + (cy + oy) % M) * M + (cx + ox) % M
            for b in range(0, M ** 3, chunk):
                i, j = torch.broadcast_tensors(table[b:b + chunk, :, None], table[other[b:b + chunk]][:, None, :])
                keep = (i >= 0) & (j >= 0)
                if (ox, oy, oz) == (0, 0, 0):
                    keep = keep & (i < j)
                i, j = i[keep], j[keep]
                d = self.image(x[i] - x[j])
                near = d.square().sum(1) < radius * radius
                i, j = i[near], j[near]
                ok = (i // self.sites != j // self.sites) | ~self.excl[i % self.sites, j % self.sites]
                found.append(torch.stack([i[ok], j[ok]]))
        return torch.cat(found, 1)

    def coefficients(self, i, j, theta):
        t, u = self.type[i], self.type[j]
        eps = (theta[t] * theta[u]).sqrt()
        s6 = (theta[2 + t] * theta[2 + u]).sqrt() ** 6
        return 4.0 * eps * s6, 4.0 * eps * s6 * s6

    def lj(self, x, pairs):
        """Forces, energies (truncated, shifted) and virial of the listed pairs nearer than the cutoff."""
        f, e, vir = torch.zeros_like(x), x.new_zeros(2), x.new_zeros(6)
        for b in range(0, pairs.shape[1], 20_000_000):
            i, j = pairs[:, b:b + 20_000_000]
            d = self.image(x[i] - x[j])
            r2 = d.square().sum(1)
            near = r2 < RC * RC
            i, j, d, r2 = i[near], j[near], d[near], r2[near]
            c6, c12 = self.coefficients(i, j, self.theta)
            i6 = r2 ** -3
            fij = ((12.0 * c12 * i6 - 6.0 * c6) * i6 / r2)[:, None] * d
            f.index_add_(0, i, fij)
            f.index_add_(0, j, -fij)
            en = (c12 * i6 - c6) * i6
            e = e + torch.stack([en.sum(), (en - (c12 * RC ** -6 - c6) * RC ** -6).sum()])
            vir = vir + torch.stack([(d[:, a] * fij[:, c]).sum() for a, c in ((0, 0), (1, 1), (2, 2), (0, 1), (0, 2),
                                                                             (1, 2))])
        return f, e, vir

    def bonded(self, x, kphi):
        """Bond, angle and dihedral energies and the vectors they were taken from (for the virial)."""
        p = self.p
        b = self.image(x[self.bonds[:, 1]] - x[self.bonds[:, 0]])
        eb = 0.5 * p["kb"] * (b.square().sum(1).sqrt() - p["b0"]).square().sum()
        u, w = (self.image(x[self.angles[:, k]] - x[self.angles[:, 1]]) for k in (0, 2))
        th = torch.atan2(torch.linalg.cross(u, w).square().sum(1).sqrt(), (u * w).sum(1))
        ea = 0.5 * p["ka"] * (th - p["theta0"]).square().sum()
        b1, b2, b3 = (self.image(x[self.dih[:, k + 1]] - x[self.dih[:, k]]) for k in range(3))
        m, n = torch.linalg.cross(b1, b2), torch.linalg.cross(b2, b3)
        phi = torch.atan2(b2.square().sum(1).sqrt() * (b1 * n).sum(1), (m * n).sum(1))
        ed = kphi * (1.0 + torch.cos(p["n_mult"] * phi - p["phis"])).sum()
        return eb, ea, ed, (b, u, w, b1, b2, b3)

    def forces(self, x, pairs):
        xg = x.detach().requires_grad_(True)
        eb, ea, ed, _ = self.bonded(xg, self.theta[4])
        f, _, _ = self.lj(x, pairs)
        return f - torch.autograd.grad(eb + ea + ed, xg)[0]

    def energies(self):
        x = self.x
        _, e, vir = self.lj(x, self.pairs(x, RC + 0.01))
        with torch.enable_grad():
            eb, ea, ed, vec = self.bonded(x.detach().requires_grad_(True), self.theta[4])
            g = torch.autograd.grad(eb + ea + ed, vec)
        for d, q in zip(vec, g):
            vir = vir - torch.stack([(d[:, a] * q[:, c]).sum() for a, c in ((0, 0), (1, 1), (2, 2), (0, 1), (0, 2),
                                                                           (1, 2))])
        ke = 0.5 * (self.mass * self.v.square()).sum()
        out = dict(lj=e[0], lj_shifted=e[1], bond=eb, angle=ea, dihedral=ed, kinetic=ke,
                   temperature=2.0 * ke / ((3 * self.n - 3) * KB), total=e[1] + eb + ea + ed + ke,
                   pressure=(2.0 * ke + vir[:3].sum()) / (3.0 * self.L ** 3))
        out = {k: np.array([float(v.detach())]) for k, v in out.items()}
        out["virial"] = vir.detach().cpu().numpy()[None]
        return out

    def run(self, steps, ensemble="nve", T0=0.0, tau=0.1):
        """Velocity Verlet; weak coupling with the previous step's factor; or Nose-Hoover leap-frog with the
        centre-of-mass velocity of the half step removed after the drift."""
        x, v, m = self.x, self.v, self.mass
        dof = 3 * self.n - 3
        lam, xi = 1.0, 0.0
        com = torch.zeros(3, dtype=x.dtype, device=x.device)
        Q = tau * tau * T0 / (4.0 * math.pi ** 2)

        def temperature(u):
            return float((m * u.square()).sum()) / (dof * KB)
        for k in range(steps):
            if k % 10 == 0:
                pairs = self.pairs(x, RC + SKIN)
            if k == 0:
                f = self.forces(x, pairs)
            if ensemble == "vrescale":
                new = math.sqrt(1.0 + DT / tau * (T0 / temperature(v) - 1.0))
                v, lam = v * lam, new
            if ensemble == "nose_hoover":
                v = v * (1.0 - 0.5 * DT * xi) + 0.5 * DT / m * f
                x = x + DT * v
                xi += DT * (temperature(v) - T0) / Q
                com = (m * v).sum(0) / m.sum()
                f = self.forces(x, pairs)
                v = (v - com + 0.5 * DT / m * f) / (1.0 + 0.5 * DT * xi)
            else:
                v = v + 0.5 * DT / m * f
                x = x + DT * v
                f = self.forces(x, pairs)
                v = v + 0.5 * DT / m * f
        self.x, self.v = torch.remainder(x, self.L), v
        return dict(x=self.x, v=v, img=None)

    def potential(self, x, theta, pairs):
        """U (shifted or force-shifted LJ and bonded terms), differentiable in x and theta."""
        d = self.image(x[pairs[0]] - x[pairs[1]])
        r2 = d.square().sum(1)
        c6, c12 = self.coefficients(pairs[0], pairs[1], theta)
        i6 = r2 ** -3
        e = (c12 * i6 - c6) * i6 - (c12 * RC ** -6 - c6) * RC ** -6
        if self.lj_form:
            e = e - (r2.sqrt() - RC) * (6.0 * c6 * RC ** -7 - 12.0 * c12 * RC ** -13)
        return e.sum() + sum(self.bonded(x, theta[4])[:3])

    def near(self, x, pairs):
        r2 = self.image(x[pairs[0]] - x[pairs[1]]).square().sum(1)
        return pairs[:, r2 < RC * RC]

    def adjoint(self, steps, w):
        """Trajectory means of U and the squared end-to-end distance, and the gradient of w . means in theta, by
        the chain rule through velocity Verlet (each force's vector-Jacobian product from torch)."""
        S, n_chains, m = self.sites, self.n // self.sites, self.mass
        x = self.x.reshape(-1, S, 3)
        d = x[:, 1:] - x[:, :-1]
        shift = -torch.cumsum(torch.round(d / self.L), 1) * self.L
        x = torch.cat([x[:, :1], x[:, 1:] + shift], 1).reshape(-1, 3)
        v, xs, lists, obs = self.v, [], [], [0.0, 0.0]

        def value(x, pairs, theta):
            ree = x.reshape(-1, S, 3)
            ree = ((ree[:, -1] - ree[:, 0]).square().sum()) / n_chains
            return self.potential(x, theta, pairs), ree
        for k in range(steps + 1):
            if k % 10 == 0:
                wide = self.pairs(x, RC + SKIN) if self.L >= 3 * (RC + SKIN) else self.pairs(x, RC + 0.05)
            pairs = self.near(x, wide)
            xg = x.detach().requires_grad_(True)
            u, ree = value(xg, pairs, self.theta)
            f = -torch.autograd.grad(u, xg)[0]
            obs[0] += float(u.detach()) / (steps + 1)
            obs[1] += float(ree.detach()) / (steps + 1)
            xs.append(x)
            lists.append(pairs)
            if k:
                v = v + 0.5 * DT / m * f
            if k < steps:
                v = v + 0.5 * DT / m * f
                x = x + DT * v
        ax, av, cf = torch.zeros_like(x), torch.zeros_like(x), torch.zeros_like(x)
        grad = torch.zeros_like(self.theta)
        for k in range(steps, -1, -1):
            c = cf + (0.5 * DT / m * av if k else 0.0)
            xg, th = xs[k].detach().requires_grad_(True), self.theta.detach().requires_grad_(True)
            u, ree = value(xg, lists[k], th)
            g = torch.autograd.grad(u, xg, create_graph=True)[0]
            s = -(g * c).sum() + (w[0] * u + w[1] * ree) / (steps + 1)
            gx, gt = torch.autograd.grad(s, (xg, th))
            ax, grad = ax + gx, grad + gt
            cf = 0.5 * DT / m * (av + DT * ax)
            av = av + DT * ax
        return dict(obs=np.array(obs), grad=grad.cpu().numpy())

    def structure(self):
        S, m = self.sites, self.mass.reshape(-1, self.sites, 1)
        b = self.image(torch.diff(self.x.reshape(-1, S, 3), dim=1))
        x = torch.cat([torch.zeros_like(b[:, :1]), torch.cumsum(b, 1)], 1)
        com = (m * x).sum(1, keepdim=True) / m.sum(1, keepdim=True)
        rg2 = (m * (x - com).square()).sum((1, 2)) / m.sum((1, 2))
        n1, n2 = torch.linalg.cross(b[:, :-2], b[:, 1:-1]), torch.linalg.cross(b[:, 1:-1], b[:, 2:])
        cos = (n1 * n2).sum(2) / (n1.square().sum(2) * n2.square().sum(2)).sqrt()
        trans = (cos < -0.5).double().mean()
        return dict(g=None, counts=None, r_ee=x[:, -1].cpu().numpy(), rg2=rg2.cpu().numpy(),
                    trans=np.array([float(trans)]))


def exact(case, seed):
    kind = case["kind"]
    if kind == "binning":
        return None
    if kind == "replicas":
        outs = [_Plain(m).run(case["steps"], "vrescale", m["T"]) for m in _replica_melts(case, seed)]
        return dict(x=torch.cat([o["x"] for o in outs]), v=torch.cat([o["v"] for o in outs]), img=None)
    if kind == "molecules":
        m, (bonds, types) = _molecules(case["k"], case["mixed_types"], seed)
        return _Plain(m, bonds, types).run(case["steps"])
    m = _melt(case["base"], case.get("tile", 1), case["sites"], seed, case.get("T", 500.0))
    plain = _Plain(m, lj_form=case.get("lj_form", 0))
    if kind == "adjoint":   # 0.2 s a step at 7,500 sites
        return plain.adjoint(case["steps"], (1.0, 0.5))
    if kind == "analysis":
        return plain.structure()
    if kind == "forces":
        return dict(forces=plain.forces(plain.x, plain.pairs(plain.x, RC + 0.01)), energy=plain.energies())
    out = plain.run(case["steps"], case["ensemble"], case["T"], 0.1)
    if case["frame"] == "host":
        out = {k: None if v is None else v.cpu().numpy() for k, v in out.items()}
    if case["energy"]:
        out["energy"] = plain.energies()
    return out
