"""The time steps that users of this framework run, as cases to time and compare.

A case is one pass of a program that samples a simulation: advance every
system by `steps` time steps (md_step) and read the state into the program's
own device tensors (md_get_state_device), or, for `io` = "host", couple the
step to a host program: restore a state from host memory, one step, read the
result back to the host. Passes follow one another on the same handle, as
the samples of one trajectory do.

The systems are this repository's workloads (area fractions, cutoffs, bonds,
time steps, tolerances and neighbour-list sizes of its benchmark), placed by
random sequential addition in torch so that making them is quick. Positions
and the float64 path's velocities are returned as the float64 the interface
gives; the mixed path's velocities, which are integrated from float32 forces
and float32 noise, are kept as float32 by the program.
"""
from __future__ import annotations

import itertools
import math

import numpy as np
import torch

from paper_1411_3019_gb300 import md

D0 = 2.0 ** (1.0 / 6.0)  # WCA cutoff
DEV = "cuda" if torch.cuda.is_available() else "cpu"
F64 = torch.float64

# Neighbour list of each model where `lists` is set: (skin, entries per particle).
LISTS = {"sphere": (0.4, 64), "ellipsoid_torus": (0.4, 64), "replicas": (0.4, 64), "beads": (0.4, 128),
         "bump_crowders": (0.4, 64), "capsids": (0.4, 256), "thylakoids": (0.4, 64), "plane2d": (0.5, 64),
         "lj_liquid": (0.3, 128), "nve": (0.3, 128)}


def _case(name, model, n, systems=1, precision="mixed", lists=True, steps=20, io="device"):
    return dict(name=name, model=model, n=n, systems=systems, precision=precision, lists=lists, steps=steps, io=io)


def listed():
    return [
        # The smallest call: one step of a thousand particles on a sphere, sampled after every step
        # (a program that drives the step itself), with the interface's defaults (a cell list every step).
        _case("sphere_1k_sampled", "sphere", 1000, lists=False, steps=1),
        # The plain float64 path on the paper's sphere of a thousand WCA particles.
        _case("sphere_1k_fp64", "sphere", 1000, precision="fp64", steps=20),
        # Energy conservation study: four small systems of smoothed Lennard-Jones particles on a sphere, a
        # cylinder, a torus and a plane, float64, no thermostat, energies read with the state.
        _case("nve_surfaces_fp64", "nve", 500, systems=4, precision="fp64", lists=False, steps=20),
        # A host program coupled to every step: restore from pinned host arrays, step, read back to the host.
        _case("sphere_40k_coupled", "sphere", 40_001, steps=1, io="host"),
        # Bead molecules on a spherical template: bonds, exclusions, five types, two cutoffs.
        _case("beads_100k", "beads", 100_000, steps=20),
        # A dense liquid with a long cutoff, cell list every step (the interface's default).
        _case("lj_liquid_97k", "lj_liquid", 97_336, lists=False, steps=10),
        # The float64 path at size: ellipsoid and torus.
        _case("ellipsoid_torus_60k_fp64", "ellipsoid_torus", 60_000, systems=2, precision="fp64", steps=20),
        # The benchmark's headline: 200,000 particles on an ellipsoid and 50,000 on a torus.
        _case("ellipsoid_torus_250k", "ellipsoid_torus", 250_000, systems=2, steps=50),
        # Virus-capsid assembly: cones of four beads with bonds, bend angles and a spherical wall.
        _case("capsids_1024", "capsids", 245_760, systems=1024, steps=20),
        # Crowded diffusion on the thylakoid composite surface.
        _case("thylakoids_128", "thylakoids", 320_000, systems=128, steps=20),
        # An ensemble of independent spheres of 50 to 2,000 particles.
        _case("replicas_512", "replicas", sum(_replicas(512)[0]), systems=512, steps=20),
        # Particles on a Gaussian bump in a bath of free crowders between walls.
        _case("bump_crowders_1m", "bump_crowders", 1_000_000, steps=20),
    ]


def _replicas(systems):
    """Sizes and radii of an ensemble of spheres: 50 to 2,000 particles, radius 5 to 40, area fraction 0.05 to 0.5."""
    r = np.random.RandomState(systems)
    counts, radii = [], []
    while len(counts) < systems:
        m, rad = int(r.randint(50, 2001)), 5 + 35 * r.rand()
        if 0.05 <= m * D0 * D0 / (16 * rad * rad) <= 0.5:
            counts.append(m)
            radii.append(rad)
    return counts, radii


def draw(rng):
    """One more case of the same ranges."""
    model = rng.choice(["sphere", "sphere", "ellipsoid_torus", "replicas", "beads", "bump_crowders", "capsids",
                        "thylakoids", "plane2d", "lj_liquid", "nve"])
    lo, hi = {"sphere": (400, 300_000), "ellipsoid_torus": (5_000, 300_000), "replicas": (10_000, 560_000),
              "beads": (5_000, 150_000), "bump_crowders": (30_000, 600_000), "capsids": (4_800, 245_760),
              "thylakoids": (5_000, 320_000), "plane2d": (2_000, 400_000), "lj_liquid": (4_000, 110_000),
              "nve": (200, 4_000)}[model]
    n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    systems, lists, precision, io = 1, rng.random() < 0.8, "mixed", "device"
    if model == "sphere" and rng.random() < 0.3:
        io = "host"
    if model in ("sphere", "ellipsoid_torus", "beads", "plane2d") and rng.random() < 0.3:
        precision, n = "fp64", max(lo, n // 6)
    if model == "ellipsoid_torus":
        systems = 2
    elif model == "replicas":
        systems = max(8, n // 1100)
        n = sum(_replicas(systems)[0])
    elif model == "beads":
        n -= n % 5
    elif model == "capsids":
        systems = max(4, n // 240)
        n = 240 * systems
    elif model == "thylakoids":
        systems = max(2, n // rng.randint(2000, 2800))
        n = n // systems * systems
    elif model == "lj_liquid":
        n = max(15, round(n ** (1 / 3))) ** 3
    elif model == "nve":
        systems, precision = 4, rng.choice(["fp64", "fp64", "mixed"])
    steps = 1 if io == "host" else rng.choice([1, 5, 10, 20])
    return {k: v for k, v in _case("", model, n, systems, precision, lists, steps, io).items() if k != "name"}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _close_pairs(pts, grp, reach, lo, L, periodic):
    """Pairs (a, b) of points of one group closer than `reach`: cells of that edge, half of the 27 neighbours."""
    n = pts.shape[0]
    nc, cell = [], []
    for d in range(3):
        if periodic[d]:
            m = int(L[d] / reach)
            c = torch.remainder(torch.floor((pts[:, d] - lo[d]) / (L[d] / m)).long(), m)
        else:
            c = torch.floor((pts[:, d] - pts[:, d].min()) / reach).long() + 1
            m = int(c.max()) + 2
        nc.append(m)
        cell.append(c)
    key = ((grp * nc[2] + cell[2]) * nc[1] + cell[1]) * nc[0] + cell[0]
    key, order = torch.sort(key, stable=True)
    pts, grp, cell = pts[order], grp[order], [c[order] for c in cell]
    at = torch.arange(n, device=pts.device)
    found = []
    for off in [o for o in itertools.product((-1, 0, 1), repeat=3) if o >= (0, 0, 0)]:
        q = [torch.remainder(cell[d] + off[d], nc[d]) if periodic[d] else cell[d] + off[d] for d in range(3)]
        k = ((grp * nc[2] + q[2]) * nc[1] + q[1]) * nc[0] + q[0]
        left, right = torch.searchsorted(key, k), torch.searchsorted(key, k, right=True)
        if off == (0, 0, 0):
            left = at + 1
        count = right - left
        i = torch.repeat_interleave(at, count)
        j = torch.arange(i.numel(), device=pts.device) + (left - torch.cumsum(count, 0) + count)[i]
        d = _images(pts[i] - pts[j], L, periodic)
        near = (d * d).sum(1) < reach * reach
        found.append((order[i[near]], order[j[near]]))
    return torch.cat([f[0] for f in found]), torch.cat([f[1] for f in found])


def _images(d, L, periodic):
    for k in range(3):
        if periodic[k]:
            d[:, k] -= L[k] * torch.round(d[:, k] / L[k])
    return d


def _place(sample, counts, dmin, gen, lo=(0, 0, 0), L=(1, 1, 1), periodic=(0, 0, 0), ratio=4.0, fixed=None):
    """Random sequential addition: counts[g] points of sample(groups, gen) in group g, none closer than dmin to an
    earlier one of its group (nor to `fixed` points of group 0); all groups at once. Returns them group by group."""
    need = torch.tensor(counts, device=DEV)
    have = torch.zeros_like(need)
    fx = torch.empty((0, 3), dtype=F64, device=DEV) if fixed is None else fixed
    x, g = fx, torch.zeros(fx.shape[0], dtype=torch.long, device=DEV)
    for _ in range(200):
        lack = need > have
        if not bool(lack.any()):
            break
        more = torch.where(lack, ((need - have) * ratio).long() + 24, torch.zeros_like(need))
        cx, cg = sample(torch.repeat_interleave(torch.arange(len(counts), device=DEV), more), gen)
        old = lack[g]
        px, pg = torch.cat([x[old], cx]), torch.cat([g[old], cg])
        m = int(old.sum())
        a, b = _close_pairs(px, pg, dmin, lo, L, periodic)
        first, second = torch.minimum(a, b), torch.maximum(a, b)
        state = torch.zeros(px.shape[0], dtype=torch.int8, device=DEV)  # 0 open, 1 placed, 2 rejected
        state[:m] = 1
        while bool((state == 0).any()):
            hit = torch.zeros_like(state, dtype=torch.bool)
            hit[second[state[first] == 1]] = True
            state[hit & (state == 0)] = 2
            wait = torch.zeros_like(hit)
            wait[second[state[first] == 0]] = True
            state[~wait & (state == 0)] = 1
        new = (state[m:] == 1).nonzero()[:, 0]
        ng = cg[new]
        rank = torch.arange(ng.numel(), device=DEV) - torch.searchsorted(ng, ng)
        new = new[rank < (need - have)[ng]]
        have += torch.bincount(cg[new], minlength=len(counts))
        x, g = torch.cat([x, cx[new]]), torch.cat([g, cg[new]])
    x, g = x[fx.shape[0]:], g[fx.shape[0]:]
    return x[torch.sort(g, stable=True).indices].contiguous()


def _rand(n, gen):
    return torch.rand(n, dtype=F64, device=DEV, generator=gen)


def _unit(n, gen):
    v = torch.randn((n, 3), dtype=F64, device=DEV, generator=gen)
    return v / v.norm(dim=1, keepdim=True)


def _on_surface(kind, p, L=None, lo=None):
    """Sampler of points uniform by area on one surface centred at the origin."""
    def sample(groups, gen):
        n = groups.numel()
        if kind == "sphere":
            return p[0] * _unit(n, gen), groups
        if kind == "ellipsoid":
            v = _unit(n, gen)
            a = torch.tensor(p[:3], dtype=F64, device=DEV)
            w = (v * (a.prod() / a)).norm(dim=1)
            keep = _rand(n, gen) < w / float((a.prod() / a).max())
            return (v * a)[keep], groups[keep]
        if kind == "torus":
            th, ph = 2 * math.pi * _rand(n, gen), 2 * math.pi * _rand(n, gen)
            keep = _rand(n, gen) < (p[0] + p[1] * torch.cos(th)) / (p[0] + p[1])
            rho = p[0] + p[1] * torch.cos(th)
            return torch.stack([rho * torch.cos(ph), rho * torch.sin(ph), p[1] * torch.sin(th)], 1)[keep], groups[keep]
        if kind == "cylinder":
            ph = 2 * math.pi * _rand(n, gen)
            return torch.stack([p[0] * torch.cos(ph), p[0] * torch.sin(ph), lo[2] + L[2] * _rand(n, gen)], 1), groups
        if kind == "gaussian_bump":
            x, y = lo[0] + L[0] * _rand(n, gen), lo[1] + L[1] * _rand(n, gen)
            z = p[0] * torch.exp(-(x * x + y * y) / (2 * p[1] ** 2))
            slope = z / p[1] ** 2 * torch.sqrt(x * x + y * y)
            keep = _rand(n, gen) < torch.sqrt(1 + slope ** 2) / math.sqrt(1 + (p[0] / (p[1] * math.sqrt(math.e))) ** 2)
            return torch.stack([x, y, z], 1)[keep], groups[keep]
        x, y = lo[0] + L[0] * _rand(n, gen), lo[1] + L[1] * _rand(n, gen)  # plane, xy2d
        return torch.stack([x, y, torch.zeros_like(x)], 1), groups
    return sample


def _on_thylakoid(p, Lz):
    """Sampler of points uniform by area on the thylakoid composite (centre at the origin, z periodic)."""
    Rb, Lx, Rc, Lb = p
    xf = Lb / 2 + Rc  # the face planes at x = -xf and xf
    area = [4 * math.pi * Rc * Lz, 2 * math.pi * Rb * Lb,
            2 * (math.pi * Rc * Rc * (math.pi - 2) + math.pi ** 2 * Rc * Rb), 8 * Lx * Lz]

    def sample(groups, gen):
        n = groups.numel()
        part = torch.multinomial(torch.tensor(area, dtype=F64, device=DEV).expand(1, 4), n, True, generator=gen)[0]
        r1, r2, r3, r4 = (_rand(n, gen) for _ in range(4))
        side = torch.where(r3 < 0.5, -1.0, 1.0).to(F64)
        z = Lz * (r1 - 0.5)
        # corners: quarter cylinders about (side (xf + Rc [+ Lx]), +- Lx/2), facing out of the block
        far, up = torch.floor(2 * (2 * r3 % 1)), torch.where(r4 < 0.5, -1.0, 1.0).to(F64)
        an = r2 * math.pi / 2
        out_x = torch.where(far == 1, side, -side)
        corner = torch.stack([side * (xf + Rc + far * Lx) + out_x * Rc * torch.cos(an),
                              up * (Lx / 2 + Rc * torch.sin(an)), z], 1)
        ph = 2 * math.pi * r2
        bridge = torch.stack([Lb * (r1 - 0.5), Rb * torch.cos(ph), Rb * torch.sin(ph)], 1)
        al = r1 * math.pi / 2
        rr = Rb + Rc - Rc * torch.cos(al)
        conn = torch.stack([side * (Lb / 2 + Rc * torch.sin(al)), rr * torch.cos(ph), rr * torch.sin(ph)], 1)
        face = torch.floor(4 * r4)  # 0: towards the bridge, 1: away from it, 2 and 3: the sides
        t = Lx * (r2 - 0.5)
        plane = torch.stack([torch.where(face < 2, side * (xf + face * (Lx + 2 * Rc)), side * (xf + Rc + Lx / 2) + t),
                             torch.where(face < 2, t, (2 * face - 5) * (Lx / 2 + Rc)), z], 1)
        x = torch.where((part == 0)[:, None], corner, torch.where((part == 1)[:, None], bridge,
                        torch.where((part == 2)[:, None], conn, plane)))
        hole = (part == 3) & (face == 0) & (torch.hypot(t, z) < Rb + Rc)
        keep = ~hole & ((part != 2) | (_rand(n, gen) < rr / (Rb + Rc)))
        return x[keep], groups[keep]
    return sample


def _params(precision, nt=1, **over):
    one = np.ones((nt, nt))
    prm = dict(dt=0.002, kT=1.0, gamma=1.0, rattle_tol=1e-12 if precision == "fp64" else 1e-10, max_newton=30,
               precision=precision, ntypes=nt, mass=[1.0] * nt, eps=one.copy(), sigma=one.copy(), rcut=D0 * one,
               box_lo=(0.0,) * 3, box_hi=(0.0,) * 3, periodic=(0, 0, 0))
    prm.update(over)
    return prm


def _surface(kind, *p):
    return {"kind": kind, "center": (0.0, 0.0, 0.0), "p": tuple(p)}


def _box(lo, hi, periodic):
    return dict(box_lo=tuple(map(float, lo)), box_hi=tuple(map(float, hi)), periodic=periodic)


def _systems(case, seed):
    """surfaces, params, counts, x, type, constrained of a case's systems."""
    gen = torch.Generator(device=DEV)
    gen.manual_seed(int(seed))
    model, n, ns, prec = case["model"], case["n"], case["systems"], case["precision"]
    key = int(seed) & 0xFFFFFFFF
    typ = con = None
    if model == "sphere":
        # the thousand-particle sphere of the paper's size is crowded (R = 10), larger ones are at area fraction 0.4
        R = 10.0 if n <= 1000 else math.sqrt(n * D0 * D0 / (16 * 0.4))
        surfaces, prms, counts = [_surface("sphere", R)], [_params(prec, seed=key, dt=0.001 if n <= 1000 else 0.002)], [n]
        x = _place(_on_surface("sphere", (R,)), counts, 0.8 if n <= 1000 else 1.0, gen)
    elif model == "ellipsoid_torus":
        n_tor = n // 5
        s, t = 1.66 * math.sqrt((n - n_tor) / 200_000), math.sqrt(n_tor / 50_000)
        ax, ring = (150 * s, 120 * s, 90 * s), (120 * t, 40 * t)
        surfaces, counts = [_surface("ellipsoid", *ax), _surface("torus", *ring)], [n - n_tor, n_tor]
        prms = [_params(prec, seed=key, replica=k) for k in range(2)]
        x = torch.cat([_place(_on_surface(q["kind"], q["p"]), [m], 1.0, gen) for q, m in zip(surfaces, counts)])
    elif model == "replicas":
        counts, R = _replicas(ns)
        surfaces = [_surface("sphere", q) for q in R]
        prms = [_params(prec, seed=key, replica=k) for k in range(ns)]
        Rt = torch.tensor(R, dtype=F64, device=DEV)
        x = _place(lambda g, gn: (Rt[g][:, None] * _unit(g.numel(), gn), g), counts, 1.0, gen)
    elif model == "beads":
        mol = n // 5
        R = 60 * math.sqrt(mol / 20_000)
        one = np.ones((5, 5))
        eps, rc = one.copy(), D0 * one
        eps[3, 3], rc[3, 3] = 2.0, 2.5
        e = R + 15.0
        prms = [_params(prec, 5, eps=eps, rcut=rc, seed=key, beads_per_mol=5, bond_k=100.0, bond_r0=1.0,
                        exclude_intramol=1, **_box((-e,) * 3, (e,) * 3, (0, 0, 0)))]
        surfaces, counts = [_surface("sphere", R)], [n]
        u = _place(_on_surface("sphere", (R,)), [mol], 1.0, gen) / R
        x = (u[:, None, :] * (R + torch.arange(5, dtype=F64, device=DEV))[None, :, None]).reshape(-1, 3)
        typ = torch.arange(n, device=DEV) % 5
        con = typ == 0
    elif model == "capsids":
        sig = np.array([1.0, 1.35, 1.75, 1.0])
        sij = 0.5 * (sig[:, None] + sig[None, :])
        rc = D0 * sij
        rc[1, 1] = rc[2, 2] = 4.0
        r0 = D0 * sij / 2
        R = math.sqrt(60 * 0.81 / 0.45 / 4)
        rad = R + np.concatenate([[0.0], np.cumsum([r0[0, 1], r0[1, 2], r0[2, 3]])])
        e = rad[3] + 6.0
        prms = [_params(prec, 4, eps=4.0 * np.ones((4, 4)), sigma=sij, rcut=rc, mass=list(sig ** 3), seed=key, replica=k,
                        beads_per_mol=4, bond_k=50.0, bond_r0=0.0, bond_r0_mix=1, angle_k=250.0, angle_theta0=math.pi,
                        exclude_intramol=1, wall_enable=1, wall_kind=1, wall_radius=R - 1.0, wall_eps=1.0,
                        wall_sigma=1.0, **_box((-e,) * 3, (e,) * 3, (0, 0, 0))) for k in range(ns)]
        surfaces, counts = [_surface("sphere", R)] * ns, [240] * ns
        u = _place(_on_surface("sphere", (R,)), [60] * ns, 1.8, gen, ratio=12.0) / R
        x = (u[:, None, :] * torch.tensor(rad, dtype=F64, device=DEV)[None, :, None]).reshape(-1, 3)
        typ = torch.arange(n, device=DEV) % 4
        con = typ == 0
    elif model == "thylakoids":
        p, Lz = (1.5, 15.0, 3.0, 10.0), 30.0
        ex, ey = 5.0 + 3.0 + 21.0 + 3.0, 13.5
        prms = [_params(prec, seed=key, replica=k, **_box((-ex, -ey, -Lz / 2), (ex, ey, Lz / 2), (0, 0, 1)))
                for k in range(ns)]
        surfaces, counts = [_surface("thylakoid", *p)] * ns, [n // ns] * ns
        x = _place(_on_thylakoid(p, Lz), counts, 0.9, gen, (-ex, -ey, -Lz / 2), (1.0, 1.0, Lz), (0, 0, 1))
    elif model == "bump_crowders":
        n_surf = n // 10
        s = math.sqrt(n_surf / 100_000)
        L, A, w = 495.8 * s, 33.05 * s, 24.79 * s
        h = (n - n_surf) * math.pi * D0 ** 3 / 6 / 0.2 / (L * L)
        zlo, zhi = -h / 2 - 0.5, A + h / 2 + 0.5
        box = _box((-L / 2, -L / 2, zlo - 2), (L / 2, L / 2, zhi + 2), (1, 1, 0))
        prms = [_params(prec, seed=key, wall_enable=1, wall_lo_z=zlo, wall_hi_z=zhi, wall_eps=1.0, wall_sigma=1.0, **box)]
        surfaces, counts = [_surface("gaussian_bump", A, w)], [n]
        lo, Ls = (-L / 2, -L / 2, 0.0), (L, L, 1.0)
        xs = _place(_on_surface("gaussian_bump", (A, w), Ls, lo), [n_surf], 1.0, gen, lo, Ls, (1, 1, 0))

        def bath(g, gn):
            q = torch.stack([_rand(g.numel(), gn) for _ in range(3)], 1)
            return q * torch.tensor([L, L, zhi - zlo - 2 * D0], dtype=F64, device=DEV) + torch.tensor(
                [-L / 2, -L / 2, zlo + D0], dtype=F64, device=DEV), g
        x = torch.cat([xs, _place(bath, [n - n_surf], 1.0, gen, lo, Ls, (1, 1, 0), 2.0, xs)])
        con = torch.arange(n, device=DEV) < n_surf
    elif model == "plane2d":
        L = math.sqrt(n * math.pi * D0 * D0 / 4 / 0.4)
        prms = [_params(prec, seed=key, **_box((-L / 2, -L / 2, -1.0), (L / 2, L / 2, 1.0), (1, 1, 0)))]
        surfaces, counts = [_surface("xy2d")], [n]
        lo, Ls = (-L / 2, -L / 2, 0.0), (L, L, 1.0)
        x = _place(_on_surface("xy2d", (), Ls, lo), [n], 1.0, gen, lo, Ls, (1, 1, 0))
        con = torch.zeros(n, dtype=torch.bool, device=DEV)
    elif model == "lj_liquid":
        k, a = round(n ** (1 / 3)), 1.0833
        L = k * a
        prms = [_params(prec, seed=key, dt=0.001, rcut=2.5 * np.ones((1, 1)), **_box((-L / 2,) * 3, (L / 2,) * 3, (1, 1, 1)))]
        surfaces, counts = [_surface("none")], [n]
        g = torch.arange(k, dtype=F64, device=DEV)
        grid = torch.stack(torch.meshgrid(g, g, g, indexing="ij"), -1).reshape(-1, 3)
        x = (grid + 0.5) * a - L / 2 + 0.12 * (torch.rand((n, 3), dtype=F64, device=DEV, generator=gen) - 0.5)
        con = torch.zeros(n, dtype=torch.bool, device=DEV)
    else:  # nve: the four surfaces of the energy study at area fraction 0.3
        area = n * math.pi * D0 * D0 / 4 / 0.3
        Rc, rt = 6.0, 3.0
        Lc, Lp = area / (2 * math.pi * Rc), math.sqrt(area)
        surfaces = [_surface("sphere", math.sqrt(area / (4 * math.pi))), _surface("cylinder", Rc, 2.0),
                    _surface("torus", max(area / (4 * math.pi ** 2 * rt), 4.5), rt), _surface("plane", 0.0, 0.0, 1.0)]
        boxes = [{}, _box((-9, -9, -Lc / 2), (9, 9, Lc / 2), (0, 0, 1)), {},
                 _box((-Lp / 2, -Lp / 2, -3), (Lp / 2, Lp / 2, 3), (1, 1, 0))]
        prms = [_params(prec, seed=key, replica=k, dt=0.0005, gamma=0.0, pair_form=1, rcut=2.5 * np.ones((1, 1)), **b)
                for k, b in enumerate(boxes)]
        counts = [n] * 4
        parts = []
        for q, b in zip(surfaces, boxes):
            lo = b.get("box_lo", (0.0,) * 3)
            Ls = tuple(h - l for h, l in zip(b.get("box_hi", (1.0,) * 3), lo))
            parts.append(_place(_on_surface(q["kind"], q["p"], Ls, lo), [n], 1.0, gen, lo, Ls, b.get("periodic", (0, 0, 0))))
        x = torch.cat(parts)
    if case["lists"]:
        for q in prms:
            q["cell_size"] = float(max(map(max, q["rcut"]))) + LISTS[model][0]
    total = sum(counts)
    typ = torch.zeros(total, dtype=torch.int32, device=DEV) if typ is None else typ.to(torch.int32)
    con = torch.ones(total, dtype=torch.uint8, device=DEV) if con is None else con.to(torch.uint8)
    mass = torch.tensor(prms[0]["mass"], dtype=F64, device=DEV)[typ.long()]
    v = torch.randn((total, 3), dtype=F64, device=DEV, generator=gen) / torch.sqrt(mass)[:, None]
    if model == "plane2d":
        v[:, 2] = 0.0
    return surfaces, prms, counts, x.contiguous(), v, typ, con


class _Handle:
    def __init__(self, h):
        self.h = h

    def __del__(self):
        try:
            md.md_destroy(self.h)
        except Exception:  # noqa: BLE001 (the interpreter is going away)
            pass


HOST_STEP = 1000  # step counter of a coupled program's state


def prepare(case, seed):
    surfaces, prms, counts, x, v, typ, con = _systems(case, seed)
    h = md.md_create(surfaces[0], prms[0], counts[0]) if len(counts) == 1 else md.md_create_batch(surfaces, prms, counts)
    st = {"handle": _Handle(h), "case": case}
    if case["lists"]:
        md.md_set_neighbor_list(h, *LISTS[case["model"]])
    if DEV == "cuda":
        torch.cuda.current_stream().synchronize()  # the handle works on a stream of its own
    md.md_set_state_device(h, x, v, typ, None, con)
    if case["io"] == "host":
        st["x"], st["p"] = (torch.empty(x.shape, dtype=F64, pin_memory=True).numpy() for _ in range(2))
        st["x"][:] = x.cpu().numpy()
        st["p"][:] = _project(surfaces, counts, x, v, con).cpu().numpy()  # mass 1
    else:
        st["x"], st["v"] = torch.empty_like(x), torch.empty_like(v)
    return st


def run(st):
    case, h = st["case"], st["handle"].h
    mixed = case["precision"] == "mixed"
    if case["io"] == "host":
        md.md_restore(h, st["x"], st["p"], HOST_STEP)
        md.md_step(h, case["steps"])
        got = md.md_get_state(h, ("x", "v"))
        return {"x": got["x"], "v": got["v"].astype(np.float32) if mixed else got["v"], "step": got["step"]}
    md.md_step(h, case["steps"])
    md.md_get_state_device(h, st["x"], st["v"])
    out = {"x": st["x"], "v": st["v"].float() if mixed else st["v"]}
    if case["model"] == "nve" and not mixed:
        obs = md.md_observables(h)
        out["energy"] = np.array([[o["kinetic"], o["potential"]] for o in obs])
    return out


def work(case):
    """State read once (x and p) and written once (x and v); for every particle and step the noise, the force
    combination and the constraint (about 300 operations) and its pairs in range (about 40 operations each)."""
    n = 4 * case["n"] if case["model"] == "nve" else case["n"]
    pairs = {"lj_liquid": 52.0, "capsids": 30.0, "beads": 6.0, "bump_crowders": 3.0, "nve": 8.0}.get(case["model"], 4.0)
    return {"bytes": n * (96.0 if case["precision"] == "fp64" or case["io"] == "host" else 84.0),
            "flops": case["steps"] * n * (300.0 + 40.0 * pairs / 2)}


# ---------------------------------------------------------------------------
# the same steps in 64 bits, in plain torch
# ---------------------------------------------------------------------------
def _piece(p, x, L):
    """Piece of the thylakoid at x (held for a solve): type, sign or 0, two centre coordinates, radius."""
    Rb, Lx, Rc, Lb = p
    xf = Lb / 2 + Rc
    dz = x[:, 2] - L[2] * torch.round(x[:, 2] / L[2])
    r = torch.hypot(x[:, 1], dz)
    side = torch.where(x[:, 0] <= 0, -1.0, 1.0).to(F64)
    inner = xf + Rc  # inner square: side * [inner, inner + Lx] in x, +- Lx/2 in y
    u = side * x[:, 0]
    ex = torch.where(u < inner, u - inner, torch.where(u > inner + Lx, u - inner - Lx, torch.zeros_like(u)))
    y = x[:, 1]
    ey = torch.where(y < -Lx / 2, y + Lx / 2, torch.where(y > Lx / 2, y - Lx / 2, torch.zeros_like(y)))
    inside = (ex == 0) & (ey == 0)
    dxl, dxh, dyl, dyh = u - (inner - Rc), inner + Lx + Rc - u, y + Lx / 2 + Rc, Lx / 2 + Rc - y
    nearx = torch.minimum(dxl, dxh) <= torch.minimum(dyl, dyh)
    ex = torch.where(inside & nearx, torch.where(dxl < dxh, -1.0, 1.0).to(F64), ex)
    ey = torch.where(inside & ~nearx, torch.where(dyl < dyh, -1.0, 1.0).to(F64), ey)
    kind = torch.where(ex != 0, 0, 1)
    kind = torch.where((ex != 0) & (ey != 0), 2, kind)
    kind = torch.where((kind == 0) & (ex < 0) & (r < Rb + Rc), 4, kind)
    mid = (x[:, 0].abs() < xf) & (r < Rb + Rc)
    kind = torch.where(mid, torch.where(x[:, 0].abs() <= Lb / 2, 3, 4), kind)
    side = torch.where(mid & (x[:, 0] > 0), 1.0, torch.where(mid, -1.0, side))
    c0 = side * torch.where(kind == 2, torch.where(ex < 0, inner, inner + Lx),
                            torch.where(kind == 4, Lb / 2, torch.where(ex < 0, inner - Rc, inner + Lx + Rc)))
    c1 = torch.where(kind == 2, torch.sign(ey) * Lx / 2, torch.sign(ey) * (Lx / 2 + Rc))
    return kind, c0, c1


def _g(kind, p, x, L, held=None):
    """g and grad g of a surface; p is a tensor of shape parameters, or one row for each point."""
    if kind == "plane":
        n = torch.zeros_like(x)
        n[:, 2] = 1.0
        return x[:, 2].clone(), n
    if kind == "sphere":
        return (x * x).sum(1) - p[..., 0] ** 2, 2 * x
    if kind == "ellipsoid":
        w = x / p[:3] ** 2
        return (w * x).sum(1) - 1, 2 * w
    if kind == "cylinder":
        y = x.clone()
        y[:, 2] = 0.0
        return (y * y).sum(1) - p[0] ** 2, 2 * y
    if kind == "torus":
        rho = torch.hypot(x[:, 0], x[:, 1])
        t = rho - p[0]
        n = 2 * x
        n[:, :2] *= (t / rho)[:, None]
        return t * t + x[:, 2] ** 2 - p[1] ** 2, n
    if kind == "gaussian_bump":
        d = x[:, :2] - torch.tensor(L[:2], dtype=F64, device=x.device) * torch.round(
            x[:, :2] / torch.tensor(L[:2], dtype=F64, device=x.device))
        e = p[0] * torch.exp(-(d * d).sum(1) / (2 * p[1] ** 2))
        return x[:, 2] - e, torch.cat([e[:, None] * d / p[1] ** 2, torch.ones_like(e)[:, None]], 1)
    k, c0, c1 = held  # thylakoid
    Rb, Rc = float(p[0]), float(p[2])
    dz = x[:, 2] - L[2] * torch.round(x[:, 2] / L[2])
    a, y, zero = x[:, 0] - c0, x[:, 1], torch.zeros_like(dz)
    r = torch.hypot(y, dz)
    b, t = y - c1, r - (Rb + Rc)
    q = 2 * t / torch.where(r > 0, r, torch.ones_like(r))
    # a plane's gradient is taken along +x or +y: its sign changes neither g = 0 nor the constrained motion
    g = torch.where(k == 0, a, torch.where(k == 1, b, torch.where(k == 2, a * a + b * b - Rc * Rc, torch.where(
        k == 3, r * r - Rb * Rb, a * a + t * t - Rc * Rc))))
    nx = torch.where(k == 0, zero + 1, torch.where((k == 1) | (k == 3), zero, 2 * a))
    ny = torch.where(k == 0, zero, torch.where(k == 1, zero + 1, torch.where(k == 2, 2 * b, torch.where(k == 3, 2 * y, q * y))))
    nz = torch.where(k == 3, 2 * dz, torch.where(k == 4, q * dz, zero))
    return g, torch.stack([nx, ny, nz], 1)


def _parts(surfaces, counts, con):
    """(kind, parameters, indexes of the constrained particles) of each surface kind; spheres of a batch together."""
    ends = np.cumsum([0] + list(counts))
    got = []
    for kind in dict.fromkeys(s["kind"] for s in surfaces):
        which = [k for k, s in enumerate(surfaces) if s["kind"] == kind]
        if kind in ("none", "xy2d"):
            continue
        at = torch.cat([torch.arange(ends[k], ends[k + 1], device=DEV) for k in which])
        sub = con[at] != 0
        p = torch.tensor(surfaces[which[0]]["p"], dtype=F64, device=DEV)
        if kind == "sphere":
            p = torch.repeat_interleave(torch.tensor([surfaces[k]["p"][0] for k in which], dtype=F64, device=DEV),
                                        torch.tensor([counts[k] for k in which], device=DEV))[sub][:, None]
        got.append((kind, p, at[sub]))
    return got


def _lengths(prm):
    return [float(h - l) for h, l in zip(prm["box_hi"], prm["box_lo"])]


def _project(surfaces, counts, x, v, con, L=None):
    """v without its normal part on constrained particles."""
    v = v.clone()
    for kind, p, at in _parts(surfaces, counts, con):
        held = _piece([float(q) for q in p], x[at], L) if kind == "thylakoid" else None
        _, n = _g(kind, p, x[at], L, held)
        v[at] -= ((n * v[at]).sum(1) / (n * n).sum(1))[:, None] * n
    return v


def _normals(seed, replica, pid, k):
    """Three normals of each particle at step k: Philox4x32-10 (Salmon et al., SC'11), then Box-Muller."""
    m = 0xFFFFFFFF
    c = [pid, torch.full_like(pid, k & m), torch.full_like(pid, k >> 32), torch.zeros_like(pid)]
    k0, k1 = torch.full_like(pid, seed & m), replica
    for r in range(10):
        if r:
            k0, k1 = (k0 + 0x9E3779B9) & m, (k1 + 0xBB67AE85) & m
        a, b = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57  # modulo 2^64
        c = [((b >> 32) & m) ^ c[1] ^ k0, b & m, ((a >> 32) & m) ^ c[3] ^ k1, a & m]
    u = [((w >> 9).to(F64) + 0.5) * 2.0 ** -23 for w in c]
    r01, r23 = torch.sqrt(-2 * torch.log(u[0])), torch.sqrt(-2 * torch.log(u[2]))
    return torch.stack([r01 * torch.cos(2 * math.pi * u[1]), r01 * torch.sin(2 * math.pi * u[1]),
                        r23 * torch.cos(2 * math.pi * u[3])], 1)


class _Exact:
    def __init__(self, case, seed):
        self.surfaces, self.prms, self.counts, self.x, self.v, typ, self.con = _systems(case, seed)
        prm = self.prm = self.prms[0]
        self.typ, self.n = typ.long(), self.x.shape[0]
        f = lambda a: torch.tensor(np.asarray(a), dtype=F64, device=DEV)  # noqa: E731
        self.m = f(prm["mass"])[self.typ][:, None]
        self.eps, self.sig, self.rc = f(prm["eps"]), f(prm["sigma"]), f(prm["rcut"])
        self.sys = torch.repeat_interleave(torch.arange(len(self.counts), device=DEV), torch.tensor(self.counts, device=DEV))
        first = torch.tensor(np.cumsum([0] + list(self.counts))[:-1], device=DEV)
        self.pid = torch.arange(self.n, device=DEV) - first[self.sys]
        self.replica = torch.tensor([p.get("replica", 0) for p in self.prms], device=DEV)[self.sys]
        self.parts = _parts(self.surfaces, self.counts, self.con)
        boxes = [(tuple(_lengths(p)), tuple(p["periodic"]), tuple(p["box_lo"])) for p in self.prms]
        self.same = [(b, [k for k, q in enumerate(boxes) if q == b]) for b in dict.fromkeys(boxes)]
        self.L = _lengths(prm)
        self.bpm = prm.get("beads_per_mol", 0)
        self.reach = float(self.rc.max()) + 0.4

    def pairs(self):
        """Candidate pairs within the largest cutoff + 0.4 (a particle moves far less than 0.2 between calls)."""
        found = []
        for (L, per, lo), which in self.same:
            at = (self.sys[:, None] == torch.tensor(which, device=DEV)).any(1).nonzero()[:, 0] if len(self.same) > 1 else None
            x = self.x if at is None else self.x[at]
            y = x.clone()
            for d in range(3):
                if per[d]:
                    y[:, d] = lo[d] + torch.remainder(y[:, d] - lo[d], L[d])
            a, b = _close_pairs(y, self.sys if at is None else self.sys[at], self.reach, lo, L, per)
            if at is not None:
                a, b = at[a], at[b]
            if self.prm.get("exclude_intramol"):
                keep = (self.sys[a] != self.sys[b]) | (self.pid[a] // self.bpm != self.pid[b] // self.bpm)
                a, b = a[keep], b[keep]
            found.append((a, b, L, per))
        self.list = found

    def forces(self):
        f, u = torch.zeros_like(self.x), torch.zeros(self.n, dtype=F64, device=DEV)
        for a, b, L, per in self.list:
            d = _images(self.x[a] - self.x[b], L, per)
            r2 = (d * d).sum(1)
            rc = self.rc[self.typ[a], self.typ[b]]
            near = r2 < rc * rc
            a, b, d, r2, rc = a[near], b[near], d[near], r2[near], rc[near]
            e, s = self.eps[self.typ[a], self.typ[b]], self.sig[self.typ[a], self.typ[b]]
            q, qc = (s * s / r2) ** 3, (s / rc) ** 6
            fr, v = 24 * e * q * (2 * q - 1) / r2, 4 * e * (q * q - q) - 4 * e * (qc * qc - qc)
            if self.prm.get("pair_form"):
                slope, r = -24 * e * (2 * qc * qc - qc) / rc, torch.sqrt(r2)
                fr, v = fr + slope / r, v - (r - rc) * slope
            f.index_add_(0, a, fr[:, None] * d)
            f.index_add_(0, b, -fr[:, None] * d)
            u.index_add_(0, a, 0.5 * v)
            u.index_add_(0, b, 0.5 * v)
        prm = self.prm
        if self.bpm > 1:
            c, g = self.x.view(-1, self.bpm, 3), f.view(-1, self.bpm, 3)
            d = c[:, :-1] - c[:, 1:]
            r = d.norm(dim=2, keepdim=True)
            t = self.typ.view(-1, self.bpm)
            r0 = D0 * self.sig[t[:, :-1], t[:, 1:]][:, :, None] / 2 if prm.get("bond_r0_mix") else prm["bond_r0"]
            fb = -2 * prm["bond_k"] * (r - r0) / r * d
            g[:, :-1] += fb
            g[:, 1:] -= fb
            if prm.get("angle_k"):
                p, w = c[:, :-2] - c[:, 1:-1], c[:, 2:] - c[:, 1:-1]
                C = torch.linalg.cross(p, w)
                s, q = C.norm(dim=2, keepdim=True), (p * w).sum(2, keepdim=True)
                th0 = prm["angle_theta0"]
                off = torch.atan2(s * math.cos(th0) - q * math.sin(th0), q * math.cos(th0) + s * math.sin(th0))
                k = torch.where(s > 0, -2 * prm["angle_k"] * off / s, torch.zeros_like(s))
                fa = k * torch.linalg.cross(p, C) / (p * p).sum(2, keepdim=True)
                fc = k * torch.linalg.cross(C, w) / (w * w).sum(2, keepdim=True)
                g[:, :-2] += fa
                g[:, 2:] += fc
                g[:, 1:-1] -= fa + fc
        if prm.get("wall_enable"):
            free = (self.con == 0)[:, None]
            if prm.get("wall_kind"):
                r = self.x.norm(dim=1, keepdim=True)
                walls = [(r - prm["wall_radius"], self.x / r)]
            else:
                z = self.x[:, 2:]
                up = torch.tensor([[0.0, 0.0, 1.0]], dtype=F64, device=DEV)
                walls = [(z - prm["wall_lo_z"], up), (prm["wall_hi_z"] - z, -up)]
            for h, n in walls:
                q = (prm["wall_sigma"] / h) ** 6
                push = 24 * prm["wall_eps"] * (2 * q * q - q) / h
                f += torch.where(free & (h < D0 * prm["wall_sigma"]), push, torch.zeros_like(push)) * n
        if self.surfaces[0]["kind"] == "xy2d":
            f[:, 2] = 0.0
        return f, u

    def noise(self, k):
        prm = self.prm
        if not prm["gamma"] * prm["kT"]:
            return torch.zeros_like(self.x)
        r = _normals(prm["seed"], self.replica, self.pid, k) * torch.sqrt(2 * self.m * prm["kT"] * prm["gamma"] / prm["dt"])
        if self.surfaces[0]["kind"] == "xy2d":
            r[:, 2] = 0.0
        return r

    def combined(self, p, k, first):
        f, u = self.forces()
        prm = self.prm
        if first:
            return f - prm["gamma"] * p + self.noise(k), u
        return (f - prm["gamma"] * p + 0.5 * (self.noise(k) + self.noise(k - 1))) / (1 + 0.5 * prm["gamma"] * prm["dt"]), u

    def steps(self, p, k, count, first):
        """count steps from (x^k, p): Algorithm S1 in multiplier form; then v and the energies at the last step."""
        dt = self.prm["dt"]
        for s in range(count):
            if s % 10 == 0:
                self.pairs()
            F, _ = self.combined(p, k, first)
            q = p + (0.5 * dt if first else dt) * F
            y = self.x + dt / self.m * q
            for kind, sp, at in self.parts:
                held = _piece([float(w) for w in sp], self.x[at], self.L) if kind == "thylakoid" else None
                _, n0 = _g(kind, sp, self.x[at], self.L, held)
                mu = torch.zeros(at.numel(), dtype=F64, device=DEV)
                ya = y[at]
                for _ in range(8):
                    g, n1 = _g(kind, sp, ya - mu[:, None] * n0, self.L, held)
                    mu += g / (n1 * n0).sum(1)
                y[at] = ya - mu[:, None] * n0
                q[at] -= self.m[at] / dt * mu[:, None] * n0
            self.x, p, k, first = y, q, k + 1, False
        self.pairs()
        F, u = self.combined(p, k, first)
        return _project(self.surfaces, self.counts, self.x, (p + 0.5 * dt * F) / self.m, self.con, self.L), u


def exact(case, seed):
    e = _Exact(case, seed)
    v0 = _project(e.surfaces, e.counts, e.x, e.v, e.con, e.L)
    host = case["io"] == "host"
    v, u = e.steps(e.m * v0, HOST_STEP if host else 0, case["steps"], not host)
    out = {"x": e.x, "v": v}
    if host:
        out["step"] = None
    if case["model"] == "nve" and case["precision"] == "fp64":
        K = torch.zeros(4, dtype=F64, device=DEV).index_add_(0, e.sys, 0.5 * (e.m * v * v).sum(1))
        U = torch.zeros(4, dtype=F64, device=DEV).index_add_(0, e.sys, u)
        out["energy"] = torch.stack([K, U], 1)
    return out
