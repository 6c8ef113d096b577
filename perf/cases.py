"""Workloads of the short-range force path that its speed is measured on.

Each case is one unit of work as a simulation code asks for it through the
public entry points of ``paper_1211_4864_gb300``: a force step (binning,
lists, force, kick, moments), the deterministic force with the potential, a
gradient of the force or of a short trajectory, a batch of independent
sub-volumes replayed as one CUDA graph, split-operator sub-cycles, the tree
list builder, or the binning and lists alone.  All have the particle loading of
the standard workloads (one particle per grid cell cubed on average), r_c = 3,
eps = 0.01 and chaining-mesh cells of at least r_c.

Particles: "uniform" (independent positions), "lattice" (a unit lattice with
Gaussian displacements of rms 0.5, as cosmological initial conditions) and
"clustered" (60 % uniform, 40 % in NFW halos of log-uniform mass, as an evolved
density field).  Masses: equal, as in HACC's own runs, or "varied".
"""

import math

import numpy as np
import torch

import paper_1211_4864_gb300 as hs

RCUT, EPS, DT = 3.0, 0.01, 0.01
# poly[5] of the default grid-force fit at r_c = 3, eps = 0.01 (float32 values)
COEFFS = (0.3096082806587219, -0.10157718509435654, 0.018662139773368835, -0.0020956508815288544,
          0.00013053168368060142, -3.366024202478002e-06)
DEV = "cuda"
HALO_MASS_RATIO = 50050.0 / 14462.0  # E[M^2] / E[M]^2 of the log-uniform halo masses 1e2..1e5
EXACT_PAIRS = 3.0e10  # exact() evaluates about 1.5e9 pairs a second


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------

def case(kind, dist, n, L, halos=0, masses="equal", split=32, sym=True, **more):
    c = {"kind": kind, "dist": dist, "n": int(n), "L": float(L), "halos": int(halos), "masses": masses,
         "split": int(split), "sym": bool(sym)}
    c.update(more)
    return c


def listed():
    out = []

    def add(name, *a, **k):
        c = case(*a, **k)
        c["name"] = name
        out.append(c)

    # the smallest call: one step of a 4096-particle box, as in a unit-sized sub-domain
    add("step_uniform_4k", "step", "uniform", 4096, 16.0)
    # a step on near-uniform initial conditions: cells of about 28 particles, few pairs inside the cutoff
    add("step_lattice_2m", "step", "lattice", 128 ** 3, 128.0)
    # the flagship: a step on an evolved, strongly clustered field, very uneven lists
    add("step_clustered_16m", "step", "clustered", 256 ** 3, 256.0, halos=2000, split=128)
    # the same field at an ordinary, odd size with particles of different masses (the general-mass kernels)
    add("step_masses_1m", "step", "clustered", 1030301, 101.5, halos=123, masses="varied", split=64)
    # the bitwise reproducible force with the potential energy, as an energy check or a regression run asks for
    add("gather_uniform_300k", "gather", "uniform", 300007, 67.0)
    # four kick-drift steps and their gradient in positions and velocities (reproducible kernels)
    add("traj_clustered_262k", "traj", "clustered", 64 ** 3, 64.0, halos=100, sym=False, steps=4)
    # one force and its gradient in positions and masses, each pair evaluated once
    add("grad_masses_500k", "grad", "clustered", 500009, 79.37, halos=60, masses="varied", split=64)
    # one force and its gradient in positions on near-uniform particles, each pair evaluated once
    add("grad_lattice_2m", "grad", "lattice", 128 ** 3, 128.0)
    # many independent sub-volumes of different sizes in one captured graph
    add("batch_32_volumes", "batch", "mixed", 32, 0.0, split=128, lo=4096, hi=262144)
    # split-operator sub-cycles between two long-range kicks
    add("sks_lattice_262k", "sks", "lattice", 64 ** 3, 64.0, cycles=5)
    # the RCB tree as the list builder
    add("tree_clustered_262k", "tree", "clustered", 64 ** 3, 64.0, halos=31, split=64)
    # binning and lists alone (every integer result), as a code that only needs cell order or pair counts
    add("bin_clustered_4m", "bin", "clustered", 4000037, 158.74, halos=477, split=64)
    return out


def draw(rng):
    """One more case of the listed ranges: any kind, 1.5k to 2M particles (log-uniform, any parity)."""
    kind = rng.choice(["step", "step", "gather", "traj", "grad", "batch", "sks", "tree", "bin"])
    if kind == "batch":
        lo = int(math.exp(rng.uniform(math.log(1500), math.log(10000))))
        return case("batch", "mixed", rng.randint(2, 96), 0.0, split=rng.choice([32, 64, 128]),
                    sym=rng.random() < 0.7, lo=lo, hi=int(lo * math.exp(rng.uniform(0.5, 2.5))))
    top = {"traj": 3.0e5, "tree": 5.0e5, "sks": 1.0e6, "grad": 1.0e6}.get(kind, 2.2e6)
    n = int(math.exp(rng.uniform(math.log(1500), math.log(top))))
    dist = rng.choice(["uniform", "lattice", "clustered", "clustered"])
    halos = 0
    if dist == "lattice":
        n = int(round(n ** (1.0 / 3.0))) ** 3
    L = round(n ** (1.0 / 3.0), 2)
    if dist == "clustered":
        halos = max(1, round(n * rng.uniform(0.8, 3.0) * 2000.0 / 256 ** 3))
    c = case(kind, dist, n, L, halos, masses=rng.choice(["equal", "equal", "varied"]),
             split=rng.choice([32, 64, 128]), sym=rng.random() < 0.6)
    if kind == "traj":
        c["steps"] = rng.randint(1, 4)
    if kind == "sks":
        c["cycles"] = rng.randint(2, 6)
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _uniform(g, n, L):
    return torch.rand((n, 3), generator=g, device=DEV, dtype=torch.float64) * L


def _nfw(g, counts):
    """Offsets from their halo's centre of the particles of all halos (NFW radii by bisection, isotropic)."""
    n, h = int(counts.sum()), counts.shape[0]
    k = torch.tensor(counts, device=DEV)
    conc = 5.0 + 5.0 * torch.rand(h, generator=g, device=DEV, dtype=torch.float64)
    r200 = (3.0 * k.double() / (800.0 * math.pi)) ** (1.0 / 3.0)
    c = torch.repeat_interleave(conc, k)
    rs = torch.repeat_interleave(r200 / conc, k)
    mu = lambda x: torch.log1p(x) - x / (1.0 + x)  # noqa: E731
    u = torch.rand(n, generator=g, device=DEV, dtype=torch.float64) * mu(c)
    lo, hi = torch.zeros_like(u), c.clone()
    for _ in range(40):
        mid = 0.5 * (lo + hi)
        below = mu(mid) < u
        lo, hi = torch.where(below, mid, lo), torch.where(below, hi, mid)
    r = 0.5 * (lo + hi) * rs
    cz = 2.0 * torch.rand(n, generator=g, device=DEV, dtype=torch.float64) - 1.0
    phi = 2.0 * math.pi * torch.rand(n, generator=g, device=DEV, dtype=torch.float64)
    sz = torch.sqrt((1.0 - cz * cz).clamp(min=0.0))
    return torch.stack([r * sz * torch.cos(phi), r * sz * torch.sin(phi), r * cz], dim=1)


def _clustered(g, rng, n, L, halos):
    budget = int(round(0.4 * n))
    raw = np.exp(rng.uniform(math.log(1e2), math.log(1e5), halos))
    counts = np.floor(raw * (budget / raw.sum())).astype(np.int64)
    counts[np.argsort(-raw)[:1]] += budget - int(counts.sum())
    centres = torch.repeat_interleave(_uniform(g, halos, L), torch.tensor(counts, device=DEV), dim=0)
    return torch.cat([_uniform(g, n - budget, L), centres + _nfw(g, counts)])


def _positions(g, rng, dist, n, L, halos):
    """float32 [3, n] in [0, L), generation order (background first, halo by halo)."""
    L32 = float(np.float32(L))
    if dist == "uniform":
        p = _uniform(g, n, L32)
    elif dist == "lattice":
        side = round(n ** (1.0 / 3.0))
        a = (torch.arange(side, device=DEV, dtype=torch.float64) + 0.5) * (L32 / side)
        z, y, x = torch.meshgrid(a, a, a, indexing="ij")
        p = torch.stack([x.reshape(-1), y.reshape(-1), z.reshape(-1)], dim=1)
        p = p + 0.5 * torch.randn(p.shape, generator=g, device=DEV, dtype=torch.float64)
    else:
        p = _clustered(g, rng, n, L32, halos)
    p = torch.remainder(p, L32).float()
    p[p >= L32] = 0.0
    return p.t().contiguous()


def _volumes(case):
    """Particle counts and box sides of a batch: log-uniform counts, density one."""
    rng = np.random.default_rng(case["n"] * 1000003 + case["lo"])
    counts = np.rint(np.exp(rng.uniform(math.log(case["lo"]), math.log(case["hi"]), case["n"]))).astype(np.int64)
    return counts, np.array([float(c) ** (1.0 / 3.0) for c in counts], np.float32)


def _inputs(case, seed):
    """pos, v float32 [3, N], m float32 [N], box sides, volume offsets; from the seed alone."""
    g = torch.Generator(device=DEV).manual_seed(1 + int(seed))
    rng = np.random.default_rng(1 + int(seed))
    if case["kind"] == "batch":
        counts, L = _volumes(case)
        parts = []
        for b, c in enumerate(counts):
            halos = max(1, int(round(2000.0 * c / 256 ** 3)))
            dist = "uniform" if 2 * b < len(counts) else "clustered"
            parts.append(_positions(g, rng, dist, int(c), float(L[b]), halos))
        pos = torch.cat(parts, dim=1).contiguous()
        off = np.concatenate([[0], np.cumsum(counts)]).astype(np.int64)
    else:
        pos = _positions(g, rng, case["dist"], case["n"], case["L"], case["halos"])
        L = np.array([case["L"]], np.float32)
        off = np.array([0, case["n"]], np.int64)
    n = pos.shape[1]
    v = 0.1 * torch.randn((3, n), generator=g, device=DEV)
    if case["masses"] == "varied":
        m = torch.exp(0.7 * torch.randn(n, generator=g, device=DEV))
    else:
        m = torch.ones(n, device=DEV)
    # cotangents of a loss (gradient cases)
    lam = torch.randn((3, n), generator=g, device=DEV)
    return pos, v, m, lam, L, off


def _params():
    return hs.SRParams(EPS, RCUT, np.array(COEFFS, np.float32))


def prepare(case, seed):
    pos, v, m, lam, L, off = _inputs(case, seed)
    kw = {"builder": "rcb", "leaf_max": 64} if case["kind"] == "tree" else {}
    sr = hs.ShortRange(L, off, RCUT, split_T=case["split"], **kw)
    s = {"case": case, "sr": sr, "prm": _params(), "pos": pos, "v": v, "m": m, "a": torch.empty_like(pos)}
    kind = case["kind"]
    if kind in ("grad", "traj"):
        s["lam"] = lam
        s["pos"] = pos.requires_grad_(True)
        if kind == "traj":
            s["v"] = v.requires_grad_(True)
        elif case["masses"] == "varied":
            s["m"] = m.requires_grad_(True)
    if kind == "batch":
        # warmed up and captured on copies of the velocities, which the replayed kick updates in place
        keep = v.clone()
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            s["mom"] = _step(s)
        torch.cuda.current_stream().wait_stream(side)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            s["mom"] = _step(s)
        v.copy_(keep)
        s["graph"] = graph
    return s


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

def _step(s):
    """Binning, lists, force, kick and the float64 moments."""
    sr = s["sr"]
    sr.prepare(s["pos"], s["m"])
    force = sr.force_symmetric if s["case"]["sym"] else sr.force
    force(s["prm"], s["a"])
    sr.kick(s["v"], s["a"], DT)
    return sr.moments(s["m"], s["v"], s["a"])


def _nearest(d, L):
    """Displacements to the nearest image (the sub-cycles wrap positions into the box)."""
    return d - L * torch.round(d / L)


def run(s):
    case, sr, prm = s["case"], s["sr"], s["prm"]
    kind = case["kind"]
    if kind == "step":
        mom = _step(s)
        return {"a": s["a"], "v": s["v"], "moments": mom, "pairs": sr.n_pairs}
    if kind == "batch":
        s["graph"].replay()
        return {"a": s["a"], "v": s["v"], "moments": s["mom"], "pairs": sr.n_pairs}
    if kind == "gather":
        sr.prepare(s["pos"], s["m"])
        a = sr.force(prm, s["a"])
        phi = sr.potential(prm)
        return {"a": a, "phi": phi, "moments": sr.moments(s["m"], s["v"], a, phi)}
    if kind == "grad":
        a = hs.sr_force_autograd(s["pos"], s["m"], sr, prm, symmetric=case["sym"])
        wrt = [s["pos"], s["m"]] if s["m"].requires_grad else [s["pos"]]
        return {"a": a.detach(), "grads": torch.autograd.grad(a, wrt, s["lam"])}
    if kind == "traj":
        disp, v = hs.trajectory_autograd(s["pos"], s["v"], s["m"], sr, prm, DT, case["steps"],
                                         symmetric=case["sym"])
        grads = torch.autograd.grad([disp, v], [s["pos"], s["v"]], [s["lam"], 0.1 * s["lam"]])
        return {"disp": disp.detach(), "v": v.detach(), "grads": grads}
    if kind == "sks":
        pos, v = s["pos"].clone(), s["v"].clone()  # the long-range step keeps the state it started from
        a = sr.sks_subcycles(pos, v, s["m"], prm, DT, case["cycles"], s["a"])
        return {"moved": _nearest(pos - s["pos"], case["L"]), "v": v, "a": a}
    if kind == "tree":
        sr.prepare(s["pos"], s["m"])
        force = sr.force_symmetric if case["sym"] else sr.force
        return {"a": force(prm, s["a"]), "perm": sr.perm, "pairs": sr.n_pairs}
    sr.prepare(s["pos"], s["m"])  # "bin"
    return {"cell": sr.cell_of, "start": sr.cell_start, "perm": sr.perm, "records": sr.sorted4,
            "entries": sr.nbr_cell, "images": sr.nbr_shift, "pairs": sr.n_pairs, "tasks": sr.n_tasks}


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

def _near(n, L, dist, halos):
    """About how many partners a particle has inside the cutoff."""
    ball = 4.0 / 3.0 * math.pi * RCUT ** 3
    rho = n / float(L) ** 3
    if dist != "clustered":
        return ball * rho
    own = 0.4 * 0.95 * HALO_MASS_RATIO * 0.4 * n / halos if halos > 1 else 0.4 * 0.95 * 0.4 * n
    return min(float(n), 0.6 * ball * rho + own)


def _pairs(case):
    """(particles, unordered pairs inside the cutoff) of one force evaluation, estimated from the recipe."""
    if case["kind"] != "batch":
        n = case["n"]
        return n, 0.5 * n * _near(n, case["L"], case["dist"], case["halos"])
    counts, L = _volumes(case)
    total = 0.0
    for b, c in enumerate(counts):
        dist = "uniform" if 2 * b < len(counts) else "clustered"
        total += 0.5 * c * _near(int(c), L[b], dist, max(1, int(round(2000.0 * c / 256 ** 3))))
    return int(counts.sum()), float(total)


def work(case):
    n, pairs = _pairs(case)
    kind = case["kind"]
    force = 34.0 * pairs  # each pair once: 22 for the term, 12 to add it to both particles
    adjoint = 60.0 * pairs
    inputs = 16.0 * n  # x, y, z, m
    if kind in ("step", "batch"):
        return {"bytes": inputs + (12 + 24) * n, "flops": force + 6.0 * n}
    if kind == "gather":
        return {"bytes": inputs + (12 + 12 + 4) * n, "flops": force + 22.0 * pairs}
    if kind == "grad":
        return {"bytes": inputs + (12 + 12 + 12) * n, "flops": force + adjoint}
    if kind == "traj":
        return {"bytes": inputs + (12 + 24 + 24 + 24) * n, "flops": case["steps"] * (2 * force + adjoint)}
    if kind == "sks":
        return {"bytes": inputs + (12 + 24 + 12) * n, "flops": case["cycles"] * force}
    if kind == "tree":
        return {"bytes": inputs + 16.0 * n, "flops": force}
    cells = max(3.0, math.floor(case["L"] / RCUT)) ** 3
    return {"bytes": inputs + 24.0 * n + cells * (4 + 27 * 5), "flops": 12.0 * n}


# ---------------------------------------------------------------------------
# tolerances
# ---------------------------------------------------------------------------

def tolerance(case):
    """About four times the largest error against exact() seen over the listed and forty drawn cases: float32 pair
    terms and sums leave 2e-7 to 3e-7 of the forces (2-norm), the potential (a difference of nearly equal terms)
    9e-7, the force gradient 2e-6, whose single values reach 9e-4 where close pairs nearly cancel.  Trajectories and
    sub-cycles amplify the float32 offsets and positions of close pairs from step to step, and the displacements over
    a few sub-cycles keep about 1e-3 of the positions' float32 storage."""
    kind = case["kind"]
    if kind == "bin":
        return "exact"
    if kind == "traj":
        return {"rel": 1.4e-4, "max": 4e-2}
    if kind == "sks":
        return {"rel": 2e-3, "max": 0.15}
    if kind == "grad":
        return {"rel": 8e-6, "max": 4e-3}
    if kind == "gather":
        return {"rel": 4e-6, "max": 5e-5}
    return {"rel": 1.2e-6, "max": 5e-5}


# ---------------------------------------------------------------------------
# the same in 64 bits, in plain torch
# ---------------------------------------------------------------------------

def _pair_lists(pos, L):
    """Chunks (i, j, d) of all ordered pairs of neighbouring cells (side at least r_c) of one periodic box."""
    n = pos.shape[1]
    nc = max(1, int(L / RCUT))
    w = L / nc
    x = pos - L * torch.floor(pos / L)
    c3 = (x / w).long().clamp(0, nc - 1)
    cell = (c3[2] * nc + c3[1]) * nc + c3[0]
    order = torch.argsort(cell)
    start = torch.searchsorted(cell[order], torch.arange(nc ** 3 + 1, device=pos.device))
    xs, cs = x[:, order], c3[:, order]
    seen = set()
    for dz in (-1, 0, 1):
        for dy in (-1, 0, 1):
            for dx in (-1, 0, 1):
                t = (dx % nc, dy % nc, dz % nc)
                if t in seen:  # fewer than three cells a side: each neighbour once
                    continue
                seen.add(t)
                nb = (((cs[2] + dz) % nc) * nc + (cs[1] + dy) % nc) * nc + (cs[0] + dx) % nc
                cnt = start[nb + 1] - start[nb]
                cum = torch.cumsum(cnt, 0)
                total, lo = int(cum[-1]), 0
                while lo < n:
                    base = int(cum[lo - 1]) if lo else 0
                    if base >= total:
                        break
                    hi = max(lo + 1, int(torch.searchsorted(cum, base + (1 << 25))))
                    hi = min(hi, n)
                    k = cnt[lo:hi]
                    i = torch.repeat_interleave(torch.arange(lo, hi, device=pos.device), k)
                    at = torch.arange(i.shape[0], device=pos.device) - (cum[i] - cnt[i] - base)
                    j = start[nb[i]] + at
                    d = xs[:, j] - xs[:, i]
                    d -= L * torch.round(d / L)
                    s = (d * d).sum(0)
                    keep = (s < RCUT * RCUT) & (i != j)
                    yield order[i[keep]], order[j[keep]], d[:, keep], s[keep]
                    lo = hi


def _poly(c, s):
    r = torch.zeros_like(s)
    for a in reversed(c):
        r = r * s + a
    return r


def _law(s):
    c = [float(np.float32(v)) for v in COEFFS]
    e = float(np.float32(EPS))
    return (s + e) ** -1.5 - _poly(c, s)


def _law_slope(s):
    c = [float(np.float32(v)) for v in COEFFS]
    e = float(np.float32(EPS))
    return -1.5 * (s + e) ** -2.5 - _poly([k * c[k] for k in range(1, 6)], s)


def _law_potential(s):
    c = [float(np.float32(v)) for v in COEFFS]
    e = float(np.float32(EPS))
    P = lambda t: t * _poly([c[k] / (k + 1) for k in range(6)], t)  # noqa: E731
    rc2 = torch.full((), RCUT * RCUT, dtype=torch.float64, device=s.device)
    return (rc2 + e) ** -0.5 - (s + e) ** -0.5 + 0.5 * (P(rc2) - P(s))


def _force64(pos, m, L, potential=False):
    a = torch.zeros_like(pos)
    phi = torch.zeros_like(m)
    for i, j, d, s in _pair_lists(pos, L):
        f = _law(s) * m[j]
        for k in range(3):
            a[k].index_add_(0, i, f * d[k])
        if potential:
            phi.index_add_(0, i, m[j] * _law_potential(s))
    return (a, phi) if potential else a


def _adjoint64(pos, m, lam, L, mass=False):
    g = torch.zeros_like(pos)
    gm = torch.zeros_like(m)
    for i, j, d, s in _pair_lists(pos, L):
        f = _law(s)
        mu = m[i] * lam[:, j] - m[j] * lam[:, i]
        r = 2.0 * _law_slope(s) * (d * mu).sum(0)
        for k in range(3):
            g[k].index_add_(0, i, f * mu[k] + r * d[k])
        if mass:
            gm.index_add_(0, i, -f * (d * lam[:, j]).sum(0))
    return g, gm


def _moments64(m, v, a, phi=None):
    out = torch.zeros(9, dtype=torch.float64, device=m.device)
    out[0:3] = (m * v).sum(1)
    out[3:6] = (m * a).sum(1)
    out[6] = 0.5 * (m * (v * v).sum(0)).sum()
    out[7] = (m * a.square().sum(0).sqrt()).sum()
    if phi is not None:
        out[8] = 0.5 * (m * phi).sum()
    return out


def _candidates(case):
    """About how many ordered pairs one force evaluation of exact() visits."""
    n, pairs = _pairs(case)
    return 2.0 * pairs / (0.8 if case["dist"] == "clustered" else 0.155) + 730.0 * n


def exact(case, seed):
    kind = case["kind"]
    rounds = {"traj": 2 * case.get("steps", 1), "sks": case.get("cycles", 1), "grad": 2}.get(kind, 1)
    if kind == "bin" or rounds * _candidates(case) > EXACT_PAIRS:
        return None
    pos, v, m, lam, L, off = _inputs(case, seed)
    pos, v, m, lam = pos.double(), v.double(), m.double(), lam.double()
    L0 = float(L[0])
    if kind in ("step", "batch"):
        a = torch.cat([_force64(pos[:, b:e], m[b:e], float(Lv)) for Lv, b, e in zip(L, off[:-1], off[1:])], dim=1)
        v = v + float(np.float32(DT)) * a
        return {"a": a, "v": v, "moments": _moments64(m, v, a), "pairs": None}
    if kind == "gather":
        a, phi = _force64(pos, m, L0, potential=True)
        return {"a": a, "phi": phi, "moments": _moments64(m, v, a, phi)}
    if kind == "grad":
        g, gm = _adjoint64(pos, m, lam, L0, mass=case["masses"] == "varied")
        return {"a": _force64(pos, m, L0), "grads": (g, gm) if case["masses"] == "varied" else (g,)}
    if kind == "traj":
        h = float(np.float32(DT))
        disp, at = torch.zeros_like(pos), []
        for _ in range(case["steps"]):
            at.append(pos + disp)
            v = v + h * _force64(at[-1], m, L0)
            disp = disp + h * v
        gx, gd, gv = torch.zeros_like(pos), lam.clone(), 0.1 * lam
        for x in reversed(at):
            gv = gv + h * gd
            g, _ = _adjoint64(x, m, h * gv, L0)
            gd = gd + g
            gx = gx + g
        return {"disp": disp, "v": v, "grads": (gx, gv)}
    if kind == "sks":
        h, pos0 = float(np.float32(DT)), pos.clone()
        for _ in range(case["cycles"]):
            pos = pos + 0.5 * h * v
            a = _force64(pos, m, L0)
            v = v + h * a
            pos = pos + 0.5 * h * v
        return {"moved": pos - pos0, "v": v, "a": a}
    return {"a": _force64(pos, m, L0), "perm": None, "pairs": None}  # "tree"
