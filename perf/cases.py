"""Performance cases: the calls a user of this library makes, over the sizes and options in earnest use.

``listed()`` names the cases, ``draw(rng)`` gives another one of the same ranges, ``prepare(case, seed)`` makes what a
program has in hand before the call, ``run(state)`` is one pass through the public entry points with all of its outputs,
``work(case)`` counts what the pass cannot do without, and ``exact(case, seed)`` evaluates the floating outputs in 64
bits with plain torch (brute-force hulls and a search over all template correspondences, no code of the library).

A case is a dict of plain values:

  path      frame (device tensors, one call), host (numpy arrays, one call), batch (many device frames, one pass),
            server (many host frames through the serving queue)
  system    crystal, poly (grains), mixed (four lattices and a disordered slab), particle (free surface, no periodic
            side), film (free surface in z), drift (a crystal in unwrapped coordinates)
  n         atoms of the frame (of the largest frame where there are several); n_min, frames: the others' range
  lattice, sigma, dtype, species, mask, rmsd_max, ordering, derived, capture: the options of the call
"""
from __future__ import annotations

import functools
import itertools
import math

import numpy as np
import torch

from paper_1603_05143_gb300 import PTM, Server
from paper_1603_05143_gb300.inputs import A_BCC_FE, A_FCC_CU, A_HCP, A_L12, A_SC, unit_cell

DEVICE = "cuda" if torch.cuda.is_available() else "cpu"
LATTICE = {"fcc": A_FCC_CU, "hcp": A_HCP, "bcc": A_BCC_FE, "sc": A_SC, "l10": A_L12, "l12": A_L12, "b2": A_BCC_FE}
OUTPUTS = ("structure", "alloy", "rmsd", "scale", "quat", "strain", "correspondence")
DERIVED = ("von_mises", "rodrigues")
DISORDERED_DENSITY = 0.0565          # atoms per cubic Angstrom, the liquid slab of the mixed-phase configuration
ALL, FCC_HCP_BCC = 31, 2 | 4 | 16
DEFAULTS = {"path": "frame", "system": "crystal", "n": 4000, "lattice": "fcc", "sigma": 0.10, "dtype": "float32",
            "species": False, "mask": ALL, "rmsd_max": 0.0, "ordering": "euclidean", "derived": False, "frames": 1,
            "n_min": 0, "capture": False}


def listed():
    c = lambda name, **kw: dict(DEFAULTS, name=name, **kw)  # noqa: E731
    return [
        # an interactive call on a unit test or a viewer's selection: latency and launches
        c("frame_tiny_256", lattice="l12", n=256, species=True, sigma=0.08),
        # the paper's introductory crystal, double precision as an MD code hands it over
        c("frame_fcc_4000_f64", n=4000, dtype="float64"),
        # an analysis step with every derived output, a cut-off and the RMSD histogram that chooses it
        c("frame_b2_53k_derived", lattice="b2", n=53240, species=True, sigma=0.12, mask=FCC_HCP_BCC, rmsd_max=0.15,
          derived=True),
        # a hot polycrystal, the million-atom production frame
        c("frame_poly_1m", system="poly", n=1 << 20, sigma=0.15),
        # phase coexistence near melting, an alloy frame of the largest size
        c("frame_mixed_4m", system="mixed", n=1 << 22, sigma=0.20, species=True),
        # topological neighbour order, for hot crystals
        c("frame_topo_262k", system="poly", n=262147, sigma=0.15, ordering="topological"),
        # a trajectory written in unwrapped coordinates, strained cell
        c("frame_drift_200k", system="drift", lattice="hcp", n=202500, sigma=0.08),
        # a free nanoparticle: no periodic side, vacuum around it
        c("frame_particle_131k", system="particle", n=131071, sigma=0.10),
        # a simulation's frame held in host memory, double precision
        c("host_bcc_250k_f64", path="host", lattice="bcc", n=250000, sigma=0.12, dtype="float64"),
        # a parameter scan of small cells, replayed as one graph
        c("batch_48_small", path="batch", frames=48, n_min=500, n=16000, sigma=0.15, species=True, capture=True),
        # the large uneven batch of the library's benchmark
        c("batch_256_uneven", path="batch", frames=256, n_min=1000, n=1000000, sigma=0.25, species=True, capture=True),
        # frames arriving from a running simulation, through the serving queue
        c("server_40", path="server", system="crystal", frames=40, n_min=4000, n=262144, sigma=0.2, species=True),
    ]


def draw(rng):
    def log_n(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    c = dict(DEFAULTS)
    c["sigma"] = rng.choice([0.0, round(rng.uniform(0.02, 0.25), 3), round(rng.uniform(0.02, 0.25), 3)])
    c["species"] = rng.random() < 0.5
    c["lattice"] = rng.choice(sorted(LATTICE))
    kind = rng.choice(["frame", "frame", "poly", "mixed", "topo", "drift", "particle", "film", "host", "batch", "server"])
    if kind == "frame":
        c.update(n=log_n(200, 1500000), dtype=rng.choice(["float32", "float32", "float64"]), derived=rng.random() < 0.3,
                 mask=rng.choice([ALL, ALL, FCC_HCP_BCC]), rmsd_max=rng.choice([0.0, 0.0, 0.12]))
    elif kind == "poly":
        c.update(system="poly", n=log_n(20000, 2000000), sigma=round(rng.uniform(0.05, 0.2), 3))
    elif kind == "mixed":
        c.update(system="mixed", n=log_n(30000, 3000000), sigma=round(rng.uniform(0.05, 0.25), 3), species=True)
    elif kind == "topo":
        c.update(ordering="topological", n=log_n(2000, 300000), sigma=round(rng.uniform(0.05, 0.2), 3))
    elif kind in ("drift", "particle", "film"):
        c.update(system=kind, n=log_n(3000, 300000), sigma=round(rng.uniform(0.02, 0.2), 3))
    elif kind == "host":
        c.update(path="host", n=log_n(2000, 500000), dtype=rng.choice(["float32", "float64"]))
    elif kind == "batch":
        c.update(path="batch", frames=rng.randrange(3, 120), n_min=500, n=log_n(2000, 200000), capture=rng.random() < 0.5)
    else:
        c.update(path="server", frames=rng.randrange(4, 60), n_min=1000, n=log_n(4000, 150000))
    return c


# ------------------------------------------------------------------------------------------------------------- inputs
def _rotation(rng):
    q = rng.normal(size=4)
    w, x, y, z = q / np.linalg.norm(q)
    return np.array([[1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y)],
                     [2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x)],
                     [2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)]])


def _t(x):
    return torch.as_tensor(np.ascontiguousarray(x), dtype=torch.float64, device=DEVICE)


def _lattice_points(kind, a, reps, centred=False):
    """Points of reps conventional cells (n x 3), their cell and their species."""
    cell, basis, sp = unit_cell(kind, a)
    g = [torch.arange(r, dtype=torch.float64, device=DEVICE) - (r // 2 if centred else 0) for r in reps]
    grid = torch.stack(torch.meshgrid(*g, indexing="ij"), -1).reshape(-1, 1, 3)
    frac = (grid + _t(basis)[None]).reshape(-1, 3)
    species = torch.as_tensor(sp, device=DEVICE).repeat(int(np.prod(reps)))
    return frac @ _t(cell), cell * np.asarray(reps)[:, None], species


def _reps(kind, n, most=False):
    """About n atoms in a nearly cubic box (at least n with `most`), three cells a side at least."""
    cell, basis, _ = unit_cell(kind, 1.0)
    side = (n / len(basis) * abs(np.linalg.det(cell))) ** (1 / 3)
    reps = [max(3, int(round(side / cell[i, i]))) for i in range(3)]
    while most and np.prod(reps) * len(basis) < n:
        reps[int(np.argmin([reps[i] * cell[i, i] for i in range(3)]))] += 1
    return reps


def _wrap(pos, cell):
    f = pos @ _t(np.linalg.inv(cell))
    f = f - torch.floor(f)
    return torch.where(f >= 1, torch.zeros_like(f), f) @ _t(cell)


def _noise(pos, sigma, gen):
    return pos + sigma * torch.randn(pos.shape, generator=gen, dtype=torch.float64, device=DEVICE) if sigma > 0 else pos


def _crystal(kind, n, sigma, rng, gen, wrap=True, drift=None):
    """A strained, rotated crystal in its periodic (triclinic) cell."""
    pos, cell, sp = _lattice_points(kind, LATTICE[kind], _reps(kind, n))
    E = rng.uniform(-0.05, 0.05, (3, 3))
    lin = (np.eye(3) + 0.5 * (E + E.T)) @ _rotation(rng)
    cell = cell @ lin.T
    pos = _noise(pos @ _t(lin.T), sigma, gen)
    if drift is not None:
        pos = pos + _t(drift @ cell)
    return (_wrap(pos, cell) if wrap else pos), cell, (True, True, True), sp


def _poly(n, sigma, rng, gen, grains=16, faults=4):
    """Voronoi grains of fcc in a cube, four of them with a stacking fault, boundaries thinned, exactly n atoms."""
    a = A_FCC_CU
    L = (n / 4.0) ** (1 / 3) * a
    centres = rng.random((grains, 3)) * L
    m = int(math.ceil(0.5 * math.sqrt(3) * L / a)) + 1
    base, _, _ = _lattice_points("fcc", a, [2 * m + 1] * 3, centred=True)
    base = base[(base * base).sum(1) <= 0.75 * L * L]
    parts = []
    for g in range(grains):
        p = base
        if g < faults:
            up = p.sum(1) / math.sqrt(3) > a / (4 * math.sqrt(3))
            p = torch.where(up[:, None], p + _t(a / 6 * np.array([1.0, 1.0, -2.0])), p)
        off = p @ _t(_rotation(rng).T)
        off = off[(off.abs() < L / 2).all(1)]
        own = (off * off).sum(1)
        keep = torch.ones(len(off), dtype=torch.bool, device=DEVICE)
        for h in range(grains):
            if h != g:
                d = centres[h] - centres[g]
                e = off - _t(d)
                e = e - L * torch.round(e / L)
                # nearer to its own centre, by enough that atoms across a boundary are about 1.5 Angstrom apart
                keep &= (e * e).sum(1) - own > 1.5 * float(np.linalg.norm(d - L * np.round(d / L)))
        parts.append(off[keep] + _t(centres[g]))
    pos = torch.cat(parts)
    if len(pos) > n:
        pos = pos[torch.randperm(len(pos), generator=gen, device=DEVICE)[:n]]
    elif len(pos) < n:
        pos = torch.cat([pos, L * torch.rand((n - len(pos), 3), generator=gen, dtype=torch.float64, device=DEVICE)])
    cell = np.eye(3) * L
    return _wrap(_noise(pos, sigma, gen), cell), cell, (True, True, True), None


def _mixed(n, sigma, rng, gen):
    """Slabs of bcc, fcc, L1_2 (10 % antisites) and sc along x, and a disordered slab with the rest of the n atoms."""
    phases = [("bcc", A_BCC_FE), ("fcc", A_FCC_CU), ("l12", A_L12), ("sc", A_SC)]
    rho = [len(unit_cell(k, a)[1]) / a ** 3 for k, a in phases] + [DISORDERED_DENSITY]
    ly = (n / (0.4 * sum(rho))) ** (1 / 3)
    t = 2 * ly / 5
    parts, species = [], []
    for i, (kind, a0) in enumerate(phases):
        side = max(1, int(round(ly / a0)))
        a = ly / side
        p, _, sp = _lattice_points(kind, a, [int(math.ceil(t / a)), side, side])
        keep = p[:, 0] < t - 1e-6
        p, sp = p[keep], sp[keep]
        if kind == "l12":
            flip = torch.rand(len(sp), generator=gen, device=DEVICE) < 0.10
            sp = torch.where(flip, 1 - sp, sp)
        parts.append(p + _t([i * t, 0.0, 0.0]))
        species.append(sp)
    rest = n - sum(len(p) for p in parts)
    d = (t * ly * ly / rest) ** (1 / 3)
    k = [max(1, int(math.ceil(s / d))) for s in (t, ly, ly)]
    p, _, sp = _lattice_points("sc", 1.0, k)
    p = p[torch.randperm(len(p), generator=gen, device=DEVICE)[:rest]] * _t([t / k[0], ly / k[1], ly / k[2]])
    parts.append(_noise(p, 0.42, gen) + _t([4 * t, 0.0, 0.0]))
    species.append(sp[:rest])
    cell = np.diag([2 * ly, ly, ly])
    return _wrap(_noise(torch.cat(parts), sigma, gen), cell), cell, (True, True, True), torch.cat(species)


def _free(kind, n, sigma, rng, gen, film):
    """The n sites nearest a centre (a particle), or a film of a third of the box's height; vacuum beyond."""
    a = LATTICE[kind]
    if film:
        cell0, basis, _ = unit_cell(kind, a)
        side = (n / len(basis) * abs(np.linalg.det(cell0)) * 3) ** (1 / 3)
        reps = [max(4, int(round(side / cell0[0, 0]))), max(4, int(round(side / cell0[1, 1])))]
        reps.append(max(2, int(round(n / len(basis) / reps[0] / reps[1]))))
        pos, cell, sp = _lattice_points(kind, a, reps)
        cell[2, 2] += 30.0
        pos = _noise(pos, sigma, gen) + _t([0.0, 0.0, 15.0])
        f = pos @ _t(np.linalg.inv(cell))
        f[:, :2] -= torch.floor(f[:, :2])
        return f @ _t(cell), cell, (True, True, False), sp
    pos, _, sp = _lattice_points(kind, a, [2 * r for r in _reps(kind, n, most=True)], centred=True)
    near = torch.argsort((pos * pos).sum(1), stable=True)[:n]
    pos, sp = pos[near], sp[near]
    r = float((pos * pos).sum(1).max().sqrt())
    pos = _noise(pos @ _t(_rotation(rng).T), sigma, gen) + (r + 10.0)
    return pos, np.eye(3) * 2 * (r + 10.0), (False, False, False), sp


def _one(case, seed, n=None, lattice=None, sigma=None):
    """One frame: positions and species on the device, cell, periodicity."""
    rng = np.random.default_rng([17, seed])
    gen = torch.Generator(DEVICE)
    gen.manual_seed(seed)
    n, kind = n or case["n"], lattice or case["lattice"]
    sigma = case["sigma"] if sigma is None else sigma
    system = case["system"]
    if system == "poly":
        f = _poly(n, sigma, rng, gen)
    elif system == "mixed":
        f = _mixed(n, sigma, rng, gen)
    elif system in ("particle", "film"):
        f = _free(kind, n, sigma, rng, gen, system == "film")
    elif system == "drift":
        f = _crystal(kind, n, sigma, rng, gen, wrap=False, drift=rng.uniform(-1.5, 1.5, 3))
    else:
        f = _crystal(kind, n, sigma, rng, gen)
    pos, cell, pbc, sp = f
    dtype = torch.float64 if case["dtype"] == "float64" else torch.float32
    sp = (sp if sp is not None else torch.zeros(len(pos), device=DEVICE)).to(torch.int8) if case["species"] else None
    return {"positions": pos.to(dtype).contiguous(), "cell": cell, "pbc": pbc, "species": sp}


def _sizes(case):
    """Sizes of the frames, spread over the logarithm of [n_min, n]: the same for every seed."""
    if case["frames"] == 1:
        return [case["n"]]
    u = np.random.default_rng([3, case["frames"], case["n"]]).random(case["frames"])
    return [int(round(case["n_min"] * (case["n"] / case["n_min"]) ** x)) for x in u]


def _frames(case, seed):
    if case["frames"] == 1:
        return [_one(case, seed)]
    kinds = ("fcc", "hcp", "bcc", "l10", "l12", "sc")
    out = []
    for i, n in enumerate(_sizes(case)):
        u = np.random.default_rng([11, seed, i]).random()
        # noise up to sigma, and one perfect frame in ten
        out.append(_one(case, 1000 * seed + i, n, kinds[i % len(kinds)], 0.0 if i % 10 == 9 else case["sigma"] * u))
    return out


# ---------------------------------------------------------------------------------------------------------- the calls
@functools.lru_cache(maxsize=None)
def _context():
    return PTM(0)


def _pinned(shape, dtype):
    return torch.empty(shape, dtype=dtype, pin_memory=True).numpy()


def prepare(case, seed):
    case = dict(DEFAULTS, **case)
    frames = _frames(case, seed)
    s = {"case": case, "ptm": _context(), "mask": case["mask"], "rmsd_max": case["rmsd_max"] or math.inf,
         "outputs": OUTPUTS + (DERIVED if case["derived"] else ())}
    if case["path"] == "frame":
        s.update(frames[0])
    elif case["path"] == "batch":
        s["batch"] = s["ptm"].batch(frames, mask=s["mask"], rmsd_max=s["rmsd_max"])
        if case["capture"]:
            st = torch.cuda.Stream()
            s["batch"].run()                        # the first run outside capture, as the benchmark does
            torch.cuda.synchronize()
            s["batch"].capture(st)
    elif case["path"] == "host":
        f = frames[0]
        s.update(f, positions=f["positions"].cpu().numpy(), species=None if f["species"] is None else f["species"].cpu().numpy())
    else:
        s["server"] = Server(s["ptm"])
        total = sum(len(f["positions"]) for f in frames)
        kinds = {"structure": ((), torch.int8), "alloy": ((), torch.int8), "rmsd": ((), torch.float32),
                 "scale": ((), torch.float32), "quat": ((4,), torch.float32), "strain": ((3, 3), torch.float32),
                 "correspondence": ((15,), torch.int32)}
        s["out"] = {k: _pinned((total, *shape), dt) for k, (shape, dt) in kinds.items()}
        s["requests"], at = [], 0
        for f in frames:
            n = len(f["positions"])
            pos = _pinned((n, 3), f["positions"].dtype)
            pos[:] = f["positions"].cpu().numpy()
            sp = None
            if f["species"] is not None:
                sp = _pinned((n,), torch.int8)
                sp[:] = f["species"].cpu().numpy()
            s["requests"].append((pos, f["cell"], f["pbc"], sp, {k: v[at:at + n] for k, v in s["out"].items()}))
            at += n
    return s


def run(s):
    path = s["case"]["path"]
    if path == "frame":
        out = s["ptm"].classify(s["positions"], s["cell"], s["pbc"], species=s["species"], mask=s["mask"],
                                rmsd_max=s["rmsd_max"], outputs=s["outputs"], ordering=s["case"]["ordering"])
        if s["case"]["derived"]:
            out["histogram"] = s["ptm"].rmsd_histogram(out["structure"], out["rmsd"], nbins=100, rmsd_max=0.3)
        return out
    if path == "host":
        return s["ptm"].classify_host(s["positions"], s["cell"], s["pbc"], species=s["species"], mask=s["mask"],
                                      rmsd_max=s["rmsd_max"])
    if path == "batch":
        s["batch"].run()
        return {k: torch.cat([o[k] for o in s["batch"].outputs]) for k in OUTPUTS}
    tickets = [s["server"].submit(pos, cell, pbc, species=sp, mask=s["mask"], rmsd_max=s["rmsd_max"], out=out)
               for pos, cell, pbc, sp, out in s["requests"]]
    for t in tickets:
        s["server"].wait(t)
        s["server"].release(t)
    return s["out"]


def work(case):
    """Bytes: positions and species read once, every output written once.  Operations, per atom: four candidates of 13
    points superposed (18 a point, 214 a solution), 2000 for the winner's outputs, 126 for the vectors; in the
    topological order 18 faces of 17 cuts of about 6 corners, 4 each."""
    case = dict(DEFAULTS, **case)
    per = (24 if case["dtype"] == "float64" else 12) + (1 if case["species"] else 0) + 122 + (16 if case["derived"] else 0)
    flops = 4 * (13 * 18 + 214) + 2000 + 126 + (18 * 17 * 6 * 4 if case["ordering"] == "topological" else 0)
    n = sum(_sizes(case))
    return {"bytes": n * per, "flops": n * flops}


# ------------------------------------------------------------------------------------------- the outputs in 64 bits
# Neighbours by distance, hulls by testing every triple of neighbours on the integers the method quantises them to, and
# every correspondence between the hull and a triangulation of a template's faces, through a labelling of the vertices
# in the order of a walk around them from one directed edge (an adjacency matrix under that labelling, whose first facet
# is fixed, determines the oriented graph).
def _templates():
    g, phi = math.sqrt(0.5), (1 + math.sqrt(5)) / 2
    sgn = (1, -1)
    fcc = [p for x in sgn for y in sgn for p in ((x * g, y * g, 0), (x * g, 0, y * g), (0, x * g, y * g))]
    ring = [(math.cos(k * math.pi / 3), math.sin(k * math.pi / 3), 0) for k in range(6)]
    tri = [(math.cos(k) / math.sqrt(3), math.sin(k) / math.sqrt(3), z * math.sqrt(2 / 3))
           for k in (math.pi / 6, 5 * math.pi / 6, 3 * math.pi / 2) for z in sgn]
    ico = [p for x in sgn for y in sgn for p in ((0, x, y * phi), (x, y * phi, 0), (y * phi, 0, x))]
    axes = [tuple(s * float(i == k) for i in range(3)) for k in range(3) for s in sgn]
    bcc = [(x / 2, y / 2, z / 2) for x in sgn for y in sgn for z in sgn] + axes
    out = []
    for pts in (axes, fcc, ring + tri, ico, bcc):
        p = np.array(pts, float)
        out.append(p * (len(p) + 1) / np.linalg.norm(p, axis=1).sum())
    return out


def _template_rotations(p):
    """Proper rotations of the point set and the permutations they make."""
    i1 = next(i for i in range(1, len(p)) if np.linalg.norm(np.cross(p[0], p[i])) > 1e-6)
    frame = lambda u, v: np.stack([u, v, np.cross(u, v)], 1)  # noqa: E731
    inv, found = np.linalg.inv(frame(p[0], p[i1])), {}
    for u, v in itertools.permutations(range(len(p)), 2):
        R = frame(p[u], p[v]) @ inv
        if np.abs(R @ R.T - np.eye(3)).max() < 1e-9:
            d = np.linalg.norm((p @ R.T)[:, None] - p[None], axis=2)
            if d.min(1).max() < 1e-9:
                found.setdefault(tuple(d.argmin(1)), R)
    return np.array(list(found)), np.array(list(found.values()))


def _template_facets(p):
    """Every triangulation of the hull's faces, counter-clockwise seen from outside: (m, f, 3)."""
    faces = set()
    for a, b, c in itertools.combinations(range(len(p)), 3):
        nrm = np.cross(p[b] - p[a], p[c] - p[a])
        h = (p - p[a]) @ nrm * np.sign(nrm @ p[a])
        if h.max() < 1e-9 and abs(nrm @ p[a]) > 1e-9:
            faces.add(tuple(np.nonzero(h > -1e-9)[0]))
    fixed, split = [], []
    for f in sorted(faces):
        mid = p[list(f)].mean(0)
        e = p[f[0]] - mid
        e2 = np.cross(mid / np.linalg.norm(mid), e)
        f = sorted(f, key=lambda i: math.atan2((p[i] - mid) @ e2, (p[i] - mid) @ e))
        if len(f) == 3:
            fixed.append([tuple(f)])
        else:
            a, b, c, d = f
            split.append(([(a, b, c), (a, c, d)], [(b, c, d), (b, d, a)]))
    return np.array([sum(fixed + list(ch), []) for ch in itertools.product(*split)])


def _third(facets, k):
    """th[i, u, v]: third vertex of the facet left of the directed edge u -> v (facets (m, f, 3))."""
    th = torch.zeros((len(facets), k * k), dtype=torch.int64, device=facets.device)
    for e in range(3):
        u, v, w = facets[..., e], facets[..., (e + 1) % 3], facets[..., (e + 2) % 3]
        th.scatter_(1, u * k + v, w)
    return th


def _labelled(th, adj, k, u, v):
    """Labels from the directed edge u -> v: each vertex in label order is walked around, counter-clockwise from where
    it was first reached, and new vertices are labelled as they are met.  Returns a code of the labelled graph and the
    vertex of each label."""
    m = len(th)
    row = torch.arange(m, device=th.device)
    label = torch.full((m, k), -1, dtype=torch.int64, device=th.device)
    vertex = torch.zeros((m, k), dtype=torch.int64, device=th.device)
    come = torch.zeros((m, k), dtype=torch.int64, device=th.device)
    label[row, u], label[row, v] = 0, 1
    vertex[:, 0], vertex[:, 1], come[:, 0], come[:, 1] = u, v, v, u
    count = torch.full((m,), 2, dtype=torch.int64, device=th.device)
    for i in range(k):
        x, cur = vertex[:, i], come[:, i]
        for _ in range(k - 1):
            cur = th[row, x * k + cur]
            new = label[row, cur] < 0
            at = row[new]
            label[at, cur[new]] = count[new]
            vertex[at, count[new]], come[at, count[new]] = cur[new], x[new]
            count = count + new
    weight = torch.as_tensor(np.random.default_rng(29).integers(-2 ** 62, 2 ** 62, (k, k)), device=th.device)
    order = torch.gather(adj, 1, vertex[:, :, None].expand(-1, -1, k))
    order = torch.gather(order, 2, vertex[:, None, :].expand(-1, k, -1))
    return (order * weight).sum((1, 2)), vertex


def _adjacency(th_facets, k):
    adj = torch.zeros((len(th_facets), k * k), dtype=torch.int64, device=th_facets.device)
    for e in range(3):
        u, v = th_facets[..., e], th_facets[..., (e + 1) % 3]
        adj.scatter_(1, u * k + v, torch.ones_like(u))
        adj.scatter_(1, v * k + u, torch.ones_like(u))
    return adj.view(-1, k, k)


@functools.lru_cache(maxsize=None)
def _candidates(k, mask):
    """Codes of the graphs of the templates with k points, and per code its correspondences (template, slot of label)
    up to the template's rotations: (sorted codes, first row, rows per code, template, slots)."""
    codes, which, slots = [], [], []
    for t, p in enumerate(_templates()):
        if len(p) != k or not mask >> t & 1:
            continue
        facets = torch.as_tensor(_template_facets(p), device=DEVICE)
        perms = torch.as_tensor(_template_rotations(p)[0], device=DEVICE)
        th, adj = _third(facets, k), _adjacency(facets, k)
        pack = 16 ** torch.arange(k, device=DEVICE)
        for f, e in itertools.product(range(facets.shape[1]), range(3)):
            code, vertex = _labelled(th, adj, k, facets[:, f, e], facets[:, f, (e + 1) % 3])
            key = torch.stack([code, (perms[:, vertex] * pack).sum(2).amin(0)], 1)
            codes.append(torch.unique(key, dim=0))
            which.append(torch.full((len(codes[-1]),), t, device=DEVICE))
    if not codes:
        return None
    rows = torch.unique(torch.cat([torch.cat(codes), torch.cat(which)[:, None]], 1), dim=0)
    code, count = torch.unique_consecutive(rows[:, 0], return_counts=True)
    slots = rows[:, 1:2] >> (4 * torch.arange(k, device=DEVICE)) & 15
    return code, torch.cumsum(count, 0) - count, count, rows[:, 2], slots


def _nearest(pos, cell, pbc, k=14, reach=6.0):
    """The k nearest images of every atom: vectors (n, k, 3) by distance.  Small boxes against every image of every
    atom, others by cells of 6 Angstrom, or 9 where an atom's neighbours lie further away; None where 9 do not do."""
    n, H, inv = len(pos), _t(cell), _t(np.linalg.inv(cell))
    f = pos @ inv
    whole = torch.stack([torch.floor(f[:, c]) if pbc[c] else torch.zeros_like(f[:, c]) for c in range(3)], 1)
    pos = pos - whole @ H                                 # only distances are wanted: any image will do
    f = f - whole
    width = 1 / np.linalg.norm(np.linalg.inv(cell), axis=0)
    span = [(0.0, 1.0) if pbc[c] else (float(f[:, c].min()), float(f[:, c].max()) + 1e-9) for c in range(3)]
    nb = [max(1, int((b - a) * width[c] / reach)) for c, (a, b) in enumerate(span)]
    out = torch.empty((n, k, 3), dtype=torch.float64, device=pos.device)
    if any(pbc[c] and nb[c] < 3 for c in range(3)):
        if n > 8000:
            return None
        images = [s for s in itertools.product(*[(-1, 0, 1) if p else (0,) for p in pbc])]
        images.sort(key=lambda s: s != (0, 0, 0))
        table = torch.cat([pos + _t(np.array(s) @ cell) for s in images])
        for a in range(0, n, 256):
            d = table[None] - pos[a:a + 256, None]
            r2 = (d * d).sum(2)
            r2[torch.arange(len(r2)), torch.arange(a, a + len(r2))] = math.inf
            at = torch.topk(r2, k, largest=False, sorted=True).indices
            out[a:a + 256] = torch.gather(d, 1, at[..., None].expand(-1, -1, 3))
        return out
    idx = torch.stack([((f[:, c] - span[c][0]) / (span[c][1] - span[c][0]) * nb[c]).long().clamp(0, nb[c] - 1)
                       for c in range(3)], 1)
    flat = (idx[:, 0] * nb[1] + idx[:, 1]) * nb[2] + idx[:, 2]
    order = torch.argsort(flat, stable=True)
    count = torch.bincount(flat, minlength=int(np.prod(nb)))
    most, start = int(count.max()), torch.cumsum(count, 0) - count
    for a in range(0, n, 4096):
        i = torch.arange(a, min(a + 4096, n), device=pos.device)
        ds = []
        for s in itertools.product((-1, 0, 1), repeat=3):
            c = idx[i] + torch.tensor(s, device=pos.device)
            nbt = torch.tensor(nb, device=pos.device)
            w = torch.div(c, nbt, rounding_mode="floor")
            ok = torch.stack([(w[:, q] == 0) | bool(pbc[q]) for q in range(3)], 1).all(1)
            c = c - w * nbt
            cf = (c[:, 0] * nb[1] + c[:, 1]) * nb[2] + c[:, 2]
            j = start[cf][:, None] + torch.arange(most, device=pos.device)
            ok = ok[:, None] & (torch.arange(most, device=pos.device) < count[cf][:, None])
            j = order[j.clamp(max=n - 1)]
            ok &= (j != i[:, None]) | (w != 0).any(1)[:, None]
            d = pos[j] - pos[i][:, None] + (w.double() @ H)[:, None]
            ds.append(torch.where(ok[..., None], d, torch.full_like(d, 1e9)))
        d = torch.cat(ds, 1)
        r2, at = torch.topk((d * d).sum(2), k, largest=False, sorted=True)
        if float(r2.max()) > reach ** 2:
            return _nearest(pos, cell, pbc, k, 9.0) if reach < 9.0 else None
        out[a:a + len(i)] = torch.gather(d, 1, at[..., None].expand(-1, -1, 3))
    return out


def _horn(S):
    """Largest root of the characteristic polynomial of Horn's matrix of S (m, 3, 3), and that matrix."""
    K = torch.empty((len(S), 4, 4), dtype=torch.float64, device=S.device)
    tr = S[:, 0, 0] + S[:, 1, 1] + S[:, 2, 2]
    K[:, 0, 0] = tr
    K[:, 0, 1:] = torch.stack([S[:, 1, 2] - S[:, 2, 1], S[:, 2, 0] - S[:, 0, 2], S[:, 0, 1] - S[:, 1, 0]], 1)
    K[:, 1:, 0] = K[:, 0, 1:]
    K[:, 1:, 1:] = S + S.transpose(1, 2) - tr[:, None, None] * torch.eye(3, dtype=torch.float64, device=S.device)
    c2, c1, c0 = -2 * (S * S).sum((1, 2)), -8 * torch.linalg.det(S), torch.linalg.det(K)
    lam = torch.sqrt(-1.5 * c2)                            # sqrt(3) |S| is above the sum of the singular values
    for _ in range(60):
        dp = (4 * lam * lam + 2 * c2) * lam + c1
        lam = lam - torch.where(dp > 0, ((lam * lam + c2) * lam + c1) * lam + c0, torch.zeros_like(dp)) / dp.clamp(min=1e-300)
    return lam, K


def _exact_chunk(d, mask, rmsd_max):
    n, dev = len(d), d.device
    top = d.abs().amax((1, 2))
    q = torch.round(d * torch.pow(2.0, 19 - torch.floor(torch.log2(top)) - 1)[:, None, None]).long()
    best = torch.full((n,), math.inf, dtype=torch.float64, device=dev)
    T = [torch.cat([torch.zeros((1, 3), dtype=torch.float64, device=dev), _t(p)]) for p in _templates()]
    win_t = torch.full((n,), -1, dtype=torch.int64, device=dev)
    win = torch.zeros((n, 14), dtype=torch.int64, device=dev)      # template slot of neighbour j
    for k in (6, 12, 14):
        cand = _candidates(k, mask)
        if cand is None:
            continue
        tri = torch.tensor(list(itertools.combinations(range(k), 3)), device=dev)
        a, b, c = (q[:, tri[:, e]] for e in range(3))
        nrm = torch.cross(b - a, c - a, dim=2)
        h = torch.zeros((n, len(tri)), dtype=torch.int64, device=dev)
        for p in range(k):
            s = torch.sign((nrm * (q[:, p:p + 1] - a)).sum(2))
            h += torch.where((tri == p).any(1)[None], torch.zeros_like(s), s)
        face = h.abs() == k - 3
        out = torch.sign((nrm * a).sum(2)) * -torch.sign(h) > 0    # the centre strictly inside
        row = torch.nonzero((face.sum(1) == 2 * k - 4) & (out | ~face).all(1)).flatten()
        if not len(row):
            continue
        at = torch.nonzero(face[row])[:, 1].view(len(row), 2 * k - 4)
        fac = tri[at]
        flip = torch.gather(h[row], 1, at) > 0
        fac = torch.where(flip[..., None], fac[..., [0, 2, 1]], fac)
        whole = (torch.nn.functional.one_hot(fac.flatten(1), k).sum(1) > 0).all(1)
        row, fac = row[whole], fac[whole]
        if not len(row):
            continue
        code, vertex = _labelled(_third(fac, k), _adjacency(fac, k), k, fac[:, 0, 0], fac[:, 0, 1])
        codes, first, count, which, slots = cand
        i = torch.searchsorted(codes, code).clamp(max=len(codes) - 1)
        hit = codes[i] == code
        row, i, vertex = row[hit], i[hit], vertex[hit]
        v = torch.cat([torch.zeros((len(row), 1, 3), dtype=torch.float64, device=dev), d[row, :k]], 1)
        gv = ((v - v.mean(1, keepdim=True)) ** 2).sum((1, 2))
        for r in range(int(count[i].max()) if len(row) else 0):
            use = torch.nonzero(count[i] > r).flatten()
            g = first[i[use]] + r
            slot = torch.empty((len(use), k), dtype=torch.int64, device=dev).scatter_(1, vertex[use], slots[g])
            w = torch.stack([x if len(x) == k + 1 else torch.zeros((k + 1, 3), dtype=torch.float64, device=dev) for x in T])
            w = w[which[g]]
            w = torch.gather(w, 1, torch.cat([torch.zeros_like(slot[:, :1]), slot + 1], 1)[..., None].expand(-1, -1, 3))
            lam, _ = _horn(torch.einsum("nia,nib->nab", w, v[use]))
            r2 = ((w * w).sum((1, 2)) - lam * lam / gv[use]) / (k + 1)
            better = r2 < best[row[use]] - 1e-13
            u = row[use][better]
            best[u], win_t[u] = r2[better], which[g][better]
            win[u, :k] = slot[better]
    res = {"rmsd": torch.full((n,), math.inf, dtype=torch.float64, device=dev)}
    for name, shape in (("scale", (n,)), ("quat", (n, 4)), ("strain", (n, 3, 3)), ("von_mises", (n,)), ("rodrigues", (n, 3))):
        res[name] = torch.zeros(shape, dtype=torch.float64, device=dev)
    res["quat"][:, 0] = 1
    for t, p in enumerate(_templates()):
        row = torch.nonzero(win_t == t).flatten()
        if not len(row):
            continue
        k = len(p)
        v = torch.cat([torch.zeros((len(row), 1, 3), dtype=torch.float64, device=dev), d[row, :k]], 1)
        v = v - v.mean(1, keepdim=True)
        w = T[t][torch.cat([torch.zeros((len(row), 1), dtype=torch.int64, device=dev), win[row, :k] + 1], 1)]
        S = torch.einsum("nia,nib->nab", w, v)
        lam, K = _horn(S)
        quat = torch.linalg.eigh(K)[1][..., -1]
        scale = lam / (v * v).sum((1, 2))
        x0, x1, x2, x3 = quat.unbind(1)
        R = torch.stack([1 - 2 * (x2 * x2 + x3 * x3), 2 * (x1 * x2 - x0 * x3), 2 * (x1 * x3 + x0 * x2),
                         2 * (x1 * x2 + x0 * x3), 1 - 2 * (x1 * x1 + x3 * x3), 2 * (x2 * x3 - x0 * x1),
                         2 * (x1 * x3 - x0 * x2), 2 * (x2 * x3 + x0 * x1), 1 - 2 * (x1 * x1 + x2 * x2)], 1).view(-1, 3, 3)
        rmsd = (((scale[:, None, None] * v - w @ R.transpose(1, 2)) ** 2).sum((1, 2)) / (k + 1)).sqrt()
        # the equivalent orientation of the smallest angle
        G = torch.linalg.eigh(torch.stack([_horn(_t(r.T)[None])[1][0] for r in _template_rotations(p)[1]]))[1][..., -1]
        prod = torch.stack([
            x0[:, None] * G[:, 0] - x1[:, None] * G[:, 1] - x2[:, None] * G[:, 2] - x3[:, None] * G[:, 3],
            x0[:, None] * G[:, 1] + x1[:, None] * G[:, 0] + x2[:, None] * G[:, 3] - x3[:, None] * G[:, 2],
            x0[:, None] * G[:, 2] - x1[:, None] * G[:, 3] + x2[:, None] * G[:, 0] + x3[:, None] * G[:, 1],
            x0[:, None] * G[:, 3] + x1[:, None] * G[:, 2] - x2[:, None] * G[:, 1] + x3[:, None] * G[:, 0]], 2)
        pick = prod[..., 0].abs().argmax(1)
        quat = prod[torch.arange(len(row), device=dev), pick]
        quat = quat * torch.where(quat[:, :1] < 0, -1.0, 1.0)
        # both sets scaled to mean distance one; the templates' second moments are isotropic
        A = 3 * S.transpose(1, 2) / float((p * p).sum()) / torch.linalg.norm(v, dim=2).mean(1)[:, None, None]
        e, X = torch.linalg.eigh(A @ A.transpose(1, 2))
        sig = e.clamp(min=0).sqrt()
        sig[:, 0] *= torch.where(torch.linalg.det(A) < 0, -1.0, 1.0)
        P = X @ (sig[:, :, None] * X.transpose(1, 2))
        dev_p = P - torch.diagonal(P, dim1=1, dim2=2).sum(1)[:, None, None] / 3 * torch.eye(3, dtype=torch.float64, device=dev)
        ok = rmsd <= rmsd_max
        for name, x in (("rmsd", rmsd), ("scale", scale), ("quat", quat), ("strain", P),
                        ("von_mises", (1.5 * (dev_p ** 2).sum((1, 2))).sqrt()), ("rodrigues", quat[:, 1:] / quat[:, :1])):
            res[name][row[ok]] = x[ok]
    return res


def exact(case, seed):
    """The floating outputs in 64 bits.  None where several frames or a large one would take long, where a perfect
    lattice's coplanar faces and equal distances are split by the method's tie rules, and for the topological order,
    whose groups of nearly equal face areas are such a rule too; whole numbers have no 64-bit value of their own."""
    case = dict(DEFAULTS, **case)
    if sum(_sizes(case)) > 300000 or case["frames"] > 1 or case["sigma"] < 0.02 or case["ordering"] != "euclidean":
        return None
    f = _one(case, seed)
    d = _nearest(f["positions"].double(), f["cell"], f["pbc"])
    if d is None:
        return None
    parts = [_exact_chunk(d[a:a + 8192], case["mask"], case["rmsd_max"] or math.inf) for a in range(0, len(d), 8192)]
    names = OUTPUTS + (DERIVED if case["derived"] else ())
    out = {k: torch.cat([p[k] for p in parts]) if k in parts[0] else None for k in names}
    if case["derived"]:
        out["histogram"] = None
    return out
