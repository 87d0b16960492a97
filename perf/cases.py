"""The work a user of this package has it do, as cases that can be timed and compared.

A case names a surface (sphere, ellipsoid or a smoothed molecular surface) on its grid, one public entry
point, and the arithmetic that entry point is called with:

  matvec  one application of the operator of Eq. (2.30) to a density on the device, direct sum or treecode;
  map     the reaction potential of Eq. (2.31) at many points (a potential map);
  energy  the polarization energy of Eq. (3.3), one evaluation point per charge;
  solve   a solve on a handle that exists (new charges are part of the handle);
  step    the whole call for a new surface: setup, solve, energy;
  batch   several systems solved together.

The single-precision operator and map return FP64 arrays that carry single precision; a caller of those
keeps them as float32 (the vectors of an inner FP32 Krylov iteration, the voxels of a potential map), and
so does run().  Everything else is kept in FP64.

exact() restates the discretization in plain FP64 torch from its definition: finite-difference geometry
(Sec. 2.1), correction nodes and weights (Sec. 2.4, with the lattice limits of Eq. (2.29) by Ewald
summation through the incomplete gamma function), K-reg rows (Sec. 2.3), the dense sum, and GMRES.
"""
import functools
import math

import numpy as np
import torch

import paper_2210_03699_gb300 as ctr

EPS_IN, EPS_OUT, KAPPA = 1.0, 80.0, 0.1257   # dielectric constants and screening of Sec. 2.6
TUBE = 2.0                                   # tube half-width in grid spacings (Sec. 2.6)
PRECISION = {"fp32": ctr.FP32_REFINE, "df64": ctr.DF64, "fp64": ctr.FP64}
RATIO = EPS_OUT / EPS_IN
LAM = (0.5 * (1.0 + RATIO), 0.5 * (1.0 + 1.0 / RATIO))
# Floating-point operations of one ordered pair of nodes (K11, K12, K21, K22 of Eq. (1.4) and four weighted
# sums, a fused multiply-add as two, exponential and reciprocal root as one each) and of one (point, node)
# pair of Eq. (2.31); operator applications that a solve to 1e-10 needs.
PAIR_FLOPS, MAP_FLOPS, APPLICATIONS = 62, 33, 14


# ---------------------------------------------------------------- cases
def listed():
    return [
        # the sphere of Sec. 2.6 (3 214 nodes): one application of the inner operator, where launches count
        dict(name="matvec_fp32_sphere_3k", do="matvec", precision="fp32", surface="sphere", size=2.0, h=0.25),
        # a 250-atom molecule: one application of the inner operator of a refined solve
        dict(name="matvec_fp32_molecule", do="matvec", precision="fp32", surface="molecule", size=250, h=0.5),
        # the refinement residual's operator on the ellipsoid at h = 0.1 (44 597 nodes)
        dict(name="matvec_df64_ellipsoid_45k", do="matvec", precision="df64", surface="ellipsoid", size=4.0, h=0.1),
        # the default arithmetic of matvec() on the ellipsoid at h = 0.2 (11 203 nodes)
        dict(name="matvec_fp64_ellipsoid_11k", do="matvec", precision="fp64", surface="ellipsoid", size=4.0, h=0.2),
        # the accelerated operators (Sec. 2.5) at h = 0.05 (178 575 nodes): inner and residual arithmetic
        dict(name="matvec_tree_fp32_179k", do="matvec", precision="fp32", surface="ellipsoid", size=4.0, h=0.05,
             tree=True),
        dict(name="matvec_tree_df64_179k", do="matvec", precision="df64", surface="ellipsoid", size=4.0, h=0.05,
             tree=True),
        # a potential map of 200 000 points around the ellipsoid at h = 0.1
        dict(name="map_fp32_200k_points", do="map", precision="fp32", surface="ellipsoid", size=4.0, h=0.1,
             points=200000),
        # the energy of a 500-atom molecule, one evaluation point per atom, FP64
        dict(name="energy_molecule_500", do="energy", surface="molecule", size=500, h=0.5),
        # the smallest solve with the default options (FP64 throughout): the sphere of Sec. 2.6
        dict(name="solve_fp64_sphere_3k", do="solve", precision="fp64", surface="sphere", size=2.0, h=0.25),
        # a small molecule, mixed precision: many short steps
        dict(name="solve_molecule_60", do="solve", precision="fp32", surface="molecule", size=60, h=0.5),
        # a new surface from its signed distance to its energy, the benchmark's size
        dict(name="step_ellipsoid_179k", do="step", precision="fp32", surface="ellipsoid", size=4.0, h=0.05),
        # molecules of 20 to 120 atoms solved together
        dict(name="batch_molecules_6", do="batch", precision="fp32", surface="molecule", size=20, largest=120,
             members=6, h=0.5),
    ]


def draw(rng):
    """One more case of the listed ranges (nodes 3e3 to 1.8e5, points 1 to 2e5, 20 to 500 atoms)."""
    def between(lo, hi):
        return math.exp(rng.uniform(math.log(lo), math.log(hi)))

    def surface(lo, hi):
        """A surface of about lo..hi nodes: M = 4 area / h^2 (a tube of half-width 2 h)."""
        kind, nodes = rng.choice(("sphere", "ellipsoid", "molecule")), between(lo, hi)
        if kind == "sphere":
            size = round(rng.uniform(1.5, 6.0), 3)
            return dict(surface=kind, size=size, h=round(math.sqrt(16.0 * math.pi * size * size / nodes), 5))
        if kind == "ellipsoid":
            size = round(rng.uniform(3.0, 6.0), 3)
            # the tube and its stencils stay off the medial axis (c^2/a = size/4 below the surface)
            return dict(surface=kind, size=size, h=round(min(0.055 * size, math.sqrt(27.9 * size * size / nodes)), 5))
        h = rng.choice((0.5, 0.35))
        atoms = min(500, max(20, int(nodes * h * h / 68.0)))   # about 17 A^2 of surface per atom
        return dict(surface=kind, size=atoms, h=h)

    do = rng.choice(("matvec", "matvec", "matvec", "tree", "map", "energy", "solve", "step", "batch"))
    if do == "matvec":
        p = rng.choice(("fp32", "df64", "fp64"))
        case = dict(do=do, precision=p, **surface(3e3, {"fp32": 1.7e5, "df64": 9e4, "fp64": 2.5e4}[p]))
        if rng.random() < 0.2 and case["h"] > 0.1:
            case["kreg"] = True
        return case
    if do == "tree":
        return dict(do="matvec", precision=rng.choice(("fp32", "df64")), tree=True, **surface(4e4, 1.7e5))
    if do == "map":
        p = rng.choice(("fp32", "fp32", "df64", "fp64"))
        hi = {"fp32": 2e5, "df64": 5e4, "fp64": 5e3}[p]
        return dict(do=do, precision=p, points=int(between(1, hi)), **surface(3e3, 9e4))
    if do == "energy":
        return dict(do=do, **surface(3e3, 9e4))
    if do == "solve":
        p = rng.choice(("fp32", "fp32", "fp64"))
        return dict(do=do, precision=p, **surface(3e3, {"fp32": 4e4, "fp64": 7e3}[p]))
    if do == "step":
        return dict(do=do, precision="fp32", **surface(3e3, 9e4))
    small = rng.randint(20, 60)
    return dict(do=do, precision="fp32", surface="molecule", size=small, largest=rng.randint(small, 150),
                members=rng.randint(2, 8), h=0.5)


# ---------------------------------------------------------------- surfaces
def _walk(atoms):
    """Self-avoiding random walk of `atoms` steps of 1.5 A: centres and radii."""
    g = np.random.Generator(np.random.PCG64(atoms))
    pos, fails = [np.zeros(3)], 0
    while len(pos) < atoms:
        step = g.normal(size=3)
        new = pos[-1] + 1.5 * step / np.linalg.norm(step)
        if len(pos) > 1 and np.min(np.linalg.norm(np.array(pos[:-1]) - new, axis=1)) < 2.0:
            fails += 1
            if fails > 100 and len(pos) > 2:
                pos.pop()
                fails = 0
            continue
        pos.append(new)
        fails = 0
    xyz = np.array(pos)
    return xyz - xyz.mean(axis=0), g.choice([1.2, 1.5, 1.6, 1.7, 1.8], size=atoms)


def _member_sizes(case):
    """Atom counts of a batch, evenly spread over the logarithm."""
    n, lo, hi = case["members"], case["size"], case["largest"]
    return [int(round(lo * (hi / lo) ** (i / max(1, n - 1)))) for i in range(n)]


@functools.lru_cache(maxsize=None)
def _surface(kind, size, h):
    """(grid n, origin, signed distance as a flat CUDA tensor, x fastest; atom centres of a molecule)."""
    atoms = None
    if kind == "molecule":
        atoms, radii = _walk(int(size))
        lo, hi = (atoms - radii[:, None]).min(axis=0), (atoms + radii[:, None]).max(axis=0)
        lo, hi = lo - 2.0 - (TUBE + 4) * h, hi + 2.0 + (TUBE + 4) * h
    else:
        axes = np.array([1.0, 1.0, 1.0] if kind == "sphere" else [1.0, 0.75, 0.5]) * size
        lo, hi = -(axes + (TUBE + 4) * h), axes + (TUBE + 4) * h
    n = [int(math.ceil((b - a) / h)) + 1 for a, b in zip(lo, hi)]
    if kind != "molecule":   # a node at the centre
        n = [v + 1 - v % 2 for v in n]
        lo = [-h * (v // 2) for v in n]
    origin = tuple(float(v) for v in lo)
    ax = [origin[c] + h * torch.arange(n[c], dtype=torch.float64, device="cuda") for c in range(3)]
    Z, Y, X = torch.meshgrid(ax[2], ax[1], ax[0], indexing="ij")
    p = torch.stack([X.reshape(-1), Y.reshape(-1), Z.reshape(-1)], dim=1)
    if kind == "sphere":
        d = p.square().sum(1).sqrt() - size
    elif kind == "ellipsoid":
        d = _ellipsoid_distance(p, torch.tensor(axes, device="cuda"))
    else:   # smoothed molecular surface: soft minimum (1 A) of the distances to the atoms' balls
        c, r = torch.tensor(atoms, device="cuda"), torch.tensor(radii, device="cuda")
        d = torch.cat([-torch.logsumexp(r - torch.cdist(q, c), dim=1) for q in p.split(1 << 18)])
    return tuple(n), origin, d.contiguous(), atoms


def _ellipsoid_distance(p, a):
    """Signed distance (positive outside): bisection for the multiplier t of the closest point (a coordinate
    on a symmetry plane is taken a hair off it, where the closest point is unique)."""
    y, a2 = p.abs().clamp_min(1e-12), a * a
    low = torch.full_like(y[:, 0], -float(a2.min()))
    high = low + (a2 * y * y).sum(1).sqrt()
    for _ in range(80):
        t = 0.5 * (low + high)
        f = (a * y / (t[:, None] + a2)).square().sum(1)
        low, high = torch.where(f > 1, t, low), torch.where(f > 1, high, t)
    d = (y - a2 * y / (0.5 * (low + high)[:, None] + a2)).square().sum(1).sqrt()
    return torch.where((p / a).square().sum(1) > 1, d, -d)


def _charges(case, seed, atoms):
    """Charges inside the surface: at a molecule's atoms, else three within 0.6 of the semi-axes."""
    g = np.random.Generator(np.random.PCG64(seed))
    if atoms is not None:
        return atoms, g.normal(0.0, 0.4, size=len(atoms))
    axes = np.array([1.0, 1.0, 1.0] if case["surface"] == "sphere" else [1.0, 0.75, 0.5]) * case["size"]
    u = g.normal(size=(3, 3))
    u *= (g.uniform(size=(3, 1)) ** (1 / 3)) / np.linalg.norm(u, axis=1, keepdims=True)
    return 0.6 * axes * u, g.uniform(0.2, 1.0, size=3) * np.array([1.0, -1.0, 1.0])


def _options(case):
    o = dict(tube_halfwidth=TUBE * case["h"], precision=PRECISION[case.get("precision", "fp32")])
    if case.get("kreg"):
        o["method"] = ctr.METHOD_KREG
    if case.get("tree"):
        o["farfield"] = ctr.FARFIELD_TREECODE
    return ctr.Options(**o)


def _inputs(case, seed, size=None):
    """(arguments of CtrIbim, case with its member's size)."""
    case = dict(case, size=case["size"] if size is None else size)
    n, origin, d, atoms = _surface(case["surface"], case["size"], case["h"])
    xyz, q = _charges(case, seed, atoms)
    return (n, origin, case["h"], d.clone(), EPS_IN, EPS_OUT, KAPPA, xyz, q), case


def _field(case, seed, g):
    """psi and its normal derivative on the nodes, of the size and smoothness of a solution, from the
    charges' Coulomb field g = (g1, g2)."""
    m = g.numel() // 2
    return (g[:m] / EPS_OUT).contiguous(), (-EPS_IN * g[m:]).contiguous()


def _density(seed, g):
    """A Krylov vector: the right-hand side's shape plus noise of half its size."""
    noise = torch.randn(g.numel(), dtype=torch.float64, generator=torch.Generator().manual_seed(seed)).to(g.device)
    m = g.numel() // 2
    scale = torch.cat([g[:m].square().mean().sqrt().expand(m), g[m:].square().mean().sqrt().expand(m)])
    return g / scale + 0.5 * noise


def _points(case, seed):
    """Evaluation points of a map: around grid nodes at least two tube half-widths off the surface."""
    n, origin, d, _ = _surface(case["surface"], case["size"], case["h"])
    gen = torch.Generator().manual_seed(seed)
    free = torch.nonzero(d.abs() > 2 * TUBE * case["h"]).reshape(-1).cpu()
    at = free[torch.randint(free.numel(), (case["points"],), generator=gen)]
    ijk = torch.stack([at % n[0], (at // n[0]) % n[1], at // (n[0] * n[1])], dim=1).double()
    jitter = torch.rand(ijk.shape, dtype=torch.float64, generator=gen) - 0.5
    return (torch.tensor(origin, dtype=torch.float64) + case["h"] * (ijk + jitter)).to(d.device)


# ---------------------------------------------------------------- measured passes
def prepare(case, seed):
    do, state = case["do"], {"case": case}
    if do == "batch":
        state["systems"] = []
        for k, size in enumerate(_member_sizes(case)):
            args, c = _inputs(case, seed + 1000 * k, size)
            state["systems"].append(ctr.CtrIbim(*args, options=_options(c)))
        return state
    args, _ = _inputs(case, seed)
    if do == "step":
        state["args"] = args
        return state
    s = state["system"] = ctr.CtrIbim(*args, options=_options(case))
    if do == "solve":
        return state
    g = torch.from_numpy(s.rhs()).cuda()
    if do == "matvec":
        state["x"] = _density(seed, g)
    else:
        state["psi"], state["dpsi"] = _field(case, seed, g)
    if do == "map":
        state["points"] = _points(case, seed)
    return state


def run(state):
    case = state["case"]
    do = case["do"]
    if do == "matvec":
        y = state["system"].matvec(state["x"], PRECISION[case["precision"]])
        return y.float() if case["precision"] == "fp32" else y
    if do == "map":
        v = state["system"].potential_map(state["psi"], state["dpsi"], state["points"], PRECISION[case["precision"]])
        return v.float() if case["precision"] == "fp32" else v
    if do == "energy":
        energy, at_charges = state["system"].energy(state["psi"], state["dpsi"])
        return {"energy": energy, "at_charges": at_charges}
    if do == "solve":
        psi, dpsi, _ = state["system"].solve(device=True)
        return {"psi": psi, "dpsi": dpsi}
    if do == "step":
        with ctr.CtrIbim(*state["args"], options=_options(case)) as s:
            psi, dpsi, _ = s.solve(device=True)
            energy, at_charges = s.energy(psi, dpsi)
        return {"psi": psi, "dpsi": dpsi, "energy": energy, "at_charges": at_charges}
    return [{"psi": psi, "dpsi": dpsi} for psi, dpsi, _ in ctr.batch_solve(state["systems"], device=True)]


def work(case):
    """Bytes and operations of one pass: the nodes' positions, normals and weights and the vectors, once;
    every ordered pair of nodes once (a solve: once per application it needs)."""
    def nodes(size):
        d = _surface(case["surface"], size, case["h"])[2]
        return int((d.abs() < TUBE * case["h"]).sum())

    if case["do"] == "batch":
        ms = [nodes(s) for s in _member_sizes(case)]
        return {"bytes": sum(88 * m for m in ms) * APPLICATIONS, "flops": sum(PAIR_FLOPS * m * m for m in ms) * APPLICATIONS}
    m = nodes(case["size"])
    if case["do"] == "matvec":
        return {"bytes": 88 * m, "flops": PAIR_FLOPS * m * m * (0.05 if case.get("tree") else 1)}
    if case["do"] in ("map", "energy"):
        p = case.get("points") or (case["size"] if case["surface"] == "molecule" else 3)
        return {"bytes": 72 * m + 32 * p, "flops": MAP_FLOPS * m * p}
    return {"bytes": 88 * m * APPLICATIONS, "flops": PAIR_FLOPS * m * m * APPLICATIONS}


# ---------------------------------------------------------------- the same in plain FP64
MODES, HALF, SAMPLES = 9, 19, 64   # even Fourier modes 0..16, shifts -19/32..19/32, samples of the DFT


@functools.lru_cache(maxsize=None)
def _tables():
    """The limit of Eq. (2.29) for s = |y|^-1 e^{ik psi}, k = 0, 2, .., 16, at the shifts (i, j)/32: minus the
    regularised lattice sum of e^{ik psi}/|n - a| over n != 0, by Ewald summation (upper incomplete gamma
    functions of order (k + 1)/2 in both spaces).  Complex, (MODES, 39, 39)."""
    a = torch.arange(-HALF, HALF + 1, dtype=torch.float64) / 32.0
    a = torch.stack(torch.meshgrid(a, a, indexing="ij"), dim=-1)[:, :, None, :]
    r = torch.arange(-7, 8, dtype=torch.float64)
    n = torch.stack(torch.meshgrid(r, r, indexing="ij"), dim=-1).reshape(-1, 2)
    n = n[n.abs().sum(1) > 0]
    out = []
    for q in range(MODES):
        order = torch.tensor(q + 0.5, dtype=torch.float64)

        def harmonic(x, upper):
            rad = x.square().sum(-1).sqrt()
            safe = rad.clamp_min(1e-30)
            gamma = torch.special.gammaincc if upper else torch.special.gammainc
            return torch.complex(x[..., 0] / safe, x[..., 1] / safe) ** (2 * q) * gamma(order, math.pi * rad * rad) / safe

        total = harmonic(n - a, True).sum(-1)
        own = harmonic(-a, False)[..., 0]
        own[HALF, HALF] = 2.0 if q == 0 else 0.0
        wave = torch.polar(torch.ones(()).double(), -2.0 * math.pi * (a * n).sum(-1))
        total = total - own + (-1) ** q * (harmonic(n, True) * wave).sum(-1) - (2.0 if q == 0 else 0.0)
        out.append(-total)
    return torch.stack(out).cuda()


@functools.lru_cache(maxsize=2)
def _discretize(kind, size, h, kreg):
    """Nodes, geometry and correction entries (target, node, omega11, omega12, omega21, omega22)."""
    n, origin, d, _ = _surface(kind, size, h)
    eps = TUBE * h
    lin = torch.nonzero(d.abs() < eps).reshape(-1)
    idx = torch.stack([lin % n[0], (lin // n[0]) % n[1], lin // (n[0] * n[1])], dim=1)
    stride = (1, n[0], n[0] * n[1])

    def at(*shift):
        return d[lin + sum(s * t for s, t in zip(shift, stride))]

    e = ((1, 0, 0), (0, 1, 0), (0, 0, 1))
    minus = [tuple(-v for v in u) for u in e]
    grad = torch.stack([(at(*e[c]) - at(*minus[c])) / (2.0 * h) for c in range(3)], dim=1)
    norm = ((grad[:, 0] * grad[:, 0] + grad[:, 1] * grad[:, 1]) + grad[:, 2] * grad[:, 2]).sqrt()
    nrm = grad / norm[:, None]
    org = torch.tensor(origin, dtype=torch.float64, device=d.device)
    y = org + h * idx.double()
    dist = d[lin]
    P = y - dist[:, None] * nrm
    H = torch.zeros(lin.numel(), 3, 3, dtype=torch.float64, device=d.device)
    for a in range(3):
        for b in range(a, 3):
            corner = [at(*[s * u + t * v for u, v in zip(e[a], e[b])]) for s in (1, -1) for t in (1, -1)]
            H[:, a, b] = H[:, b, a] = (corner[0] - corner[1] - corner[2] + corner[3]) / (4.0 * h * h)
    # tangent basis and the level set's shape operator S in it
    axis = torch.nn.functional.one_hot(nrm.abs().argmin(dim=1), 3).double()
    e1 = torch.linalg.cross(nrm, axis)
    e1 = e1 / e1.norm(dim=1, keepdim=True)
    E = torch.stack([e1, torch.linalg.cross(nrm, e1)], dim=1)
    S = E @ H @ E.transpose(1, 2) / norm[:, None, None]
    mean, half = 0.5 * (S[:, 0, 0] + S[:, 1, 1]), 0.5 * (S[:, 0, 0] - S[:, 1, 1])
    rad = torch.hypot(half, 0.5 * (S[:, 0, 1] + S[:, 1, 0]))
    level = torch.stack([mean - rad, mean + rad], dim=1)
    curv = level / (1.0 - dist[:, None] * level)
    bad = ~torch.isfinite(curv).all(1) | (curv.abs().amax(1) * (eps + h) >= 0.8)
    bad |= bool(kreg)
    J = torch.where(bad, torch.ones_like(dist), (1.0 - dist * level[:, 0]) * (1.0 - dist * level[:, 1]))
    W = J * 0.5 * (1.0 + torch.cos(math.pi * dist / eps)) / eps
    node_of = torch.full((d.numel(),), -1, dtype=torch.int64, device=d.device)
    node_of[lin] = torch.arange(lin.numel(), device=d.device)
    size_n = torch.tensor(n, device=d.device)

    # correction planes of the good rows: the nearest node to the normal line on each
    parts = []
    good = torch.nonzero(~bad).reshape(-1)
    if good.numel():
        a = nrm[good].abs().argmax(dim=1)
        b, c = torch.where(a == 0, 1, 0), torch.where(a == 2, 1, 2)

        def pick(v, k):
            return v.gather(1, k[:, None]).reshape(-1)

        planes = int(math.ceil(2.0 * eps / h)) + 2
        for shift in range(-planes, planes + 1):
            ka = pick(idx[good], a) + shift
            eta = ((org[a] + h * ka.double()) - pick(P[good], a)) / pick(nrm[good], a)
            sb = ((pick(P[good], b) + eta * pick(nrm[good], b)) - org[b]) / h
            sc = ((pick(P[good], c) + eta * pick(nrm[good], c)) - org[c]) / h
            kb, kc = torch.floor(sb + 0.5), torch.floor(sc + 0.5)
            cell = torch.zeros_like(idx[good])
            for k, v in ((a, ka), (b, kb.long()), (c, kc.long())):
                cell.scatter_(1, k[:, None], v[:, None])
            ok = (eta.abs() <= eps + h) & ((cell >= 0) & (cell < size_n)).all(1)
            node = node_of[(torch.where(ok[:, None], cell, 0) * torch.tensor(stride, device=d.device)).sum(1)]
            ok = torch.nonzero(ok & (node >= 0)).reshape(-1)
            wa, wb = _weights(E[good[ok]], S[good[ok]], dist[good[ok]], b[ok], c[ok], eta[ok], (sb - kb)[ok], (sc - kc)[ok])
            parts.append(torch.stack([good[ok].double(), node[ok].double(), (1.0 - RATIO) * wa,
                                      torch.full_like(wa, KAPPA / (4.0 * math.pi)), KAPPA * KAPPA * wb,
                                      (1.0 - 1.0 / RATIO) * wa]))
    # K-reg rows: every tube node within 2 h of the normal line, omega12 only
    tau, reach = 2.0 * h, int(math.ceil((eps + 2.0 * h) / h)) + 1
    c12 = (math.exp(-KAPPA * tau) - 1.0 + KAPPA * tau) / (2.0 * math.pi * KAPPA * tau * tau)
    r = torch.arange(-reach, reach + 1, device=d.device)
    cube = torch.stack(torch.meshgrid(r, r, r, indexing="ij"), dim=-1).reshape(-1, 3)
    for rows in torch.nonzero(bad).reshape(-1).split(4096):
        cell = idx[rows][:, None, :] + cube
        inside = ((cell >= 0) & (cell < size_n)).all(-1)
        node = node_of[(torch.where(inside[..., None], cell, 0) * torch.tensor(stride, device=d.device)).sum(-1)]
        v = org + h * cell.double() - P[rows][:, None, :]
        nr = nrm[rows][:, None, :]
        s = (v[..., 0] * nr[..., 0] + v[..., 1] * nr[..., 1]) + v[..., 2] * nr[..., 2]
        t = v - s[..., None] * nr
        q2 = (t[..., 0] * t[..., 0] + t[..., 1] * t[..., 1]) + t[..., 2] * t[..., 2]
        row, col = torch.nonzero(inside & (node >= 0) & (q2 < tau * tau), as_tuple=True)
        zero = torch.zeros(row.numel(), dtype=torch.float64, device=d.device)
        parts.append(torch.stack([rows[row].double(), node[row, col].double(), zero, zero + c12, zero, zero]))
    ent = torch.cat(parts, dim=1)
    ent = ent[:, torch.argsort(ent[0], stable=True)]
    return {"h": h, "P": P, "n": nrm, "W": W, "row": ent[0].long(), "col": ent[1].long(), "w": ent[2:]}


def _weights(E, S, dist, b, c, eta, alpha, beta):
    """omega_A and omega_B (Eq. (2.28)) of correction entries: 64 samples of the angular functions, their
    even Fourier coefficients, the tables by degree-5 Lagrange interpolation in both shifts."""
    T = _tables()
    eye = torch.eye(2, dtype=torch.float64, device=E.device)
    M = -torch.linalg.solve(eye - dist[:, None, None] * S, S)
    D0 = torch.linalg.inv(eye - eta[:, None, None] * M)
    A = torch.stack([E.gather(2, k[:, None, None].expand(-1, 2, 1))[:, :, 0] for k in (b, c)], dim=2)
    th = 2.0 * math.pi * torch.arange(SAMPLES, dtype=torch.float64, device=E.device) / SAMPLES
    k = 2.0 * torch.arange(MODES, dtype=torch.float64, device=E.device)[:, None]
    scale = torch.full((MODES, 1), 2.0 / SAMPLES, dtype=torch.float64, device=E.device)
    scale[0] = 1.0 / SAMPLES
    C, Sn = scale * torch.cos(k * th), scale * torch.sin(k * th)

    def lagrange(x):
        first = torch.floor(x * 32.0).long() - 2
        nodes = (first[:, None] + torch.arange(6, device=x.device)) / 32.0
        cols = []
        for m in range(6):
            v = torch.ones_like(x)
            for l in range(6):
                if l != m:
                    v = v * (x - nodes[:, l]) / (nodes[:, m] - nodes[:, l])
            cols.append(v)
        return first + HALF, torch.stack(cols, dim=1)

    out = []
    for part in torch.arange(E.shape[0], device=E.device).split(1 << 16):
        v = D0[part] @ A[part] @ torch.stack([torch.cos(th), torch.sin(th)])
        vv = v.square().sum(1)
        lB = 1.0 / (8.0 * math.pi * vv.sqrt())
        lA = (v * (M[part] @ v)).sum(1) * lB / vv
        i0, ci = lagrange(alpha[part])
        j0, cj = lagrange(beta[part])
        t = torch.zeros(MODES, part.numel(), dtype=torch.complex128, device=E.device)
        for p in range(6):
            for r in range(6):
                t = t + ci[:, p] * cj[:, r] * T[:, i0 + p, j0 + r]
        out.append(torch.stack([((l @ C.T).T * t.real + (l @ Sn.T).T * t.imag).sum(0) for l in (lA, lB)]))
    return torch.cat(out, dim=1) if out else torch.zeros(2, 0, dtype=torch.float64, device=E.device)


def _coulomb(D, xyz, q):
    """The right-hand side (Eq. (2.12))."""
    xyz, q = torch.tensor(xyz, device="cuda"), torch.tensor(q, device="cuda") / (4.0 * math.pi * EPS_IN)
    g1, g2 = torch.zeros_like(D["W"]), torch.zeros_like(D["W"])
    for z, v in zip(xyz, q):
        d = D["P"] - z
        r = d.square().sum(1).sqrt()
        g1 += v / r
        g2 -= v * (d * D["n"]).sum(1) / r ** 3
    return torch.cat([g1, g2])


def _kernels(x, nx, P, n):
    """4 pi K11, K12, K21, K22 of Eq. (1.4) for the targets x against every node (entries at r = 0 are not
    finite; the dense sum leaves them out with the correction nodes)."""
    d = [x[:, c, None] - P[None, :, c] for c in range(3)]
    r2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2]
    dy = d[0] * n[:, 0] + d[1] * n[:, 1] + d[2] * n[:, 2]
    dx = d[0] * nx[:, 0, None] + d[1] * nx[:, 1, None] + d[2] * nx[:, 2, None]
    del d
    nn = nx @ n.T
    ri = r2.rsqrt()
    kr = KAPPA * r2 * ri
    ex = torch.exp(-kr)
    s = ri / r2
    e1 = ex * (1.0 + kr)
    K21 = s * ((1.0 - e1) * nn - (3.0 - ex * (3.0 + kr * (3.0 + kr))) * dx * dy / r2)
    return dy * s * (1.0 - RATIO * e1), -torch.expm1(-kr) * ri, K21, -dx * s * (1.0 - e1 / RATIO)


def _rows(D, rows):
    """K11, -K12, K21, -K22 rows with weights h^3 W/(4 pi), correction nodes left out."""
    K = _kernels(D["P"][rows], D["n"][rows], D["P"], D["n"])
    lo, hi = torch.searchsorted(D["row"], torch.stack([rows[0], rows[-1] + 1])).tolist()
    r, c = D["row"][lo:hi] - rows[0], D["col"][lo:hi]
    w = D["h"] ** 3 * D["W"] / (4.0 * math.pi)
    for m in K:
        m[r, c] = 0.0
    return K[0] * w, -K[1] * w, K[2] * w, -K[3] * w


def _correction(D, x):
    m = D["W"].numel()
    r1, r2, Wm = x[:m][D["col"]], x[m:][D["col"]], D["W"][D["col"]]
    h2, h3 = D["h"] ** 2, D["h"] ** 3
    w11, w12, w21, w22 = D["w"]
    y = torch.zeros_like(x)
    y.index_add_(0, D["row"], Wm * (h2 * w11 * r1 - h3 * w12 * r2))
    y.index_add_(0, D["row"] + m, Wm * (h2 * w21 * r1 - h2 * w22 * r2))
    return y


def _apply(D, x):
    m = D["W"].numel()
    y = torch.cat([LAM[0] * x[:m], LAM[1] * x[m:]]) + _correction(D, x)
    for rows in torch.arange(m, device=x.device).split(max(1, (1 << 27) // m)):
        a, b, c, d = _rows(D, rows)
        y[rows] += a @ x[:m] + b @ x[m:]
        y[rows + m] += c @ x[:m] + d @ x[m:]
        del a, b, c, d
    return y


def _solution(D, g):
    """GMRES to 1e-14 on the assembled matrix, the columns scaled by the diagonal of Eq. (2.30)."""
    m = D["W"].numel()
    A = torch.empty(2 * m, 2 * m, dtype=torch.float64, device="cuda")
    for rows in torch.arange(m, device="cuda").split(max(1, (1 << 27) // m)):
        lo, hi = int(rows[0]), int(rows[-1]) + 1
        A[lo:hi, :m], A[lo:hi, m:], A[m + lo:m + hi, :m], A[m + lo:m + hi, m:] = _rows(D, rows)
    lam = torch.cat([torch.full((m,), v, dtype=torch.float64, device="cuda") for v in LAM])
    x, r = torch.zeros_like(g), g.clone()
    for _ in range(4):
        beta = r.norm()
        V, H = [r / beta], np.zeros((61, 60))
        for j in range(60):
            z = V[j] / lam
            w = A @ z + lam * z + _correction(D, z)
            B = torch.stack(V)
            for _ in range(2):
                c = B @ w
                w = w - c @ B
                H[:j + 1, j] += c.cpu().numpy()
            H[j + 1, j] = float(w.norm())
            V.append(w / H[j + 1, j])
            rhs = np.zeros(j + 2)
            rhs[0] = float(beta)
            y, res = np.linalg.lstsq(H[:j + 2, :j + 1], rhs, rcond=None)[:2]
            if res.size and math.sqrt(float(res[0])) < 1e-9 * float(beta):
                break
        x = x + (torch.tensor(y, device="cuda") @ torch.stack(V[:j + 1])) / lam
        r = g - (A @ x + lam * x + _correction(D, x))
        if float(r.norm()) < 1e-14 * float(g.norm()):
            break
    return {"psi": x[:m].clone(), "dpsi": x[m:].clone()}


def _potential(D, psi, dpsi, points):
    """psi_rxn (Eq. (2.31)) at the points."""
    a, b = (D["h"] ** 3 * D["W"] / (4.0 * math.pi) * v for v in (psi, dpsi))
    out = []
    for z in points.split(max(1, (1 << 27) // a.numel())):
        d = [z[:, c, None] - D["P"][None, :, c] for c in range(3)]
        r2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2]
        dn = d[0] * D["n"][:, 0] + d[1] * D["n"][:, 1] + d[2] * D["n"][:, 2]
        ri = r2.rsqrt()
        kr = KAPPA * r2 * ri
        out.append((dn * ri / r2 * (RATIO * torch.exp(-kr) * (1.0 + kr) - 1.0)) @ a - (torch.expm1(-kr) * ri) @ b)
    return torch.cat(out)


def exact(case, seed):
    do = case["do"]
    if do == "batch":
        out = []
        for k, size in enumerate(_member_sizes(case)):
            args, c = _inputs(case, seed + 1000 * k, size)
            D = _discretize(c["surface"], c["size"], c["h"], False)
            out.append(_solution(D, _coulomb(D, args[7], args[8])))
        return out
    if do == "step" and work(case)["flops"] > APPLICATIONS * PAIR_FLOPS * 5e4 ** 2:
        return None   # the assembled matrix of a large system does not fit, and applying it takes seconds
    args, _ = _inputs(case, seed)
    D = _discretize(case["surface"], case["size"], case["h"], bool(case.get("kreg")))
    g = _coulomb(D, args[7], args[8])
    if do == "matvec":
        return _apply(D, _density(seed, g))
    if do in ("map", "energy"):
        psi, dpsi = _field(case, seed, g)
        points = _points(case, seed) if do == "map" else torch.tensor(args[7], device="cuda")
        v = _potential(D, psi, dpsi, points)
        return v if do == "map" else {"energy": 0.5 * float(v @ torch.tensor(args[8], device="cuda")), "at_charges": v}
    out = _solution(D, g)
    if do == "step":
        v = _potential(D, out["psi"], out["dpsi"], torch.tensor(args[7], device="cuda"))
        out = dict(out, energy=0.5 * float(v @ torch.tensor(args[8], device="cuda")), at_charges=v)
    return out
