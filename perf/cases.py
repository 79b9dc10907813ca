"""Performance cases of the docking path: what a program that uses the library has it do, through the
public entry points of ``paper_2506_20043_gb300.api``.

Kinds of case
  score    SF (Eq. 3) of given poses with the tangent gradient (``Context.score``)
  pose     SF and its vector-Jacobian product over pose parameters (``PVScore``, torch.autograd)
  xyz      the same over posed atom coordinates (``PVScoreXYZ``)
  grids    the grid maps of receptors' pocket boxes (``build_grids``, ``append``, ``pack``)
  pockets  SAS points, Eq. 1 features and ranked clusters of receptors (``surfaces``, ``features``,
           ``cluster_many``)
  dock     the Monte-Carlo search of ligands over pockets with selection and merge (``dock``)

``prepare`` makes a case's inputs from its seed (synthetic receptors at protein-like density with
carved pockets, torsion-tree ligands, uniform random poses) and the handles a program keeps: the
context, grid sets and ligands. ``exact`` restates the outputs in 64 bits with plain torch.
"""
import math
import types

import numpy as np
import torch

from paper_2506_20043_gb300 import api

DENSITY = 0.05                       # receptor heavy atoms per cubic Angstrom
SPACING = 0.375                      # grid spacing, A
RADIUS = (1.9, 1.8, 1.7, 2.0)        # XS radii of C, N, O, S
VDW = (1.70, 1.55, 1.52, 1.80)       # Bondi radii of C, N, O, S
PROBE, N_SPHERE = 1.6, 100


def listed():
    return [
        # one gradient call on a handful of poses, as an interactive refinement loop makes it
        dict(name="score_call", kind="score", poses=64, atoms=20, torsions=4, receptor=2000, box=20.0, packed=False,
             parts=False),
        # rescoring a whole pose library in one call, the maps in both layouts
        dict(name="score_batch", kind="score", poses=65536, atoms=32, torsions=8, receptor=4000, box=24.0, packed=True,
             parts=True),
        # gradient-based refinement under torch.autograd of a large, flexible ligand (two atoms per lane)
        dict(name="pose_autograd", kind="pose", poses=8191, atoms=47, torsions=11, receptor=4000, box=22.5, packed=False),
        # a generative model's coordinates scored and differentiated; a small ligand
        dict(name="xyz_autograd", kind="xyz", poses=20011, atoms=17, torsions=3, receptor=3000, box=24.0, packed=True),
        # the maps of one pocket of a small receptor held on the host, for one ligand's atom types
        dict(name="grids_one", kind="grids", receptors=1, atoms_lo=2000, atoms_hi=2000, boxes=1, box_lo=20.0, box_hi=20.0,
             n_types=6, packed=False, host=True),
        # a site set up for multi-pocket docking: ten boxes, both layouts, then a first batch of poses
        dict(name="grids_ten", kind="grids", receptors=1, atoms_lo=5000, atoms_hi=5000, boxes=10, box_lo=24.0, box_hi=24.0,
             n_types=8, packed=True, host=False),
        # a screening set: receptors of many sizes appended to one set, boxes of every size, all atom types
        dict(name="grids_screen", kind="grids", receptors=4, atoms_lo=1500, atoms_hi=8000, boxes=3, box_lo=15.0,
             box_hi=30.0, n_types=11, packed=False, host=True),
        # pocket prediction of one small receptor from host arrays
        dict(name="pockets_one", kind="pockets", receptors=1, atoms_lo=1500, atoms_hi=1500, props=7, host=True),
        # pocket prediction of a batch of receptors resident on the device
        dict(name="pockets_batch", kind="pockets", receptors=7, atoms_lo=3000, atoms_hi=8000, props=7, host=False),
        # one ligand into one pocket with few chains: the latency of a chain
        dict(name="dock_one", kind="dock", receptor=2000, pockets=1, box=20.0, ligands=1, atoms_lo=20, atoms_hi=20,
             tors_lo=4, tors_hi=4, chains=8, steps=100, packed=False, focc=0, rescore=False),
        # one drug-like ligand over ten pockets with many chains, the GPU full
        dict(name="dock_pockets", kind="dock", receptor=5000, pockets=10, box=24.0, ligands=1, atoms_lo=30, atoms_hi=30,
             tors_lo=6, tors_hi=6, chains=1000, steps=100, packed=True, focc=0, rescore=False),
        # uneven ligands over five pockets in one launch, kept poses rescored
        dict(name="dock_uneven", kind="dock", receptor=6000, pockets=5, box=24.0, ligands=24, atoms_lo=10, atoms_hi=60,
             tors_lo=0, tors_hi=15, chains=64, steps=60, packed=True, focc=0, rescore=True),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["score", "pose", "xyz", "grids", "grids", "pockets", "pockets", "dock", "dock"])
    box = round(rng.uniform(15.0, 30.0), 2)
    packed = rng.random() < 0.5
    if kind in ("score", "pose", "xyz"):
        atoms = rng.randint(8, 60)
        c = dict(kind=kind, poses=_log(rng, 64, 65536 * 20 // (atoms + 20)), atoms=atoms, torsions=rng.randint(0, atoms // 3 if atoms < 45 else 15),
                 receptor=_log(rng, 1500, 8000), box=box, packed=packed)
        if kind == "score":
            c["parts"] = rng.random() < 0.5
        return c
    if kind == "grids":
        receptors, boxes = rng.choice([(1, 1), (1, 5), (1, 10), (2, 3), (4, 3)])
        lo = round(rng.uniform(15.0, 24.0), 2)
        return dict(kind=kind, receptors=receptors, atoms_lo=_log(rng, 1500, 4000), atoms_hi=_log(rng, 4000, 8000),
                    boxes=boxes, box_lo=lo, box_hi=round(rng.uniform(lo, 24.0), 2), n_types=rng.randint(3, 8),
                    packed=packed, host=rng.random() < 0.5)
    if kind == "pockets":
        return dict(kind=kind, receptors=rng.randint(1, 7), atoms_lo=_log(rng, 1500, 4000), atoms_hi=_log(rng, 4000, 8000),
                    props=rng.choice([1, 7, 7, 20]), host=rng.random() < 0.5)
    ligands = rng.choice([1, 1, 3, 10])
    lo = rng.choice([10, 17, 24, 30])
    tors = rng.randint(0, 6)
    pockets = rng.randint(1, 5)
    return dict(kind=kind, receptor=_log(rng, 2000, 8000), pockets=pockets, box=box, ligands=ligands, atoms_lo=lo,
                atoms_hi=rng.randint(lo, lo + 10), tors_lo=tors, tors_hi=rng.randint(tors, 8),
                chains=_log(rng, 8, 4000 // (ligands * pockets)), steps=rng.randint(20, 60), packed=packed,
                focc=rng.choice([0, 0, 4]), rescore=rng.random() < 0.5)


# ------------------------------------------------------------------------------------- inputs --

def _flags(rng, element):
    polar = (element == 1) | (element == 2)
    return [(polar & (rng.random(element.shape[0]) < 0.3)).astype(np.uint8) for _ in range(2)]


def _receptor(rng, n, pockets):
    """n heavy atoms at DENSITY in a cube with `pockets` spheres of 6-10 A left empty; their centres."""
    side = (n / DENSITY) ** (1.0 / 3.0)
    radii = rng.uniform(6.0, 10.0, pockets)
    half = side / 2.0 - min(6.0, side / 4.0)
    centers = rng.uniform(-half, half, (pockets, 3))
    for i in range(1, pockets):                       # apart where a few hundred trials find room
        for _ in range(300):
            if (np.linalg.norm(centers[:i] - centers[i], axis=1) > radii[:i] + radii[i]).all():
                break
            centers[i] = rng.uniform(-half, half, 3)
    xyz = np.zeros((0, 3))
    while xyz.shape[0] < n:
        more = rng.uniform(-side / 2, side / 2, (2 * n, 3))
        d = np.linalg.norm(more[:, None] - centers[None], axis=2)
        xyz = np.concatenate([xyz, more[(d >= radii).all(axis=1)]])
    element = rng.choice(4, size=n, p=(0.62, 0.17, 0.19, 0.02)).astype(np.uint8)
    donor, acceptor = _flags(rng, element)
    rec = types.SimpleNamespace(xyz=xyz[:n].astype(np.float32), element=element, donor=donor, acceptor=acceptor)
    return rec, centers.astype(np.float32)


def _on_device(rec):
    return types.SimpleNamespace(**{k: torch.as_tensor(v).cuda() for k, v in vars(rec).items()})


def _ligand(rng, n, n_rot):
    """A heavy-atom tree grown atom by atom (1.5 A bonds, 109.5 degrees, valences, no clashes) with
    n_rot rotatable bonds (at most one per three atoms) among the non-terminal ones, centred."""
    ang, n_rot = math.radians(109.5), min(n_rot, n // 3)
    while True:
        element = rng.choice(3, size=n, p=(0.70, 0.15, 0.15)).astype(np.uint8)
        element[0] = 0
        valence = np.array((4, 3, 2))[element]
        xyz, nbrs, bonds = np.zeros((n, 3)), [[] for _ in range(n)], []
        for k in range(1, n):
            for _ in range(200):
                free = [a for a in range(k) if len(nbrs[a]) < valence[a]]
                if not free:
                    break
                p = int(rng.choice(free))
                v = rng.normal(size=3)
                if nbrs[p]:
                    u = xyz[nbrs[p][0]] - xyz[p]
                    u /= np.linalg.norm(u)
                    v -= v.dot(u) * u
                    v = math.cos(ang) * u + math.sin(ang) * v / np.linalg.norm(v)
                pos = xyz[p] + 1.5 * v / np.linalg.norm(v)
                d = np.linalg.norm(xyz[:k] - pos, axis=1)
                limit = np.full(k, 2.5)
                limit[nbrs[p]] = 2.3
                limit[p] = 0.0
                if (d >= limit).all():
                    break
            else:
                break
            if not free:
                break
            xyz[k] = pos
            nbrs[p].append(k)
            nbrs[k].append(p)
            bonds.append((p, k))
        inner = [i for i, (a, b) in enumerate(bonds) if len(nbrs[a]) > 1 and len(nbrs[b]) > 1]
        if len(bonds) == n - 1 and len(inner) >= n_rot:
            break
    rotatable = np.zeros(len(bonds), np.uint8)
    rotatable[rng.permutation(inner)[:n_rot].astype(int)] = 1
    donor, acceptor = _flags(rng, element)
    return types.SimpleNamespace(xyz=(xyz - xyz.mean(axis=0)).astype(np.float32), element=element, donor=donor,
                                 acceptor=acceptor, bonds=np.array(bonds, np.int32).reshape(-1, 2), rotatable=rotatable)


def _poses(rng, n, center, size, n_rot):
    """n POT vectors: translation uniform in the box, uniform quaternions (Shoemake), uniform torsions."""
    t = center + (rng.random((n, 3)) - 0.5) * size
    u1, u2, u3 = rng.random((3, n))
    q = np.stack([np.sqrt(1 - u1) * np.sin(2 * np.pi * u2), np.sqrt(1 - u1) * np.cos(2 * np.pi * u2),
                  np.sqrt(u1) * np.sin(2 * np.pi * u3), np.sqrt(u1) * np.cos(2 * np.pi * u3)], axis=1)
    return np.concatenate([t, q, rng.uniform(-np.pi, np.pi, (n, n_rot))], axis=1).astype(np.float32)


def _box(center, size):
    return (tuple(float(v) for v in center), (float(np.float32(size)),) * 3, SPACING)


def _spread(lo, hi, n):
    """n sizes over [lo, hi], evenly over their logarithm (the middle one for n = 1)."""
    at = np.linspace(0.0, 1.0, n) if n > 1 else np.array([0.5])
    return np.exp(math.log(lo) + at * math.log(hi / lo))


def _types(n):
    """n ligand XS types in the order ligands need them: the carbons, plain and flagged N and O, S."""
    return sorted((0, 1, 2, 6, 3, 8, 4, 7, 5, 9, 10)[:n])


def _inputs(case, seed):
    """Host inputs of a case, made from the seed alone (numpy and plain values)."""
    rng = np.random.default_rng(seed)
    kind, s = case["kind"], types.SimpleNamespace()
    if kind in ("score", "pose", "xyz"):
        s.rec, centers = _receptor(rng, case["receptor"], 1)
        s.box = _box(centers[0], case["box"])
        s.lig = _ligand(rng, case["atoms"], case["torsions"])
        s.poses = _poses(rng, case["poses"], centers[0], case["box"], int(s.lig.rotatable.sum()))
        s.weight = rng.normal(size=case["poses"]).astype(np.float32)
    elif kind == "grids":
        s.sites = []
        sizes = _spread(case["box_lo"], case["box_hi"], case["receptors"] * case["boxes"]).reshape(case["boxes"], -1)
        for i, n in enumerate(_spread(case["atoms_lo"], case["atoms_hi"], case["receptors"])):
            rec, centers = _receptor(rng, int(round(n)), case["boxes"])
            s.sites.append((rec, [_box(c, b) for c, b in zip(centers, sizes[:, i])]))
        s.types = _types(case["n_types"])
        s.lig = _ligand(rng, 20, 4)
        s.lig.element[:], s.lig.donor[:], s.lig.acceptor[:] = 0, 0, 0        # carbons: every set holds their maps
        first = s.sites[0][1][0]
        s.poses = _poses(rng, 1024, np.array(first[0]), first[1][0], int(s.lig.rotatable.sum()))
    elif kind == "pockets":
        s.recs, s.props = [], []
        for n in _spread(case["atoms_lo"], case["atoms_hi"], case["receptors"]):
            # the structure is the case's (its surface has as many points for every seed); the seed gives
            # the order of its atoms and their properties
            rec, _ = _receptor(np.random.default_rng(int(n)), int(round(n)), 4)
            order = rng.permutation(rec.xyz.shape[0])
            rec = types.SimpleNamespace(**{k: v[order] for k, v in vars(rec).items()})
            props = rng.uniform(-0.5, 0.5, (rec.xyz.shape[0], case["props"])).astype(np.float32)
            props[:, :4] = np.eye(4, dtype=np.float32)[rec.element][:, :case["props"]]
            s.recs.append(rec)
            s.props.append(props)
    else:
        s.rec, centers = _receptor(rng, case["receptor"], case["pockets"])
        s.boxes = [_box(c, case["box"]) for c in centers]
        n_lig = case["ligands"]
        shape = np.random.default_rng(n_lig)             # the ligands' sizes are the case's
        s.ligs = [_ligand(rng, int(a), int(t)) for a, t in zip(shape.integers(case["atoms_lo"], case["atoms_hi"] + 1, n_lig),
                                                               shape.integers(case["tors_lo"], case["tors_hi"] + 1, n_lig))]
        s.seed = int(rng.integers(1 << 30))
    return s


_CTX = None


def _context():
    """The one library context of the program."""
    global _CTX
    if _CTX is None:
        _CTX = api.Context(0)
    return _CTX


class _Maps:
    """The maps of one pocket, [type][z][y][x] in the library's memory, lent to torch without a copy."""

    def __init__(self, grids, pocket, types_):
        dims, _, _, ptr = grids.geometry(pocket, types_[0])
        self.grids = grids
        self.__cuda_array_interface__ = {"shape": (len(types_), int(dims[2]), int(dims[1]), int(dims[0])),
                                         "typestr": "<f4", "data": (ptr, False), "version": 2, "strides": None}


def prepare(case, seed):
    s = _inputs(case, seed)
    s.kind, s.case, s.ctx = case["kind"], case, _context()
    if s.kind in ("score", "pose", "xyz"):
        s.plig = s.ctx.ligand(s.lig)
        s.grids = s.ctx.build_grids(s.rec, [s.box], sorted(set(s.plig.xs_types.tolist())))
        if case["packed"]:
            s.grids.pack()
        if s.kind == "xyz":
            with torch.no_grad():
                x = _fk(s.lig, torch.as_tensor(s.poses, dtype=torch.float64)).float()
            s.x = x.cuda().requires_grad_()
        else:
            s.x = torch.as_tensor(s.poses).cuda().requires_grad_(s.kind == "pose")
        s.w = torch.as_tensor(s.weight).cuda()
    elif s.kind == "grids":
        s.plig = s.ctx.ligand(s.lig)
        s.x = torch.as_tensor(s.poses).cuda()
        if not case["host"]:
            s.sites = [(_on_device(r), b) for r, b in s.sites]
    elif s.kind == "pockets":
        if not case["host"]:
            s.recs = [_on_device(r) for r in s.recs]
            s.props = [torch.as_tensor(p).cuda() for p in s.props]
    else:
        s.pligs = [s.ctx.ligand(lig) for lig in s.ligs]
        s.grids = s.ctx.build_grids(s.rec, s.boxes, sorted(set(t for p in s.pligs for t in p.xs_types.tolist())))
        if case["packed"]:
            s.grids.pack()
        s.params = api.DockParams(chains=case["chains"], steps=case["steps"], seed=s.seed, focc=case["focc"],
                                  rescore=case["rescore"])
    return s


def _cavity_score(protrusion):
    """A point's score from its protrusion count (buried points score high); stands for the classifier."""
    return ((protrusion.float() - 60.0) / 120.0).clamp_(0.0, 1.0)


def run(s):
    c = s.case
    if s.kind == "score":
        return [v for v in s.ctx.score(s.grids, s.plig, 0, s.x, grad=True, parts=c["parts"]) if v is not None]
    if s.kind in ("pose", "xyz"):
        f = api.PVScore if s.kind == "pose" else api.PVScoreXYZ
        e = f.apply(s.x, s.ctx, s.grids, s.plig, 0)
        return [e.detach(), torch.autograd.grad(e, s.x, s.w)[0]]
    if s.kind == "grids":
        (rec, boxes), more = s.sites[0], s.sites[1:]
        g = s.ctx.build_grids(rec, boxes, s.types)
        for r, b in more:
            g.append(r, b)
        out = {}
        if c["packed"]:
            g.pack()
            out["score"] = s.ctx.score(g, s.plig, 0, s.x)[:2]
        out["maps"] = [torch.as_tensor(_Maps(g, p, s.types), device="cuda") for p in range(len(s.sites) * c["boxes"])]
        return out
    if s.kind == "pockets":
        surfaces = s.ctx.surfaces(s.recs) if len(s.recs) > 1 else [s.ctx.surface(s.recs[0])]
        feats = [x.features(p) for x, p in zip(surfaces, s.props)]
        sets = [(x, _cavity_score(f[1])) for x, f in zip(surfaces, feats)]
        clusters = s.ctx.cluster_many(sets)
        return [dict(points=x.points(), features=f[0], protrusion=f[1], **k.read()) for x, f, k in zip(surfaces, feats, clusters)]
    r = s.ctx.dock(s.grids, s.pligs, list(range(c["pockets"])), s.params)
    p, best = r.poses, np.full((c["ligands"], c["pockets"] * r.top_k), -1)
    for i in range(c["ligands"]):
        rank = r.ranking(i)
        best[i, :len(rank)] = rank
    return dict({k: p[k].copy() for k in ("score", "e_inter", "e_intra", "affinity", "chain")}, kept=r.n_kept, pots=r.pots,
                xyz=r.xyz, ranking=best)


# --------------------------------------------------------------------------------------- work --

def _eval_flops(atoms, torsions):
    """Operations of one score + gradient evaluation (an FMA counts 2): per torsion, per atom, per intra
    pair (about three quarters of the atom pairs of a flexible ligand), per atom moved by a torsion."""
    pairs = 0.375 * atoms * atoms * torsions / (torsions + 1.0)
    return 40.0 + 120.0 * torsions + 83.0 * atoms + 45.0 * pairs + 15.0 * torsions * atoms * 0.4


def work(case):
    kind = case["kind"]
    nodes = lambda size: (math.ceil(size / SPACING) + 1.0) ** 3  # noqa: E731
    if kind in ("score", "pose", "xyz"):
        n, a, t = case["poses"], case["atoms"], case["torsions"]
        inp = 3 * a if kind == "xyz" else 7 + t
        out = 1 + inp if kind != "score" else 1 + 6 + t + (2 if case["parts"] else 0)
        maps = min(32.0 * a * n, 4.0 * min(6, a) * nodes(case["box"]))
        return {"bytes": 4.0 * n * (inp + out) + maps, "flops": n * _eval_flops(a, t)}
    if kind == "grids":
        n_box = case["receptors"] * case["boxes"]
        atoms = case["receptors"] * 0.5 * (case["atoms_lo"] + case["atoms_hi"])
        n = n_box * 0.5 * (nodes(case["box_lo"]) + nodes(case["box_hi"]))
        # written once (and once more in cells of eight corners); 107 receptor atoms within 8 A of a
        # node, 18 operations per element class of the types
        copies = 1.0 + (8.0 if case["packed"] else 0.0)
        return {"bytes": 15.0 * atoms + 4.0 * n * case["n_types"] * copies, "flops": n * 107.0 * 18.0 * min(4, case["n_types"])}
    if kind == "pockets":
        atoms = case["receptors"] * 0.5 * (case["atoms_lo"] + case["atoms_hi"])
        points = 2.85 * atoms          # kept SAS points per atom at this density
        byts = atoms * (13.0 + 4.0 * case["props"]) + points * (12.0 + 4.0 + 4.0 + 4.0 * case["props"])
        # lattice points against a handful of neighbouring spheres, points against the atoms in reach
        return {"bytes": byts, "flops": atoms * N_SPHERE * 10.0 * 8.0 + points * (110.0 * 8.0 + 25.0 * (4.0 + 2.0 * case["props"]))}
    pairs = case["ligands"] * case["pockets"]
    a, t = 0.5 * (case["atoms_lo"] + case["atoms_hi"]), 0.5 * (case["tors_lo"] + case["tors_hi"])
    # a Monte-Carlo step's local search takes about 40 evaluations
    evals = 40.0 * pairs * case["chains"] * case["steps"]
    byts = case["pockets"] * 4.0 * min(8, a) * nodes(case["box"]) + pairs * case["chains"] * 4.0 * (7 + t)
    return {"bytes": byts, "flops": evals * _eval_flops(a, t)}


# -------------------------------------------------------------------- the outputs in 64 bits --

DEV = "cuda" if torch.cuda.is_available() else "cpu"


def _f64(a):
    return torch.as_tensor(np.asarray(a), dtype=torch.float64, device=DEV)


def _xs(element, donor, acceptor, polar_c):
    e, h = element.astype(int), donor.astype(int) + 2 * acceptor.astype(int)
    return np.where(e == 0, polar_c.astype(int), np.where(e == 1, 2 + h, np.where(e == 2, 6 + h, 10)))


def _xs_receptor(rec):
    x, hetero = _f64(rec.xyz), torch.as_tensor((rec.element == 1) | (rec.element == 2), device=DEV)
    near = torch.cat([((c[:, None] - x[None]).square().sum(2) < 1.75 ** 2) & hetero[None] for c in x.split(512)]).any(1)
    return _xs(rec.element, rec.donor, rec.acceptor, near.cpu().numpy())


def _xs_ligand(lig):
    polar = np.zeros(lig.xyz.shape[0], bool)
    for a, b in lig.bonds:
        polar[a] |= lig.element[b] in (1, 2)
        polar[b] |= lig.element[a] in (1, 2)
    return _xs(lig.element, lig.donor, lig.acceptor, polar)


def _donor(t):
    return (t == 3) | (t == 5) | (t == 7) | (t == 9)


def _acceptor(t):
    return (t == 4) | (t == 5) | (t == 8) | (t == 9)


def _element_radius(t):
    t = np.asarray(t)
    return np.array(RADIUS)[np.where(t <= 1, 0, np.where(t <= 5, 1, np.where(t <= 9, 2, 3)))]


def _terms(d):
    """(steric, hydrophobic, hydrogen-bond) terms of surface distance d (AutoDock Vina's weights)."""
    steric = -0.0356 * torch.exp(-(2.0 * d).square()) - 0.00516 * torch.exp(-(0.5 * (d - 3.0)).square()) + \
        0.840 * d.clamp(max=0.0).square()
    return steric, -0.0351 * (1.5 - d).clamp(0.0, 1.0), -0.587 * (-d / 0.7).clamp(0.0, 1.0)


def _maps64(rec, box, types_):
    """[type][z][y][x] direct sums over the receptor atoms within 8 A, tile by tile."""
    center, size, sp = box
    org = [float(np.float32(float(np.float32(center[k])) - 0.5 * size[k])) for k in range(3)]
    nd = [int(math.ceil(size[k] / sp - 1e-9)) + 1 for k in range(3)]
    xs = _xs_receptor(rec)
    x, rad = _f64(rec.xyz), _f64(_element_radius(xs))
    hyd, don, acc = (torch.as_tensor(v, device=DEV) for v in (xs == 0, _donor(xs), _acceptor(xs)))
    ax = [org[k] + sp * torch.arange(nd[k], dtype=torch.float64, device=DEV) for k in range(3)]
    out = torch.zeros([len(types_)] + nd[::-1], dtype=torch.float64, device=DEV)
    step = 16
    for z in range(0, nd[2], step):
        for y in range(0, nd[1], step):
            for w in range(0, nd[0], step):
                n = [ax[0][w:w + step], ax[1][y:y + step], ax[2][z:z + step]]
                lo, hi = torch.stack([v[0] for v in n]), torch.stack([v[-1] for v in n])
                at = ((x.clamp(lo, hi) - x).square().sum(1) < 64.0).nonzero()[:, 0]
                if at.numel() == 0:
                    continue
                p = torch.stack(torch.meshgrid(n[2], n[1], n[0], indexing="ij"), -1).flip(-1).reshape(-1, 1, 3)
                r2 = (p - x[at]).square().sum(2)
                r, near = r2.sqrt(), r2 < 64.0
                for el in range(4):
                    mine = [i for i, t in enumerate(types_) if _element_radius(t) == RADIUS[el]]
                    if not mine:
                        continue
                    st, hy, hb = _terms(r - RADIUS[el] - rad[at])
                    st, hy, hb = st * near, hy * near, hb * near
                    base = st.sum(1)
                    for i in mine:
                        t, v = types_[i], base
                        if t == 0:
                            v = v + (hy * hyd[at]).sum(1)
                        pairs = (acc[at] if _donor(t) else torch.zeros_like(hyd[at])) | \
                            (don[at] if _acceptor(t) else torch.zeros_like(hyd[at]))
                        v = v + (hb * pairs).sum(1)
                        out[i, z:z + step, y:y + step, w:w + step] = v.reshape(len(n[2]), len(n[1]), len(n[0]))
    return out, org, nd


def _tree(lig):
    """(fragment of each atom, origin atom, bond distances, per torsion (near, far, far-side atoms)), the
    torsions in the order of the rotatable bonds."""
    n = lig.xyz.shape[0]
    nbrs = [[] for _ in range(n)]
    for i, (a, b) in enumerate(lig.bonds):
        nbrs[a].append((int(b), i))
        nbrs[b].append((int(a), i))

    def reach(a, skip):
        seen, todo = {a}, [a]
        while todo:
            for b, i in nbrs[todo.pop()]:
                if not skip(i) and b not in seen:
                    seen.add(b)
                    todo.append(b)
        return seen

    frag, sizes = np.full(n, -1), []
    for a in range(n):
        if frag[a] < 0:
            f = sorted(reach(a, lambda i: lig.rotatable[i]))
            frag[f] = len(sizes)
            sizes.append(len(f))
    origin = int(np.flatnonzero(frag == int(np.argmax(sizes)))[0])
    dist = np.full((n, n), 99)
    for a in range(n):
        dist[a, a], todo = 0, [a]
        while todo:
            b = todo.pop(0)
            for c, _ in nbrs[b]:
                if dist[a, c] == 99:
                    dist[a, c] = dist[a, b] + 1
                    todo.append(c)
    tors = []
    for i in np.flatnonzero(lig.rotatable):
        a, b = (int(v) for v in lig.bonds[i])
        side = reach(b, lambda j, i=i: j == i)
        if origin in side:
            a, b, side = b, a, reach(a, lambda j, i=i: j == i)
        tors.append((a, b, sorted(side)))
    return frag, origin, dist, tors


def _fk(lig, pose):
    """Atom coordinates of POT vectors: torsions from the leaves up, then rotation and translation."""
    _, origin, _, tors = _tree(lig)
    x0 = torch.as_tensor(lig.xyz, dtype=torch.float64, device=pose.device)
    y = x0.expand(pose.shape[0], -1, -1).clone()
    for k in sorted(range(len(tors)), key=lambda k: len(tors[k][2])):       # a subtree before its parents
        a, b, side = tors[k]
        u = (x0[b] - x0[a]) / (x0[b] - x0[a]).norm()
        v = y[:, side] - x0[b]
        c, s = torch.cos(pose[:, 7 + k])[:, None, None], torch.sin(pose[:, 7 + k])[:, None, None]
        turned = v * c + torch.cross(u.expand_as(v), v, dim=2) * s + u * (v @ u)[..., None] * (1.0 - c)
        y = y.index_copy(1, torch.tensor(side, device=pose.device), turned + x0[b])
    q = pose[:, 3:7] / pose[:, 3:7].norm(dim=1, keepdim=True)
    w, u = q[:, :1, None], q[:, None, 1:].expand(-1, y.shape[1], -1)
    v = y - x0[origin]
    t = 2.0 * torch.cross(u, v, dim=2)
    return pose[:, None, :3] + v + w * t + torch.cross(u, t, dim=2)


def _energy(lig, maps, org, nd, types_, x):
    """(e_inter, e_intra) of posed atoms x [n, atoms, 3] (differentiable in x)."""
    xs = _xs_ligand(lig)
    slot = torch.tensor([list(types_).index(t) for t in xs], device=DEV)
    g = (x - _f64(org)) / SPACING
    hi = _f64([d - 1.0 for d in nd])
    gc = torch.minimum(g.clamp(min=0.0), hi)
    cell = torch.minimum(gc.detach().floor(), hi - 1.0).long()
    f = gc - cell
    val = 0.0
    flat = maps.reshape(-1)
    for c in range(8):
        o = [c & 1, (c >> 1) & 1, c >> 2]
        at = ((slot * nd[2] + cell[..., 2] + o[2]) * nd[1] + cell[..., 1] + o[1]) * nd[0] + cell[..., 0] + o[0]
        wt = 1.0
        for k in range(3):
            wt = wt * (f[..., k] if o[k] else 1.0 - f[..., k])
        val = val + wt * flat[at]
    out2 = ((g - gc) * SPACING).square().sum(2)
    far = out2 > 0.0
    val = val + 10.0 * torch.where(far, torch.where(far, out2, torch.ones_like(out2)).sqrt(), torch.zeros_like(out2))
    frag, _, dist, _ = _tree(lig)
    i, j = np.nonzero(np.triu((frag[:, None] != frag[None]) & (dist > 3), 1))
    if len(i) == 0:
        return val.sum(1), torch.zeros_like(val[:, 0])
    rad = _element_radius(xs)
    r2 = (x[:, i] - x[:, j]).square().sum(2)
    st, hy, hb = _terms(r2.clamp(min=1e-12).sqrt() - _f64(rad[i] + rad[j]))
    e = st + hy * torch.as_tensor((xs[i] == 0) & (xs[j] == 0), device=DEV) + \
        hb * torch.as_tensor((_donor(xs[i]) & _acceptor(xs[j])) | (_acceptor(xs[i]) & _donor(xs[j])), device=DEV)
    return val.sum(1), (e * (r2 < 64.0)).sum(1)


def _tangent(lig, pose, x, g):
    """dSF/d(translation, rotation vector about the origin atom, torsions) from dSF/dx."""
    _, origin, _, tors = _tree(lig)
    cols = [g.sum(1), torch.cross(x - x[:, origin:origin + 1], g, dim=2).sum(1)]
    for a, b, side in tors:
        u = x[:, b] - x[:, a]
        u = u / u.norm(dim=1, keepdim=True)
        t = torch.cross(x[:, side] - x[:, b:b + 1], g[:, side], dim=2).sum(1)
        cols.append((t * u).sum(1, keepdim=True))
    return torch.cat(cols, 1)


def _score64(lig, maps, types_, poses):
    out = []
    for p in poses.split(8192):
        x = _fk(lig, p).requires_grad_()
        ei, ej = _energy(lig, *maps, types_, x)
        g = torch.autograd.grad((ei + ej).sum(), x)[0]
        out.append((ei.detach() + ej.detach(), _tangent(lig, p, x.detach(), g), torch.stack([ei.detach(), ej.detach()], 1)))
    return [torch.cat(v) for v in zip(*out)]


def _pockets64(rec, props):
    """Kept SAS points and Eq. 1 sums of one receptor."""
    x = _f64(rec.xyz)
    a = _f64(np.float32(VDW))[torch.as_tensor(rec.element, device=DEV).long()] + float(np.float32(PROBE))
    k = np.arange(N_SPHERE)
    z = 1.0 - (2.0 * k + 1.0) / N_SPHERE
    rho, phi = np.sqrt(1.0 - z * z), k * math.pi * (3.0 - math.sqrt(5.0))
    dirs = _f64(np.stack([rho * np.cos(phi), rho * np.sin(phi), z], 1))
    p = x[:, None] + a[:, None, None] * dirs
    pts = []
    for i in torch.arange(x.shape[0], device=DEV).split(64):
        d2 = (p[i, :, None, :] - x).square().sum(3)
        inside = d2 < a.square()
        inside[torch.arange(len(i), device=DEV), :, i] = False
        pts.append(p[i][~inside.any(2)])
    pts = torch.cat(pts)
    w = _f64(props)
    feat = torch.cat([(1.0 - torch.cdist(c, x, compute_mode="donot_use_mm_for_euclid_dist") / 6.0).clamp(min=0.0) @ w
                      for c in pts.split(4096)])
    return dict(points=pts, features=feat)


def exact(case, seed):
    kind = case["kind"]
    if kind == "dock":
        return None                    # a chaotic search: no such value
    s = _inputs(case, seed)
    if kind == "pockets":
        none = dict.fromkeys(("protrusion", "cluster", "score", "center", "size", "first"))
        return [dict(_pockets64(r, p), **none) for r, p in zip(s.recs, s.props)]
    if kind == "grids":
        out = {}
        every = [_maps64(r, b, s.types) for r, bs in s.sites for b in bs]
        if case["packed"]:
            out["score"] = _score64(s.lig, every[0], s.types, _f64(s.poses))[:2]
        out["maps"] = [m[0] for m in every]
        return out
    types_ = sorted(set(_xs_ligand(s.lig).tolist()))
    maps = _maps64(s.rec, s.box, types_)
    if kind == "score":
        return _score64(s.lig, maps, types_, _f64(s.poses))[:3 if case["parts"] else 2]
    poses, energy, grad = _f64(s.poses), [], []
    if kind == "xyz":
        with torch.no_grad():
            poses = _fk(s.lig, torch.as_tensor(s.poses, dtype=torch.float64)).float().double().to(DEV)
    for v, w in zip(poses.split(8192), _f64(s.weight).split(8192)):
        v = v.clone().requires_grad_()
        ei, ej = _energy(s.lig, *maps, types_, v if kind == "xyz" else _fk(s.lig, v))
        grad.append(torch.autograd.grad(((ei + ej) * w).sum(), v)[0])
        energy.append((ei + ej).detach())
    return [torch.cat(energy), torch.cat(grad)]
