"""Performance cases of the docking library, through its public calls.

A case is one call (or one short chain of calls) that a docking program
makes, on seeded synthetic receptors, ligands and poses of the sizes of this
repository's workloads (synth.WORKLOADS): ligands of 10 to 256 atoms, up to
40 torsions, grids of 40^3 to 128^3 points with 6 to 14 affinity maps.

Kinds of case:
  score   energy and gene gradient of every pose (score_poses_dev);
  search  ADADELTA local search of every pose (local_search_dev);
  sw      Solis-Wets local search of every pose (local_search_sw_dev);
  batch   ligands of uneven size searched by one call (batch_local_search_dev);
  dock    a whole docking call on host buffers (dock).

Searches are short refinements with a small conditioning constant from poses
near the ligand's reference conformation: each step amplifies rounding (a
gradient component near zero, an atom near a grid-cell face, a clash), so that
after some hundred steps, or from clashing poses, two correct implementations
are at different poses and cannot be compared.  The work of an evaluation does
not depend on the step size.  For the same reason dock runs its Solis-Wets
form, whose decisions compare energies and rarely depend on their rounding.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

import paper_2410_10447_gb300 as adgb
import synth
from paper_2410_10447_gb300.adgb import MAX_GENES, dock_params, sw_params

SPACING = 0.375
CONFORMER_SPREAD = 0.05   # torsion deviation of a start pose from the reference (rad)
SEARCH_EPS = 1e-6         # ADADELTA conditioning constant (Zeiler 2012)


def listed():
    return [
        # rescoring a handful of poses of a small ligand: latency and launches
        dict(name="score_n16", kind="score", atoms=16, tors=4, maps=6, grid=40, poses=64, variant=0),
        # scoring the whole population of a docking run (20 runs x 150)
        dict(name="score_n32", kind="score", atoms=32, tors=8, maps=8, grid=64, poses=3000, variant=0),
        # rescoring a peptide-sized ligand on the largest grid (packed maps beyond L2)
        dict(name="score_n256", kind="score", atoms=256, tors=40, maps=14, grid=128, poses=4096, variant=0),
        # refining a handful of poses of a small ligand: the latency of one search
        dict(name="search_n16", kind="search", atoms=16, tors=4, maps=6, grid=40, poses=64, iters=30, variant=0),
        # the local search of one docking generation, the framework's main path
        dict(name="search_n32", kind="search", atoms=32, tors=8, maps=8, grid=64, poses=3000, iters=30, variant=0),
        # the same with the reduction on the tensor cores
        dict(name="search_n32_tcgen05", kind="search", atoms=32, tors=8, maps=8, grid=64, poses=3000, iters=30, variant=3),
        # odd sizes between one and two warps of atoms, a population of 1000
        dict(name="search_n45", kind="search", atoms=45, tors=11, maps=10, grid=72, poses=1000, iters=30, variant=0),
        # a large flexible ligand
        dict(name="search_n90", kind="search", atoms=90, tors=20, maps=10, grid=80, poses=1500, iters=25, variant=0),
        # a peptide: 256 atoms, 40 torsions, about 30 000 pairs, the largest grid
        dict(name="search_n256", kind="search", atoms=256, tors=40, maps=14, grid=128, poses=2048, iters=20, variant=0),
        # ligands of 10 to 128 atoms, 0 to 32 torsions in one launch
        dict(name="batch_uneven", kind="batch", ligands=96, atoms_lo=10, atoms_hi=128, tors=32, maps=10, grid=72, poses=64, iters=25, variant=0),
        # derivative-free search of one generation
        dict(name="sw_n32", kind="sw", atoms=32, tors=8, maps=8, grid=64, poses=3000, iters=60, variant=0),
        # a whole docking call: 20 runs x 150 individuals
        dict(name="dock_n32", kind="dock", atoms=32, tors=8, maps=8, grid=64, runs=20, pop=150, gens=10, iters=40, variant=0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["score", "search", "search", "search", "sw", "batch", "dock"])
    c = dict(kind=kind, maps=rng.randint(6, 14), grid=rng.randint(40, 96),
             variant=rng.choice([0, 0, 0, 3]))
    if kind == "batch":
        c.update(ligands=_log_int(rng, 12, 96), atoms_lo=rng.randint(10, 30),
                 atoms_hi=_log_int(rng, 40, 128), tors=rng.randint(4, 32), poses=_log_int(rng, 10, 64),
                 iters=rng.randint(10, 25))
        return c
    c["atoms"] = _log_int(rng, 10, 64 if kind == "dock" else 256)
    c["tors"] = rng.randint(0, max(0, min(40, c["atoms"] // 4)))
    if kind == "dock":
        c.update(runs=rng.randint(5, 20), pop=_log_int(rng, 30, 150), gens=rng.randint(2, 10),
                 iters=rng.randint(10, 40))
        return c
    if kind != "score":
        c["iters"] = rng.randint(10, 20 if c["atoms"] > 90 else 30) * (2 if kind == "sw" else 1)
    # from a handful of poses to several populations, less of them for large ligands
    c["poses"] = _log_int(rng, 40, 8000 if c["atoms"] <= 64 else 2000)
    return c


# ------------------------------------------------------------------ inputs
@functools.lru_cache(maxsize=512)
def _shape(atoms, tors, types, key=0):
    """Bond tree, torsions and pair list of the case's ligand (the case alone
    decides them, so that the work of a pass does not depend on the seed)."""
    return synth.make_ligand(7919 * key + 100 * atoms + tors, atoms, types, tors)


def _ligand(rng, atoms, tors, types, key=0):
    lig = dict(_shape(atoms, tors, types, key))
    lig["type"] = rng.integers(0, types, atoms).astype(np.int32)
    q = rng.normal(0.0, 0.3, atoms)
    lig["charge"] = (q - q.mean()).astype(np.float32)
    return lig


def _shapes(case):
    """(ligand shape, poses) of every ligand of the case."""
    if case["kind"] != "batch":
        n = case["runs"] * case["pop"] if case["kind"] == "dock" else case["poses"]
        return [(_shape(case["atoms"], case["tors"], case["maps"]), n)]
    rng = np.random.default_rng(case["atoms_lo"] * 1000 + case["atoms_hi"])
    out = []
    for k in range(case["ligands"]):
        atoms = int(rng.integers(case["atoms_lo"], case["atoms_hi"] + 1))
        tors = int(rng.integers(0, min(case["tors"], atoms // 3) + 1))
        out.append((_shape(atoms, tors, case["maps"], k), case["poses"]))
    return out


def _receptor(rng, n, n_type_maps):
    """Maps of 50 random Gaussians each, and a steep wall at the box faces on
    the affinity maps."""
    M, half = n_type_maps + 2, 0.5 * (n - 1) * SPACING
    dev = dict(dtype=torch.float32, device="cuda")
    ax = torch.arange(n, **dev) * SPACING - half
    amp = torch.tensor(rng.uniform(-2.0, 2.0, (M, 50, 1)), **dev)
    cen = torch.tensor(rng.uniform(-half, half, (3, M, 50, 1)), **dev)
    sig = torch.tensor(rng.uniform(1.0, 4.0, (M, 50, 1)), **dev)
    x, y, z = (torch.exp(-(ax - cen[d]) ** 2 / (2 * sig * sig)) for d in range(3))
    maps = torch.empty(M, n, n, n, **dev)
    for m in range(M):
        plane = (y[m, :, :, None] * x[m, :, None, :]).reshape(50, n * n)
        maps[m] = ((amp[m] * z[m]).T @ plane).reshape(n, n, n)
    wall = sum(torch.clamp((1.5 / d.clamp_min(1e-6)) ** 12, max=1e4) for d in (ax + half, half - ax))
    maps[:n_type_maps] += wall[:, None, None] + wall[None, :, None] + wall[None, None, :]
    return dict(nx=n, ny=n, nz=n, spacing=SPACING, origin=np.full(3, -half, np.float32),
                n_type_maps=n_type_maps, maps=maps.cpu().numpy())


def _off_faces(poses, lig, grid):
    """The poses none of whose atoms lies within 3e-5 A of a grid-cell face,
    where the interpolated gradient jumps: 32-bit coordinates may lie on
    either side of it."""
    u = _coords64(lig, torch.from_numpy(poses).cuda().double()) / SPACING + 0.5 * (grid - 1)
    off = ((u - u.round()).abs().amin((1, 2)) > 3e-5 / SPACING).cpu().numpy()
    return poses[off]


def _poses(rng, n, grid, n_tors):
    """Poses in the middle of the box, uniform rotations, torsions near the
    reference conformation."""
    ext = (grid - 1) * SPACING
    g = np.empty((n, 6 + n_tors))
    g[:, :3] = rng.uniform(-0.15, 0.15, (n, 3)) * ext
    v = rng.normal(size=(n, 4))
    v /= np.linalg.norm(v, axis=1, keepdims=True)
    s = np.linalg.norm(v[:, :3], axis=1)
    g[:, 3] = np.arctan2(v[:, 1], v[:, 0])
    g[:, 4] = np.arccos(np.clip(v[:, 2] / s, -1.0, 1.0))
    g[:, 5] = 2.0 * np.arctan2(s, v[:, 3])
    g[:, 6:] = rng.normal(0.0, CONFORMER_SPREAD, (n, n_tors))
    return g.astype(np.float32)


def _inputs(case, seed):
    """(receptor, [(ligand, poses)]) of a case."""
    rng = np.random.default_rng([int(seed), 2410])
    rec = _receptor(rng, case["grid"], case["maps"])
    ligs = []
    for k, (shape, n) in enumerate(_shapes(case)):
        key = k if case["kind"] == "batch" else 0
        asked = case["tors"] if case["kind"] != "batch" else shape["n_tors"]
        lig = dict(shape)
        drawn = _ligand(rng, shape["n_atoms"], asked, case["maps"], key)
        lig["type"], lig["charge"] = drawn["type"], drawn["charge"]
        if case["kind"] == "score":
            poses = _off_faces(_poses(rng, 3 * n // 2 + 64, case["grid"], shape["n_tors"]), lig, case["grid"])[:n]
        else:
            poses = _poses(rng, n, case["grid"], shape["n_tors"])
        ligs.append((lig, poses))
    return rec, ligs


def prepare(case, seed):
    rec, ligs = _inputs(case, seed)
    ctx = adgb.Context(0)
    s = dict(case=case, ctx=ctx, rid=ctx.upload_receptor_grids(rec),
             lids=[ctx.upload_ligand_torsion_tree(lig) for lig, _ in ligs])
    s["lid"] = s["lids"][0]
    kind = case["kind"]
    if kind == "dock":
        s["params"] = dock_params(n_runs=case["runs"], pop=case["pop"], max_gens=case["gens"],
                                  ls_iters=case["iters"], ls_method=1, seed=int(seed),
                                  reduce_variant=case["variant"])
        return s
    if kind == "batch":
        total = sum(len(p) for _, p in ligs)
        genes = np.zeros((total, MAX_GENES), np.float32)
        at = 0
        for _, p in ligs:
            genes[at:at + len(p), :p.shape[1]] = p
            at += len(p)
        s["start"] = torch.from_numpy(genes).cuda()
        s["bid"] = ctx.batch_create([s["rid"]] * len(ligs), s["lids"], [len(p) for _, p in ligs])
        ctx.batch_autotune(s["bid"], s["start"], iters=5)
    else:
        s["start"] = torch.from_numpy(ligs[0][1]).cuda()
    n = s["start"].shape[0]
    s["energy"] = torch.zeros(n, device="cuda")
    s["genes"] = torch.zeros_like(s["start"])   # gradients, for a scoring case
    if kind == "sw":
        s["evals"] = torch.zeros(n, dtype=torch.int32, device="cuda")
        s["params"] = sw_params(max_evals=case["iters"], rho0=0.25, seed=int(seed),
                                reduce_variant=case["variant"])
    torch.cuda.synchronize()
    return s


def run(state):
    case, ctx = state["case"], state["ctx"]
    kind = case["kind"]
    if kind == "dock":
        genes, energy, evals = ctx.dock(state["rid"], state["lid"], state["params"])
        return dict(genes=genes, energy=energy, evals=evals)
    energy, genes = state["energy"], state["genes"]
    if kind == "score":
        ctx.score_poses_dev(state["rid"], state["lid"], state["start"], energy, genes, case["variant"])
        return dict(energy=energy, grad=genes)
    genes.copy_(state["start"])   # the searches work in place
    if kind == "search":
        ctx.local_search_dev(state["rid"], state["lid"], genes, energy, case["iters"],
                             eps=SEARCH_EPS, variant=case["variant"])
    elif kind == "batch":
        ctx.batch_local_search_dev(state["bid"], genes, energy, case["iters"], eps=SEARCH_EPS,
                                   variant=case["variant"])
    else:
        ctx.local_search_sw_dev(state["rid"], state["lid"], genes, energy, state["params"],
                                evals=state["evals"])
        return dict(energy=energy, genes=genes, evals=state["evals"])
    return dict(energy=energy, genes=genes)


# -------------------------------------------------------------------- work
def work(case):
    """Operations of the scoring function and its gradient, counted from the
    method (a fused multiply-add is two): 110 an atom for the grid terms (70
    without their gradient), 20 an atom that a torsion moves and 30 an atom
    for the pose, 40 a pair (25 without its force), 12 a moved atom for the
    torsion gradients, 8 an atom for the sums, 15 a gene for the update.
    Bytes: poses in, results out, the ligand, and the map values that the
    atoms read, no more than the maps hold."""
    kind = case["kind"]
    evals = {"score": 1, "dock": (case.get("gens", 0) + 1) * case.get("iters", 0)}.get(kind, case.get("iters", 1))
    energy_only = kind in ("sw", "dock")
    flops = bytes_ = gathers = 0
    for lig, n in _shapes(case):
        N, T, P = lig["n_atoms"], lig["n_tors"], len(lig["pairs"])
        moved = int(lig["mov_off"][-1])
        if energy_only:
            one = 70 * N + 20 * moved + 30 * N + 25 * P + N + 6 * (6 + T)
        else:
            one = 110 * N + 20 * moved + 30 * N + 40 * P + 12 * moved + 8 * N
            one += 0 if kind == "score" else 15 * (6 + T)
        flops += n * evals * one
        gathers += n * evals * N * 24 * 4
        bytes_ += 32 * N + 8 * P + 32 * T
        bytes_ += case["runs"] * (4 * (6 + T) + 16) if kind == "dock" else n * (8 * (6 + T) + 4)
    bytes_ += min(gathers, 4 * (case["maps"] + 2) * case["grid"] ** 3)
    return {"bytes": bytes_, "flops": flops}


def tolerance(case):
    """Measured between this library's own forms of the same sums (one or two
    genotypes a warp, pair forces by rounds or by a buffer, shuffles or tensor
    cores): about four times the largest difference seen."""
    kind = case["kind"]
    if kind == "score":
        return {"rel": 3e-5, "max": 1e-3}
    if kind in ("sw", "dock"):
        # equal but for a rare decision between two energies that rounding makes
        return {"rel": 1e-2, "max": 0.9, "differ": 0.01}
    return {"rel": 1e-2, "max": 0.8}


# -------------------------------------------------- the same in 64 bits
W_VDW, W_HB, W_EL, W_DS = 0.1662, 0.1209, 0.1406, 0.1322   # AutoDock4.2 weights
ELEC, SIGMA, QSOL, R_MIN, W_OUT = 332.06363, 3.6, 0.01097, 0.5, 10.0
MS_A, MS_EPS0, MS_LAMBDA, MS_K = -8.5525, 78.4, 0.003627, 7.7839   # Mehler-Solmajer dielectric


def _turn(v, k, s, omc):
    kv = torch.cross(k.expand_as(v), v, dim=-1)
    return v + s * kv + omc * torch.cross(k.expand_as(v), kv, dim=-1)


def _as64(a):
    return torch.as_tensor(np.asarray(a, np.float64), dtype=torch.float64, device="cuda")


def _coords64(lig, genes):
    """Coordinates of poses genes [n][6+T] in double precision."""
    x = _as64(lig["xyz"]).expand(genes.shape[0], -1, -1)
    for k in range(lig["n_tors"]):   # root to leaf, each about its bond's present place
        a, b = (int(i) for i in lig["tors_bond"][k])
        moved = torch.as_tensor(lig["mov_atoms"][lig["mov_off"][k]:lig["mov_off"][k + 1]].astype(np.int64), device="cuda")
        if not len(moved):
            continue
        axis = x[:, b] - x[:, a]
        axis = (axis / axis.norm(dim=-1, keepdim=True))[:, None]
        psi = genes[:, 6 + k, None, None]
        new = x[:, b, None] + _turn(x[:, moved] - x[:, b, None], axis, torch.sin(psi), 1 - torch.cos(psi))
        x = x.index_copy(1, moved, new)
    phi, theta, alpha = (genes[:, j, None, None] for j in (3, 4, 5))
    u = torch.cat([torch.sin(theta) * torch.cos(phi), torch.sin(theta) * torch.sin(phi), torch.cos(theta)], -1)
    return _turn(x, u, torch.sin(alpha), 1 - torch.cos(alpha)) + genes[:, None, :3]


def _energy64(rec, lig, genes, maps):
    """Energies of poses in double precision."""
    x = _coords64(lig, genes)
    q = _as64(lig["charge"])
    t = torch.as_tensor(lig["type"].astype(np.int64), device="cuda")
    # maps at the point clamped onto the grid, and the penalty outside it
    n = rec["nx"]
    lo, h = _as64(rec["origin"]), float(rec["spacing"])
    p = torch.minimum(torch.maximum(x, lo), lo + (n - 1) * h)
    energy = W_OUT * ((x - p) ** 2).sum((1, 2))
    w = (p - lo) / h
    i0 = w.detach().floor().clamp(0, n - 2).long()
    f = w - i0
    for cz in (0, 1):
        for cy in (0, 1):
            for cx in (0, 1):
                at = ((i0[..., 2] + cz) * n + i0[..., 1] + cy) * n + i0[..., 0] + cx
                val = maps[t, at].double() + q * maps[-2][at].double() + q.abs() * maps[-1][at].double()
                weight = 1.0
                for d, c in ((0, cx), (1, cy), (2, cz)):
                    weight = weight * (f[..., d] if c else 1 - f[..., d])
                energy = energy + (weight * val).sum(1)
    if not len(lig["pairs"]):
        return energy
    i, j = (torch.as_tensor(lig["pairs"][:, d].astype(np.int64), device="cuda") for d in (0, 1))
    r2 = ((x[:, i] - x[:, j]) ** 2).sum(-1)
    r = torch.sqrt(r2.clamp_min(R_MIN ** 2))
    R, eps, vol, sol = (_as64(lig[k])[t] for k in ("R", "eps", "vol", "solpar"))
    role = torch.as_tensor(lig["hb_role"].astype(np.int64), device="cuda")[t]
    hb = ((role[i] == 1) & (role[j] == 2)) | ((role[i] == 2) & (role[j] == 1))
    s6 = (0.5 * (R[i] + R[j]) / r) ** 6
    vdw = W_VDW * torch.sqrt(eps[i] * eps[j]) * (s6 * s6 - 2 * s6)
    sh = float(lig["hb_R"]) / r
    vdw = torch.where(hb, W_HB * float(lig["hb_eps"]) * (5 * sh ** 12 - 6 * sh ** 10), vdw)
    B = MS_EPS0 - MS_A
    dielectric = MS_A + B / (1 + MS_K * torch.exp(-MS_LAMBDA * B * r))
    el = W_EL * ELEC * q[i] * q[j] / (r * dielectric)
    S = sol + QSOL * q.abs()
    ds = W_DS * (S[i] * vol[j] + S[j] * vol[i]) * torch.exp(-r2 / (2 * SIGMA ** 2))
    return energy + (vdw + el + ds).sum(1)


def exact(case, seed):
    """Energies and gene gradients in 64 bits; the searches have no such value
    (their steps amplify rounding, so that the distance from a 64-bit search
    says nothing about the precision of a step)."""
    if case["kind"] != "score":
        return None
    rec, ligs = _inputs(case, seed)
    lig, genes = ligs[0]
    maps = torch.from_numpy(rec["maps"]).cuda().reshape(rec["maps"].shape[0], -1)
    chunk = max(1, 4_000_000 // max(1, len(lig["pairs"])))
    energy, grad = [], []
    for k in range(0, len(genes), chunk):
        g = torch.from_numpy(genes[k:k + chunk]).cuda().double().requires_grad_()
        e = _energy64(rec, lig, g, maps)
        grad.append(torch.autograd.grad(e.sum(), g)[0])
        energy.append(e.detach())
    return dict(energy=torch.cat(energy), grad=torch.cat(grad))
