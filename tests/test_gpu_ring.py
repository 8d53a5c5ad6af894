"""Ring-sweep kernel (ligands of more than 32 atoms, two genotypes a block) at
the edges of its shapes: every change of atoms a lane, teams, windows and
warps, full and nearly empty last lanes, odd genotype counts, pairs listed
twice and hydrogen-bonded pairs, mixed iteration counts.  Against the FP64
oracle with the tolerances of the other scoring tests: energy max(1e-4 |E|,
1e-3 kcal/mol); gene gradient 1e-3 (2e-3 split precision) of max(|g|_inf, 1)
on poses at least 1e-4 A from grid-cell faces."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    import paper_2410_10447_gb300 as P
    P.load(build=True)
    return P


@pytest.fixture(scope="module")
def rec():
    # No wall at the box faces: ligands of this size reach them.  Inside the
    # wall a corner value of 1e4 next to 0 turns a coordinate's rounding into a
    # gradient change of up to 1e4 / h^2 * u |x| = 7e4 * 6e-8 * 8 A = 0.03
    # kcal/mol/A, times a lever arm of several A for the rotation genes: above
    # 1e-3 of the small gradients compared here.  Without it the maps' second
    # derivatives are below 50 * 2 / (1 A)^2, so the same change is below 1e-4.
    return synth.make_receptor(synth.generate.BASE_SEED + 78, 48, 4, wall=False)


def near_face(r, x, tol=1e-4):
    u = (np.asarray(x, np.float64) - np.asarray(r["origin"], np.float64)) / r["spacing"]
    return bool(np.any(np.abs(u - np.round(u)) * r["spacing"] < tol))


def check_scores(pkg, ctx, rec, lig, genes, variant):
    rid, lid = ctx.upload_receptor_grids(rec), ctx.upload_ligand_torsion_tree(lig)
    R, L = oracle.Receptor(rec), oracle.Ligand(lig)
    e, g = ctx.score_poses(rid, lid, genes, variant=variant)
    for p in range(len(genes)):
        er, gr, x, _ = oracle.score(R, L, genes[p])
        assert abs(e[p] - er) <= max(1e-4 * abs(er), 1e-3), (p, e[p], er)
        if not near_face(rec, x):
            tol = 1e-3 if variant == 0 else 2e-3
            assert np.max(np.abs(g[p] - gr)) <= tol * max(np.max(np.abs(gr)), 1.0), p
    return rid, lid


@pytest.mark.parametrize("n_atoms, n_tors, n, variant", [
    (33, 0, 1, 0), (33, 9, 3, 3), (34, 5, 2, 0), (45, 11, 5, 0), (48, 8, 4, 1), (49, 8, 3, 0),
    (50, 12, 3, 2), (51, 12, 2, 0), (80, 20, 5, 0), (81, 20, 3, 3), (96, 24, 3, 0), (97, 24, 4, 0),
    (160, 40, 3, 3), (161, 40, 3, 0), (192, 40, 2, 0), (193, 40, 3, 3), (224, 30, 3, 0), (255, 40, 3, 0)])
def test_ring_shapes_match_oracle(pkg, rec, n_atoms, n_tors, n, variant):
    lig = synth.make_ligand(41_000 + n_atoms, n_atoms, 4, n_tors)
    genes = synth.make_poses(42_000 + n_atoms, n, rec, lig["n_tors"])
    genes[:, 6:] *= 0.05      # near the reference conformation: no clashes to hide small terms
    ctx = pkg.Context(0)
    rid, lid = check_scores(pkg, ctx, rec, lig, genes, variant)
    R, L = oracle.Receptor(rec), oracle.Ligand(lig)
    best, gb, _ = ctx.local_search(rid, lid, genes.copy(), 8, variant=variant)
    for p in range(n):
        er = oracle.score(R, L, gb[p])[0]
        assert abs(best[p] - er) <= max(1e-4 * abs(er), 1e-3), (p, best[p], er)
    ctx.close()


@pytest.mark.parametrize("n_atoms", [40, 70])
def test_ring_pair_list_forms(pkg, rec, n_atoms):
    """Pairs in either order, listed twice, or none at all; two types, so
    that half of the pairs are donor-acceptor pairs."""
    lig = synth.make_ligand(43_000 + n_atoms, n_atoms, 2, 6)
    genes = synth.make_poses(44_000 + n_atoms, 3, rec, 6)
    genes[:, 6:] *= 0.05
    rng = np.random.default_rng(5)
    pairs = lig["pairs"].copy()
    flip = rng.random(len(pairs)) < 0.5
    pairs[flip] = pairs[flip][:, ::-1]
    for listed in (pairs, np.concatenate([pairs, pairs[::3, ::-1]]), pairs[:1], pairs[:0]):
        ctx = pkg.Context(0)
        check_scores(pkg, ctx, rec, dict(lig, pairs=np.ascontiguousarray(listed)), genes, 0)
        ctx.close()


def test_ring_genotype_does_not_depend_on_its_partner(pkg, rec):
    lig = synth.make_ligand(45_000, 57, 4, 10)
    genes = synth.make_poses(45_001, 7, rec, 10)
    perm = np.array([3, 0, 6, 1, 5, 2, 4])
    ctx = pkg.Context(0)
    rid, lid = ctx.upload_receptor_grids(rec), ctx.upload_ligand_torsion_tree(lig)
    b1, g1, s1 = ctx.local_search(rid, lid, genes.copy(), 20, want_state=True)
    b2, g2, s2 = ctx.local_search(rid, lid, genes[perm].copy(), 20, want_state=True)
    assert np.array_equal(b1[perm], b2) and np.array_equal(g1[perm], g2) and np.array_equal(s1[perm], s2)
    # a resumed search continues the same trajectory (its best starts anew)
    _, _, half = ctx.local_search(rid, lid, genes.copy(), 12, want_state=True)
    _, _, rest = ctx.local_search(rid, lid, genes.copy(), 8, state=half, resume=True)
    assert np.array_equal(rest, s1)
    ctx.close()


@pytest.mark.parametrize("n_atoms", [40, 60, 70, 256])
def test_ring_bits_do_not_depend_on_the_launch_size(pkg, rec, n_atoms):
    """Launches of 1 to 6 blocks an SM run kernels of different register
    budgets: a genotype's bits are the same in each."""
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    lig = synth.make_ligand(49_000 + n_atoms, n_atoms, 4, 8)
    first = synth.make_poses(49_001, 6, rec, 8)
    ctx = pkg.Context(0)
    rid, lid = ctx.upload_receptor_grids(rec), ctx.upload_ligand_torsion_tree(lig)
    ref = ctx.local_search(rid, lid, first.copy(), 6)
    for blocks in (2, 3, 4, 6):
        genes = np.tile(first, (2 * sms * blocks // 6 - 1, 1))
        b, g, _ = ctx.local_search(rid, lid, genes.copy(), 6)
        assert np.array_equal(b[-6:], ref[0]) and np.array_equal(g[-6:], ref[1]), blocks
    ctx.close()


def test_ring_mixed_iteration_counts(pkg, rec):
    """LGA with half of the individuals locally searched: both genotypes of a
    block may stop at different iterations; evaluation counts as the oracle's."""
    lig = synth.make_ligand(46_000, 52, 4, 8)
    kw = dict(n_runs=3, pop=9, max_gens=3, ls_iters=7, ls_rate=0.5, seed=11)
    ctx = pkg.Context(0)
    rid, lid = ctx.upload_receptor_grids(rec), ctx.upload_ligand_torsion_tree(lig)
    genes, energy, evals = ctx.dock(rid, lid, pkg.adgb.dock_params(**kw))
    one = pkg.Context(0, genotypes_per_warp=1)
    r1, l1 = one.upload_receptor_grids(rec), one.upload_ligand_torsion_tree(lig)
    assert np.array_equal(evals, one.dock(r1, l1, pkg.adgb.dock_params(**kw))[2])
    R, L = oracle.Receptor(rec), oracle.Ligand(lig)
    for r in range(3):
        er = oracle.score(R, L, genes[r])[0]
        assert abs(energy[r] - er) <= 1e-9 * max(abs(er), 1.0)
    ctx.close()
    one.close()


@pytest.mark.parametrize("variant", [0, 3])
def test_mixed_batch_equals_single_ligand_calls(pkg, rec, variant):
    """A batch with ligands of every class (two genotypes a warp, the ring's
    three block shapes) returns the single-ligand calls' bits."""
    import torch
    sizes = [(20, 4, 5), (45, 9, 3), (64, 12, 2), (90, 16, 7), (130, 20, 1), (170, 24, 2), (220, 30, 3)]
    ligs = [synth.make_ligand(47_000 + a, a, 4, t) for a, t, _ in sizes]
    genes = [synth.make_poses(48_000 + a, n, rec, l["n_tors"]) for (a, _, n), l in zip(sizes, ligs)]
    ctx = pkg.Context(0)
    rid = ctx.upload_receptor_grids(rec)
    lids = [ctx.upload_ligand_torsion_tree(l) for l in ligs]
    bid = ctx.batch_create([rid] * len(ligs), lids, [len(g) for g in genes])
    g0 = np.zeros((sum(len(g) for g in genes), 46), np.float32)
    at = 0
    for g in genes:
        g0[at:at + len(g), :g.shape[1]] = g
        at += len(g)
    gd, ed = torch.from_numpy(g0).cuda(), torch.empty(len(g0), device="cuda")
    ctx.batch_local_search_dev(bid, gd, ed, 15, variant=variant)
    gb, eb = gd.cpu().numpy(), ed.cpu().numpy()
    at = 0
    for lid, g in zip(lids, genes):
        b, x, _ = ctx.local_search(rid, lid, g.copy(), 15, variant=variant)
        assert np.array_equal(eb[at:at + len(g)], b), lid
        assert np.array_equal(gb[at:at + len(g), :g.shape[1]], x), lid
        at += len(g)
    ctx.close()


# one or two torsions: on either side of the line (thinned, all off the ring)
SPARSE = [(40, 1), (52, 1), (56, 1), (57, 1), (64, 2), (80, 1), (90, 1), (90, 2), (112, 1), (112, 2),
          (128, 2), (128, 4), (129, 1), (160, 1), (200, 2), (256, 2)]


def thinned(lig, share, seed=3):
    """The ligand with a share of its pairs."""
    k = max(1, int(share * len(lig["pairs"])))
    keep = np.sort(np.random.default_rng(seed).permutation(len(lig["pairs"]))[:k])
    return dict(lig, pairs=np.ascontiguousarray(lig["pairs"][keep]))


@pytest.mark.parametrize("n_atoms, n_tors", SPARSE)
def test_large_ligands_with_few_pairs_match_oracle(pkg, rec, n_atoms, n_tors):
    """Few torsions list few of a large ligand's pairs: such ligands may leave
    the ring for the other kernels, on either side of the line."""
    lig = synth.make_ligand(50_000 + n_atoms, n_atoms, 4, n_tors)
    genes = synth.make_poses(51_000 + n_atoms, 3, rec, lig["n_tors"])
    genes[:, 6:] *= 0.05
    R = oracle.Receptor(rec)
    for l in (lig, thinned(lig, 0.1)):
        ctx = pkg.Context(0)
        rid, lid = check_scores(pkg, ctx, rec, l, genes, 0)
        best, gb, _ = ctx.local_search(rid, lid, genes.copy(), 8)
        L = oracle.Ligand(l)
        for p in range(len(genes)):
            er = oracle.score(R, L, gb[p])[0]
            assert abs(best[p] - er) <= max(1e-4 * abs(er), 1e-3), (p, best[p], er)
        ctx.close()


def test_sparse_and_dense_ligands_share_a_batch(pkg, rec):
    """Ligands of every form in one batch, each at sizes where its batch form
    is its single call's: the single calls' bits."""
    import torch
    ligs = [synth.make_ligand(52_000 + a, a, 4, t) for a, t in
            ((20, 4), (40, 8), (52, 1), (56, 1), (52, 12), (96, 1), (112, 1), (112, 20), (140, 30))]
    ligs.append(thinned(synth.make_ligand(52_300, 200, 4, 8), 0.02))
    genes = [synth.make_poses(52_400 + i, 3 + i, rec, l["n_tors"]) for i, l in enumerate(ligs)]
    ctx = pkg.Context(0)
    rid = ctx.upload_receptor_grids(rec)
    lids = [ctx.upload_ligand_torsion_tree(l) for l in ligs]
    bid = ctx.batch_create([rid] * len(ligs), lids, [len(g) for g in genes])
    g0 = np.zeros((sum(len(g) for g in genes), 46), np.float32)
    at = 0
    for g in genes:
        g0[at:at + len(g), :g.shape[1]] = g
        at += len(g)
    gd, ed = torch.from_numpy(g0).cuda(), torch.empty(len(g0), device="cuda")
    ctx.batch_local_search_dev(bid, gd, ed, 15)
    gb, eb = gd.cpu().numpy(), ed.cpu().numpy()
    at = 0
    for lid, g in zip(lids, genes):
        b, x, _ = ctx.local_search(rid, lid, g.copy(), 15)
        assert np.array_equal(eb[at:at + len(g)], b), lid
        assert np.array_equal(gb[at:at + len(g), :g.shape[1]], x), lid
        at += len(g)
    ctx.close()


@pytest.mark.parametrize("n_atoms", [161, 176, 193, 220])
def test_ring_bits_of_two_windows_do_not_depend_on_the_launch_size(pkg, rec, n_atoms):
    """Three and four atoms a lane over two windows of lanes: another number
    of blocks an SM in large launches on either side of 192 atoms."""
    test_ring_bits_do_not_depend_on_the_launch_size(pkg, rec, n_atoms)
