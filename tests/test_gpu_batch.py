"""GPU tests of uneven batches: one persistent multi-ligand local-search
launch (graph-captured) over ligands of different sizes, checked against
the single-ligand path and the FP64 oracle."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu
MAXG = 46


@pytest.fixture(scope="module")
def torch():
    import torch as T
    assert T.cuda.is_available(), "GPU tests need a CUDA device"
    return T


@pytest.fixture(scope="module")
def pkg(torch):
    import paper_2410_10447_gb300 as P
    P.load(build=True)
    return P


@pytest.fixture(scope="module")
def setup():
    rec = synth.make_receptor(synth.generate.BASE_SEED + 2, 48, 10)
    ligs = synth.make_uneven_batch(11, 9, atoms=(10, 128), tors=(0, 32), n_types=10)
    ligs.append(synth.make_ligand(77, 256, 10, 40, chain_bias=0.7))   # one large ligand
    n_poses = [5, 9, 1, 12, 3, 8, 7, 2, 10, 6]
    genes = [synth.make_poses(100 + i, n, rec, L["n_tors"]) for i, (L, n) in enumerate(zip(ligs, n_poses))]
    return rec, ligs, n_poses, genes


def pack(genes):
    rows = sum(g.shape[0] for g in genes)
    out = np.zeros((rows, MAXG), np.float32)
    r = 0
    for g in genes:
        out[r:r + g.shape[0], :g.shape[1]] = g
        r += g.shape[0]
    return out


def test_batch_scores_match_single_ligand_calls(pkg, torch, setup):
    rec, ligs, n_poses, genes = setup
    ctx = pkg.Context(0)
    rid = ctx.upload_receptor_grids(rec)
    lids = [ctx.upload_ligand_torsion_tree(L) for L in ligs]
    bid = ctx.batch_create([rid] * len(ligs), lids, n_poses)
    g = torch.from_numpy(pack(genes)).cuda()
    e = torch.empty(g.shape[0], device="cuda")
    ctx.batch_local_search_dev(bid, g, e, 1)          # one evaluation = scoring
    got = e.cpu().numpy()
    r = 0
    for i, L in enumerate(ligs):
        e_ref, _ = ctx.score_poses(rid, lids[i], genes[i], with_grad=False)
        assert np.allclose(got[r:r + n_poses[i]], e_ref, rtol=1e-5, atol=1e-4), i
        # genes are untouched by a one-evaluation search
        assert np.array_equal(g.cpu().numpy()[r:r + n_poses[i], :genes[i].shape[1]], genes[i])
        r += n_poses[i]
    ctx.close()


@pytest.mark.parametrize("autotune, variant, tpp", [(False, -1, 0), (True, -1, 0), (False, 3, 0),
                                                   (False, -1, 128), (False, 3, 128)])
def test_batch_local_search_returns_its_best(pkg, torch, setup, autotune, variant, tpp):
    """tpp 128: the 256-atom ligand takes the block form of the matching
    rounds inside the multi-ligand kernel (two atoms a thread)."""
    rec, ligs, n_poses, genes = setup
    ctx = pkg.Context(0, threads_per_pose=tpp, poses_per_block=128 // tpp) if tpp else pkg.Context(0)
    rid = ctx.upload_receptor_grids(rec)
    lids = [ctx.upload_ligand_torsion_tree(L) for L in ligs]
    bid = ctx.batch_create([rid] * len(ligs), lids, n_poses)
    g0 = torch.from_numpy(pack(genes)).cuda()
    if autotune:
        cfg = ctx.batch_autotune(bid, g0, iters=5)
        assert cfg["threads_per_pose"] in (32, 64, 128) and 1 <= cfg["poses_per_block"] <= 8
        assert np.array_equal(g0.cpu().numpy(), pack(genes))      # autotune leaves genes alone
    g = g0.clone()
    e = torch.empty(g.shape[0], device="cuda")
    ctx.batch_local_search_dev(bid, g, e, 40, variant=variant)        # captured
    g2 = g0.clone()
    e2 = torch.empty_like(e)
    ctx.batch_local_search_dev(bid, g2, e2, 40, variant=variant)      # other buffers: captured again
    g2.copy_(g0)
    ctx.batch_local_search_dev(bid, g2, e2, 40, variant=variant)      # same buffers: graph replayed
    assert np.array_equal(e.cpu().numpy(), e2.cpu().numpy())
    assert np.array_equal(g.cpu().numpy(), g2.cpu().numpy())
    be = e.cpu().numpy()
    gb = g.cpu().numpy()
    r = 0
    for i, L in enumerate(ligs):
        R, OL = oracle.Receptor(rec), oracle.Ligand(L)
        G = 6 + L["n_tors"]
        for k in range(n_poses[i]):
            e_ref = oracle.score(R, OL, gb[r + k, :G])[0]
            assert abs(be[r + k] - e_ref) <= max(1e-4 * abs(e_ref), 1e-3), (i, k, be[r + k], e_ref)
            e0 = oracle.score(R, OL, genes[i][k])[0]
            assert be[r + k] <= e0 + max(1e-4 * abs(e0), 1e-3)
        r += n_poses[i]
    ctx.batch_release(bid)
    ctx.close()


def test_uneven_512_full_size_sampled(pkg, torch):
    """The uneven workload at its full size in the launch configuration
    run_batch times (512 ligands of 10-128 atoms x 64 genotypes x 300
    evaluations, one autotuned, graph-replayed persistent launch): sampled
    genotypes' returned energies equal the FP64 oracle's energy of the
    returned genotypes, and are no higher than their start energies."""
    w = synth.WORKLOADS["uneven_512"]
    rec = synth.make_receptor(synth.generate.BASE_SEED + w["index"], w["grid"], w["n_type_maps"])
    ligs = synth.make_uneven_batch(synth.generate.BASE_SEED + w["index"], 512, w["atoms"], w["tors"],
                                   w["n_types"])
    poses = 64
    ctx = pkg.Context(0)
    rid = ctx.upload_receptor_grids(rec)
    lids = [ctx.upload_ligand_torsion_tree(L) for L in ligs]
    genes = [synth.make_poses(7000 + i, poses, rec, L["n_tors"]) for i, L in enumerate(ligs)]
    g0 = torch.from_numpy(pack(genes)).cuda()
    bid = ctx.batch_create([rid] * len(ligs), lids, [poses] * len(ligs))
    ctx.batch_autotune(bid, g0, iters=15)
    g = g0.clone()
    e = torch.empty(g0.shape[0], device="cuda")
    ctx.batch_local_search_dev(bid, g, e, 300)
    be, gb = e.cpu().numpy(), g.cpu().numpy()
    assert np.all(np.isfinite(be))
    rng = np.random.default_rng(0)
    R = oracle.Receptor(rec)
    for i in sorted(rng.choice(len(ligs), 12, replace=False)):
        L = oracle.Ligand(ligs[i])
        G = 6 + ligs[i]["n_tors"]
        for k in rng.choice(poses, 2, replace=False):
            row = i * poses + k
            e_ref = oracle.score(R, L, gb[row, :G])[0]
            assert abs(be[row] - e_ref) <= max(1e-4 * abs(e_ref), 1e-3), (i, k, be[row], e_ref)
            e0 = oracle.score(R, L, genes[i][k])[0]
            assert be[row] <= e0 + max(1e-4 * abs(e0), 1e-3)
    ctx.batch_release(bid)
    ctx.close()


def test_batch_calls_with_other_buffers_back_to_back(pkg, torch):
    """Several waves of blocks, other buffers in every call, no
    synchronisation between the calls: each returns what it returns alone."""
    rec = synth.make_receptor(synth.generate.BASE_SEED + 3, 48, 6)
    ligs = [synth.make_ligand(500 + a, a, 6, 6) for a in (20, 40, 60, 90)]
    n = 400                                   # 600 blocks and more of each ligand class
    ctx = pkg.Context(0)
    rid = ctx.upload_receptor_grids(rec)
    bid = ctx.batch_create([rid] * 4, [ctx.upload_ligand_torsion_tree(L) for L in ligs], [n] * 4)
    starts = [torch.from_numpy(pack([synth.make_poses(600 + 10 * c + i, n, rec, 6) for i in range(4)])).cuda()
              for c in range(4)]

    def calls(wait):
        genes, energy = [s.clone() for s in starts], [torch.zeros(4 * n, device="cuda") for _ in starts]
        torch.cuda.synchronize()
        for c, (g, e) in enumerate(zip(genes, energy)):
            ctx.batch_local_search_dev(bid, g, e, 20 + c)
            if wait:
                torch.cuda.synchronize()
        torch.cuda.synchronize()
        return genes, energy

    alone, together = calls(True), calls(False)
    for x, y in zip(alone[0] + alone[1], together[0] + together[1]):
        assert torch.equal(x, y)
    ctx.batch_release(bid)
    ctx.close()


@pytest.mark.parametrize("variant", [0, 3])
@pytest.mark.parametrize("ppb", [1, 3, 5, 8])
def test_batch_of_small_ligands_searches_every_genotype(pkg, torch, ppb, variant):
    """Two genotypes a warp with any number of genotypes a block: a block of
    that kernel holds at most four."""
    rec = synth.make_receptor(synth.generate.BASE_SEED + 4, 40, 6)
    ligs = [synth.make_ligand(700 + a, a, 6, 4) for a in (12, 24, 32)]
    n_poses = [17, 9, 8]
    genes = [synth.make_poses(710 + i, n, rec, L["n_tors"]) for i, (L, n) in enumerate(zip(ligs, n_poses))]
    ctx = pkg.Context(0, threads_per_pose=32, poses_per_block=ppb)
    rid = ctx.upload_receptor_grids(rec)
    lids = [ctx.upload_ligand_torsion_tree(L) for L in ligs]
    bid = ctx.batch_create([rid] * 3, lids, n_poses)
    g = torch.from_numpy(pack(genes)).cuda()
    e = torch.full((sum(n_poses),), float("nan"), device="cuda")
    ctx.batch_local_search_dev(bid, g, e, 12, variant=variant)
    r = 0
    for lid, x in zip(lids, genes):
        best, y, _ = ctx.local_search(rid, lid, x.copy(), 12, variant=variant)
        assert np.array_equal(e.cpu().numpy()[r:r + len(x)], best)
        assert np.array_equal(g.cpu().numpy()[r:r + len(x), :x.shape[1]], y)
        r += len(x)
    ctx.close()


def test_context_of_the_autotuned_shape_runs_the_batch_the_same_way(pkg, torch):
    """Large ligands, whose fastest form (two genotypes a 128-thread block) is
    no launch shape of one genotype's threads; the context takes small ones too."""
    rec = synth.make_receptor(synth.generate.BASE_SEED + 6, 48, 6)
    ligs = [synth.make_ligand(900 + a, a, 6, 16) for a in (72, 90)]
    small = synth.make_ligand(901, 20, 6, 4)
    n = 300
    starts = torch.from_numpy(pack([synth.make_poses(910 + i, n, rec, 16) for i in range(2)])).cuda()

    def search(ctx, tune):
        rid = ctx.upload_receptor_grids(rec)
        bid = ctx.batch_create([rid] * 2, [ctx.upload_ligand_torsion_tree(L) for L in ligs], [n] * 2)
        chosen = ctx.batch_autotune(bid, starts, iters=10) if tune else None
        g, e = starts.clone(), torch.empty(2 * n, device="cuda")
        ctx.batch_local_search_dev(bid, g, e, 10)
        return g.cpu().numpy(), e.cpu().numpy(), chosen

    ctx = pkg.Context(0)
    g, e, chosen = search(ctx, True)
    assert (chosen["threads_per_pose"], chosen["poses_per_block"]) == (128, 2)
    again = pkg.Context(0, **chosen)
    g2, e2, _ = search(again, False)
    assert np.array_equal(g, g2) and np.array_equal(e, e2)
    rid, lid = again.upload_receptor_grids(rec), again.upload_ligand_torsion_tree(small)
    x = torch.from_numpy(pack([synth.make_poses(920, 5, rec, 4)])).cuda()
    es = torch.full((5,), float("nan"), device="cuda")
    again.batch_local_search_dev(again.batch_create([rid], [lid], [5]), x, es, 10)
    assert np.all(np.isfinite(es.cpu().numpy()))
    ctx.close()
    again.close()
