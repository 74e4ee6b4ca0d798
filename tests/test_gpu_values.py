"""fp64 game values on the GPU (minimax, best responses, on-policy) against the oracle's recursion,
chained over rounds 5 and 6 with the oracle's own strategy (rounded to float32) given to both
sides.  Both sum child by child in canonical order without fused multiply-add, so the values
agree to rounding (1e-12 relative); the best-response values bracket the on-policy and minimax
values."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import torch
    assert torch.cuda.is_available()
    from paper_2508_06559_gb300 import build as B
    from paper_2508_06559_gb300 import pasur as P
    B.build()
    c = P.Ctx(0)
    yield c
    c.close()


def mask_ids(ids):
    m = 0
    for c in ids:
        m |= 1 << int(c)
    return m


@pytest.mark.parametrize("seed", [0, 2, 5, 9])
def test_chained_values_match_oracle(ctx, seed):
    from paper_2508_06559_gb300 import pasur as P
    deck = O.deal(seed)
    o4 = O.Tree(deck, 4, [mask_ids(deck[:4])])
    o4.unfold_single()
    pools, soff, scores, lnk = o4.next_roots()
    o5 = O.Tree(deck, 5, pools)
    o5.unfold(soff, scores)
    leaf5 = o5.leaf_utilities_final()
    s5, U5 = o5.cfr(leaf5, 100)
    s4, _ = o4.cfr(o4.leaf_utilities_linked(lnk, U5), 100)
    s4f, s5f = s4.astype(np.float32), s5.astype(np.float32)
    g4 = ctx.pasur_build_round(deck, 4, [mask_ids(deck[:4])])
    g4.unfold_single()
    g4.pasur_next_roots()
    g5 = ctx.pasur_build_round(deck, 5, pools)
    g5.pasur_unfold(soff, scores)
    vals = {}
    for mode in (O.MINIMAX, O.BR_ALEX, O.BR_BOB, O.ON_POLICY):
        o_v5 = o5.root_values(leaf5, mode, s5f.astype(np.float64))
        o_v4 = o4.root_values(o4.leaf_utilities_linked(lnk, o_v5), mode, s4f.astype(np.float64))
        got = P.chain_values([g4, g5], mode, [s4f, s5f])
        got5 = g5.pasur_root_values(mode, s5f)
        assert np.allclose(got5, o_v5, rtol=1e-12, atol=1e-12)
        assert np.allclose(got, o_v4, rtol=1e-12, atol=1e-12), (mode, got, o_v4)
        vals[mode] = got[0]
    assert vals[O.BR_BOB] <= vals[O.ON_POLICY] + 1e-12 <= vals[O.BR_ALEX] + 2e-12
    assert vals[O.BR_BOB] <= vals[O.MINIMAX] + 1e-12 <= vals[O.BR_ALEX] + 2e-12
    assert abs(vals[O.MINIMAX] - O.minimax_rounds(deck, 4, mask_ids(deck[:4]))) < 1e-9
    for t in (g4, g5):
        t.free()


def test_solved_strategy_exploitability_is_small(ctx):
    """After CFR on the GPU the chained best-response gap of the solved profile is small and
    shrinks with more iterations."""
    from paper_2508_06559_gb300 import pasur as P
    deck = O.deal(2)
    gaps = []
    for T in (50, 800):
        g4 = ctx.pasur_build_round(deck, 4, [mask_ids(deck[:4])])
        g4.unfold_single()
        pools, soff, scores, _ = g4.pasur_next_roots()
        g5 = ctx.pasur_build_round(deck, 5, pools)
        g5.pasur_unfold(soff, scores)
        cfg = P.pasur_config_default(iters=T)
        g5.pasur_cfr_iterate(cfg)
        g4.pasur_cfr_iterate(cfg, g5.pasur_round_utilities())
        a = P.chain_values([g4, g5], 1)[0]
        b = P.chain_values([g4, g5], 2)[0]
        gaps.append((a - b) / 2)
        for t in (g4, g5):
            t.free()
    assert gaps[0] >= 0 and gaps[1] >= 0
    assert gaps[1] < gaps[0]


@pytest.mark.parametrize("first", [2, 3, 4])
def test_values_over_tree_shapes(ctx, first):
    """A round of one root and one score slot (its tree split over blocks below the top levels)
    and the rounds after it (split at their roots): the on-policy values against a
    level-by-level numpy pass over the exported tree (sums of products to rounding), and every
    mode with the solver's own strategies against the same strategies handed in (equal)."""
    from paper_2508_06559_gb300 import pasur as P
    deck = O.deal(5)
    cfg, roots, trees = P.pasur_config_default(iters=20), None, []
    for rnd in range(first, 6):
        t = ctx.pasur_build_round(deck, rnd, [mask_ids(deck[:4])] if roots is None else roots[0])
        t.unfold_single() if roots is None else t.pasur_unfold(roots[1], roots[2])
        if rnd < 5:
            roots = t.pasur_next_roots()
            lnk = roots[3] if rnd == first else lnk
        trees.append(t)
    nv, sigmas = None, []
    for t in reversed(trees):
        t.pasur_cfr_iterate(cfg, nv)
        sigmas.insert(0, t.pasur_avg_strategy())
        nv = t.pasur_round_utilities()
    for mode in (O.MINIMAX, O.BR_ALEX, O.BR_BOB, O.ON_POLICY):
        assert np.array_equal(P.chain_values(trees, mode), P.chain_values(trees, mode, sigmas))
    nxt = P.chain_values(trees[1:], O.ON_POLICY)
    want = P.chain_values(trees, O.ON_POLICY)
    t = ctx.pasur_build_round(deck, first, [mask_ids(deck[:4])])
    t.unfold_single()
    t.pasur_next_roots()
    t.pasur_cfr_iterate(P.pasur_config_default(iters=0), np.zeros(len(nxt), np.float32))
    gt, fgt = t.pasur_tree_sizes()
    assert np.array_equal(gt, fgt)  # one slot: an FGT node is a GT node
    val = t.pasur_leaf_values().astype(np.float64) + nxt[lnk]  # the round's difference + the next round
    for k in range(7, -1, -1):
        s = sigmas[0][fgt[1:k + 1].sum():fgt[1:k + 2].sum()].astype(np.float64)
        nchild = t.pasur_export_level(k)["nchild"]
        val = np.add.reduceat(s * val, np.concatenate([[0], np.cumsum(nchild)[:-1]]))
    assert np.allclose(val, want, rtol=1e-12, atol=1e-12)
    for x in trees + [t]:
        x.free()


@pytest.mark.parametrize("seed,rnd,slots", [(9, 3, 1), (9, 3, 3), (10, 4, 1), (61, 4, 1), (61, 5, 60), (5, 3, 2)])
def test_values_of_wide_and_narrow_rounds(ctx, seed, rnd, slots):
    """Rounds with many roots of very different sizes, on both sides of the line between a block
    per range of subtrees (two launches a call) and a launch per level (nine): 2^17 leaves, or
    5 * 2^19 with their slots.  Against a numpy pass over the exported tree: minimax exactly, the
    others to the rounding of two sums of d products of weights that add up to 1, over 8 levels."""
    from paper_2508_06559_gb300 import pasur as P
    deck = O.deal(seed)
    pools, soff, scores = np.array([mask_ids(deck[:4])], np.uint64), np.array([0, 1], np.int64), np.zeros((1, 4), np.int16)
    for r in range(rnd):
        t = ctx.pasur_build_round(deck, r, pools)
        t.pasur_unfold(soff, scores)
        pools, soff, scores, _ = t.pasur_next_roots_nolinks()
        t.free()
    clubs = [(a, b, 0, 0) for a in range(8) for b in range(8)][:slots]
    t = ctx.pasur_build_round(deck, rnd, pools)
    t.pasur_unfold(np.arange(len(pools) + 1, dtype=np.int64) * slots, np.array(clubs * len(pools), np.int16))
    gt, fgt = t.pasur_tree_sizes()
    wide = gt[8] >= 2 ** 17 or fgt[8] >= 5 * 2 ** 19
    rng = np.random.default_rng(seed)
    nxt = lnk = None
    if rnd < 5:
        lnk = t.pasur_next_roots()[3]
        nxt = rng.normal(0, 9, t.n_next_roots())
    t.pasur_cfr_iterate(P.pasur_config_default(iters=0), None if rnd == 5 else np.zeros(len(nxt), np.float32))
    leaf = t.pasur_leaf_values().astype(np.float64)  # without the next round's values: whole numbers
    if rnd < 5:
        leaf = leaf + nxt[lnk]
    leaf = leaf.reshape(-1, slots)
    nchild = [t.pasur_export_level(k)["nchild"] for k in range(8)]
    first = [np.concatenate([[0], np.cumsum(n)[:-1]]) for n in nchild]
    sigma = []
    for n, f in zip(nchild, first):
        x = 1 - rng.random((int(n.sum()), slots), np.float32)  # in (0, 1]
        sigma.append((x / np.repeat(np.add.reduceat(x, f), n, axis=0)).astype(np.float32))
    flat = np.concatenate([x.ravel() for x in sigma])
    dmax = max(int(n.max()) for n in nchild)
    for mode in (O.MINIMAX, O.BR_ALEX, O.BR_BOB, O.ON_POLICY):
        launches = ctx.pasur_launch_count()
        got = t.pasur_root_values(mode, None if mode == O.MINIMAX else flat, nxt)
        assert ctx.pasur_launch_count() - launches == (9 if wide else 2)
        val = leaf
        for k in range(7, -1, -1):
            alex = k % 2 == 0
            if mode == O.MINIMAX or mode == (O.BR_ALEX if alex else O.BR_BOB):
                val = (np.maximum if alex else np.minimum).reduceat(val, first[k])
            else:
                val = np.add.reduceat(sigma[k].astype(np.float64) * val, first[k])
        bound = 0.0 if mode == O.MINIMAX else 2 * 8 * (dmax + 1) * 2.0 ** -53 * 1.01 * np.abs(leaf).max()
        assert np.abs(got - val.ravel()).max() <= bound, mode
    t.free()
