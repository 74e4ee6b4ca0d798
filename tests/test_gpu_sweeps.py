"""The resident sweeps over the shapes they are specialised for, and the counted moves at their
largest degrees.  Block, cluster and level-streaming sweeps carry out the same arithmetic in the
same order, so every result must agree bit for bit; tree structure must equal the oracle's."""
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


@pytest.mark.parametrize("slots", [1, 2, 3, 4, 5, 6, 7, 13])
@pytest.mark.parametrize("variant", [0, 1])
def test_slots_per_lane(ctx, slots, variant):
    """Roots of 1 .. 13 solved slots (one to six to a lane, and groups of several), on pools of
    few moves and of more than eight (the spread segments): resident, split over clusters,
    level-streamed and one slot to an item agree bit for bit."""
    from paper_2508_06559_gb300 import pasur as P
    deck = O.deal(5)
    hands = set(int(c) for c in deck[44:52])
    free = [c for c in range(52) if c not in hands]
    pools = sorted([mask_ids(deck[:4]), mask_ids([c for c in free if c < 20][:9]), mask_ids([c for c in free if c >= 40][:5]), 0])
    clubs = [(a, b, 0, 0) for a in range(7) for b in range(7)][:slots]
    soff, scores = np.arange(len(pools) + 1) * slots, np.array(clubs * len(pools), np.int16)
    out = []
    for extra in ({}, {"split_bytes": 4096}, {"stream_bytes": 1}, {"slots_per_item": 1}):
        t = ctx.pasur_build_round(deck, 5, pools)
        t.pasur_unfold(soff, scores)
        for iters in (17, 1):
            t.pasur_cfr_iterate(P.pasur_config_default(iters=iters, variant=variant, **extra))
        out.append((t.pasur_avg_strategy(), t.pasur_round_utilities()))
        t.free()
    for s, u in out[1:]:
        assert np.array_equal(s, out[0][0]) and np.array_equal(u, out[0][1])


@pytest.mark.parametrize("numerics", [0, 9, 24, 39])
def test_moves_of_large_pools(ctx, numerics):
    """An ace over up to 39 numerics (over a thousand captures of one card), Jacks, Queens and
    Kings in both hands: the tree equals the oracle's node for node."""
    hands = [0, 44, 48, 40, 45, 49, 41, 46]
    deck = np.array([c for c in range(52) if c not in hands] + hands, np.uint8)
    pools = [mask_ids(range(1, 1 + numerics))]
    gt, ot = ctx.pasur_build_round(deck, 5, pools), O.Tree(deck, 5, pools)
    assert gt.pasur_tree_sizes()[0].tolist() == ot.sizes()[0].tolist()
    for k in range(9):
        g, o = gt.pasur_export_level(k), ot.level(k)
        for name in ("parent", "nchild", "lay", "pick", "state", "rus"):
            assert np.array_equal(g[name], getattr(o, name)), (k, name)
    gt.free()


@pytest.mark.parametrize("slots", [2, 3, 4, 5, 6, 13])
@pytest.mark.parametrize("variant", [0, 1])
def test_slots_of_a_block(ctx, slots, variant, monkeypatch, capfd):
    """Blocks of two to six solved slots (a lane holds a node with all of them, or one of them where
    nodes have more than four children or a level has few nodes) against one slot to a block: bit
    for bit, for roots from no pool card up.  Which launches there were is read from the
    solver's own account; the split and streamed runs of the same roots are shown to be just that."""
    from paper_2508_06559_gb300 import pasur as P
    deck = O.deal(5)
    hands = set(int(c) for c in deck[44:52])
    free = [c for c in range(52) if c not in hands]
    pools = sorted([0, mask_ids(deck[:4]), mask_ids([c for c in free if c >= 40][:5]), mask_ids([c for c in free if c < 20][:9]),
                    mask_ids([c for c in free if c < 40][:12])])
    clubs = [(a, b, 0, 0) for a in range(7) for b in range(7)][:slots]
    soff, scores = np.arange(len(pools) + 1) * slots, np.array(clubs * len(pools), np.int16)
    n = -(-slots // 6)
    shares = {slots // n + (1 if i < slots % n else 0) for i in range(n)}
    out = []
    monkeypatch.setenv("PASUR_VERBOSE", "1")
    for extra in ({"slots_per_item": 1}, {"slots_per_item": 6}, {"slots_per_item": 6, "split_bytes": 8192}, {"stream_bytes": 1}):
        t = ctx.pasur_build_round(deck, 5, pools)
        t.pasur_unfold(soff, scores)
        capfd.readouterr()
        for iters in (17, 1):
            t.pasur_cfr_iterate(P.pasur_config_default(iters=iters, variant=variant, **extra))
        log, paths = capfd.readouterr().err, t.pasur_root_paths()
        if "split_bytes" in extra:
            assert (paths == 6).any() and "cluster items" in log
        elif "stream_bytes" in extra:
            assert (paths == 5).any() and "streamed items" in log
        else:
            assert ((paths >= 0) & (paths < 5)).sum() >= 3  # the largest pools' roots fit no block
            assert {int(x.split(" of ")[1].split()[0]) for x in log.splitlines() if "block items" in x} == ({1} if extra["slots_per_item"] == 1 else shares)
        out.append((t.pasur_avg_strategy(), t.pasur_round_utilities()))
        t.free()
    for s, u in out[1:]:
        assert np.array_equal(s, out[0][0]) and np.array_equal(u, out[0][1])
