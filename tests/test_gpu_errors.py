"""Argument checks of the newer entry points: each invalid call returns its documented status
(raised as PasurError by the binding) and leaves the context usable."""
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


def raises(code, fn, *a, **k):
    from paper_2508_06559_gb300 import pasur as P
    with pytest.raises(P.PasurError) as e:
        fn(*a, **k)
    assert e.value.code == code, (e.value.code, str(e.value))


def test_surrogate_arguments(ctx):
    from paper_2508_06559_gb300 import pasur as P
    m = P.Mlp(ctx, dataset_capacity=10)
    raises(P.PASUR_EINVAL, m.set_params, np.zeros(10, np.float32))               # wrong length
    raises(P.PASUR_EINVAL, m.train, 1, 100, 1e-3)                                # batch not a multiple of 128
    raises(P.PASUR_EINVAL, m.train, 1, 128, 1e-3)                                # empty training set
    raises(P.PASUR_EOVERFLOW, m.dataset_add_rows, np.zeros((11, 256), np.uint16), np.zeros(11, np.float32))
    m.dataset_add_rows(np.zeros((3, 256), np.uint16), np.ones(3, np.float32))
    assert m.dataset_size() == 3
    m.dataset_clear()
    assert m.dataset_size() == 0
    deck = O.deal(2)
    t5 = ctx.pasur_build_round(deck, 5, [mask_ids(deck[:4])])
    t5.unfold_single()
    raises(P.PASUR_EINVAL, m.dataset_add_tree, t5)                               # not solved yet
    raises(P.PASUR_EINVAL, m.predict_next, t5)                                   # final round has no next roots
    assert m.forward(np.zeros((0, 256), np.uint16)).shape == (0,)
    t5.free()
    m.free()


def test_value_pass_and_cut_batch_arguments(ctx):
    from paper_2508_06559_gb300 import pasur as P
    deck = O.deal(2)
    t4 = ctx.pasur_build_round(deck, 4, [mask_ids(deck[:4])])
    t4.unfold_single()
    raises(P.PASUR_EINVAL, t4.pasur_root_values, 5)                              # bad mode
    raises(P.PASUR_EINVAL, t4.pasur_root_values, 0)                              # non-final round without links
    t4.free()
    cfg = P.pasur_config_default(iters=10)
    raises(P.PASUR_EINVAL, P.Batch, ctx, deck[None], 3, cfg, 2)                  # last round before first
    raises(P.PASUR_EINVAL, P.Batch, ctx, deck[None], 3, cfg, 4)                  # a cut needs the surrogate
    raises(P.PASUR_EINVAL, P.Batch, ctx, deck[None], 0, P.pasur_config_default(iters=10, split_bytes=-1))
    m = P.Mlp(ctx)
    b = P.Batch(ctx, deck[None], 3, cfg, last_round=4, mlp=m)
    raises(P.PASUR_EINVAL, b.pasur_batch_selfplay, 10, np.zeros(1, np.uint64))   # before solving
    b.pasur_batch_solve()
    raises(P.PASUR_EINVAL, b.pasur_batch_selfplay, 10, np.zeros(1, np.uint64))   # cut before the final round
    b.free()
    m.free()
    # the context still works
    t = ctx.pasur_build_round(deck, 5, [mask_ids(deck[:4])])
    t.unfold_single()
    t.pasur_cfr_iterate(cfg)
    assert np.isfinite(t.pasur_round_utilities()).all()
    t.free()


def test_call_after_a_refused_set_up(ctx):
    """A first call with settings that are refused leaves the tree as it was: the next one solves
    the round as on a fresh tree, with its own settings."""
    from paper_2508_06559_gb300 import pasur as P
    deck = O.deal(5)
    good = P.pasur_config_default(iters=40)
    out = []
    for bad in ((), ({"threads": 100}, {"split_bytes": -1}, {"stream_bytes": -1, "merge_delta": 0})):
        t = ctx.pasur_build_round(deck, 5, [mask_ids(deck[:4])])
        t.pasur_unfold([0, 3], [(0, 0, 0, 0), (0, 0, 4, 0), (1, 0, 0, 0)])
        for extra in bad:
            raises(P.PASUR_EINVAL, t.pasur_cfr_iterate, P.pasur_config_default(iters=40, **extra))
            raises(P.PASUR_EINVAL, t.pasur_avg_strategy)                         # not set up
        t.pasur_cfr_iterate(good)
        out.append((t.pasur_avg_strategy(), t.pasur_round_utilities(), t.pasur_solved_sizes()[0]))
        t.free()
    assert all(np.array_equal(a, b) for a, b in zip(*out))


@pytest.mark.parametrize("rnd,extra", [(5, {}), (4, {}), (5, {"split_bytes": 20000}), (5, {"stream_bytes": 1})])
def test_call_after_a_set_up_without_memory(rnd, extra):
    """A set-up that finds no device memory, at whatever step, gives back what it took; once there
    is memory the same call solves the round as on a fresh tree."""
    from paper_2508_06559_gb300 import pasur as P
    deck = P.pasur_deal(61)
    roots = (np.array([mask_ids(deck[:4])], np.uint64), np.array([0, 1], np.int64), np.zeros((1, 4), np.int16))
    big = P.Ctx(0)
    for r in range(rnd):
        t = big.pasur_build_round(deck, r, roots[0])
        t.pasur_unfold(roots[1], roots[2])
        roots = t.pasur_next_roots_nolinks()[:3]
        t.free()
    cfg = P.pasur_config_default(iters=20, **extra)

    def tree(c):
        t = c.pasur_build_round(deck, rnd, roots[0])
        t.pasur_unfold(roots[1], roots[2])
        return t, None if rnd == 5 else np.sin(np.arange(t.n_next_roots())).astype(np.float32)

    big.close()
    big = P.Ctx(0)  # its peak is this round's alone
    t, nxt = tree(big)
    t.pasur_cfr_iterate(cfg, nxt)
    peak = big.memory()[1]
    want = t.pasur_avg_strategy(), t.pasur_round_utilities()
    t.free()
    big.close()
    small = P.Ctx(0, hbm_budget_bytes=peak + (1 << 20))
    t, nxt = tree(small)
    used, failed = small.memory()[0], 0
    for rows in range((peak - used) // 524 + 2000, -1, -(peak - used) // 524 // 23 - 1):
        try:
            ballast = P.Mlp(small, dataset_capacity=max(rows, 0))
        except P.PasurError:
            continue
        before = small.memory()[0]
        try:
            t.pasur_cfr_iterate(cfg, nxt)
            break
        except P.PasurError as e:
            assert e.code == P.PASUR_ENOMEM
            failed += 1
            assert small.memory()[0] == before
        finally:
            ballast.free()
    else:
        t.pasur_cfr_iterate(cfg, nxt)
    assert failed >= 5
    assert np.array_equal(t.pasur_round_utilities(), want[1])
    import torch
    sigma = torch.zeros(t.n_edges(), device="cuda")  # the export's buffer is the caller's: merged rounds take one more
    try:
        t.pasur_avg_strategy(sigma)
        assert np.array_equal(sigma.cpu().numpy(), want[0])
    except P.PasurError as e:
        assert e.code == P.PASUR_ENOMEM
    t.free()
    small.close()
