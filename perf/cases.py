"""Performance cases of the Pasur solver: the calls a user of the framework makes, over the range of
deals it solves.

A case names a deal by its seed.  The deal fixes the rank of every card position and hence the shape
of every game tree; the seed given to prepare() draws the suits within each rank, so that other
seeds are other deals (clubs, points, score slots, utilities) of the same tree shape.  The score
slots of the later rounds, and with them the results' lengths, depend on the suits: results go to
buffers of the caller, a quarter larger than the deal itself needs, and suits that need more are
drawn again.

  round     one round from its real roots: build, unfold, next roots, CFR, root utilities, strategy
  game      the chain of rounds first..5 of one deal, solved backward (round-by-round CFR)
  batch     many deals planned once and solved together (pasur_batch_solve), strategies exported
  forward   the integer half alone: build, unfold and next roots of every round of a deal
  response  best-response values of both players through solved rounds (exploitability)
  selfplay  sampled games through solved rounds (fair value)
  predict   the utility surrogate's forward pass over feature rows
  train     one epoch of the surrogate's training
"""
import numpy as np
import torch

from paper_2508_06559_gb300 import pasur as P

ITERS = 1000     # iterations per round, the solver's default
# deals whose whole game has over 7e8 full-game-tree nodes: none of them is drawn (47, the first
# deal over 1e9 and the benchmark's headline, is a listed case)
LARGE = (42, 47, 69, 93, 117, 119, 129)
DEALS = [d for d in range(140) if d not in LARGE]


def listed():
    return [
        # one final round from its convention root (pool = the first four cards, score 0): the
        # smallest solve, a user looking at one position
        dict(name="final_round", kind="round", deal=2, first=5, round=5, variant=0),
        # the last four rounds of one small deal: a short chain, mostly single-slot roots
        dict(name="last_four_rounds", kind="game", deal=9, first=2),
        # the whole game of the median deal (5.8e7 full-game-tree nodes)
        dict(name="game_median", kind="game", deal=61, first=0),
        # the whole game of the headline deal (3.4e9 nodes), the paper's size: the largest solve
        dict(name="game_headline", kind="game", deal=47, first=0),
        # a middle round with given next-round utilities under DCFR, the paper's variant: what a
        # root-sharded or surrogate-backed solver calls per round
        dict(name="round_dcfr", kind="round", deal=3, first=2, round=4, variant=1),
        # rounds 4-6 of 64 deals planned once and solved together: the deal-study workload
        dict(name="batch64", kind="batch", deal=0, deals=64, first=3),
        # the forward sweep of a wide deal (3e7 game-tree nodes): trees, unfolding, next roots
        dict(name="forward_wide", kind="forward", deal=115),
        # exploitability of a solved deal: both best responses, fp64
        dict(name="best_response", kind="response", deal=10, first=2),
        # fair value of a solved deal by sampled games
        dict(name="selfplay", kind="selfplay", deal=5, first=2, games=200000),
        # the surrogate's predictions for the roots after a cut (an odd count)
        dict(name="surrogate_predict", kind="predict", rows=134613),
        # one training epoch of the surrogate, the benchmark's batch size
        dict(name="surrogate_train", kind="train", rows=40001, batch=1024),
    ]


def draw(rng):
    kind = rng.choice(["round", "round", "game", "game", "game", "batch", "forward", "response", "selfplay", "predict", "train"])
    if kind == "round":
        last = rng.randint(2, 5)
        first = rng.randint(2, last) if last < 5 else rng.choice([2, 3, 5])
        return dict(kind=kind, deal=rng.choice(DEALS), first=first, round=last, variant=rng.randint(0, 1))
    if kind == "game":
        return dict(kind=kind, deal=rng.choice(DEALS), first=rng.choice([0, 0, 1, 2, 3]))
    if kind == "batch":
        return dict(kind=kind, deal=rng.randrange(60), deals=int(round(2 ** rng.uniform(2, 6))), first=3)
    if kind == "forward":
        return dict(kind=kind, deal=rng.choice(DEALS))
    if kind == "response":
        return dict(kind=kind, deal=rng.choice(DEALS), first=rng.randint(1, 4))
    if kind == "selfplay":
        return dict(kind=kind, deal=rng.choice(DEALS), first=rng.randint(2, 4), games=int(round(10 ** rng.uniform(2, 6))))
    if kind == "predict":
        return dict(kind=kind, rows=int(round(10 ** rng.uniform(0, 5.5))))
    return dict(kind="train", rows=int(round(10 ** rng.uniform(3, 5))), batch=rng.choice([256, 512, 1000, 1024, 2048]))


# ---- inputs ------------------------------------------------------------------------------------


def deck_of(deal, *seed):
    """The deal with its suits drawn anew within every rank (no seed: the deal itself)."""
    deck = P.pasur_deal(int(deal))
    if not seed:
        return deck
    g = np.random.default_rng([int(x) for x in seed] + [int(deal)])
    to = np.concatenate([4 * r + g.permutation(4) for r in range(13)])
    return to[deck.astype(np.int64)].astype(np.uint8)


ROOM = {}  # per deal and rounds: strategies and utilities the result buffers hold


def room_needed(ctx, decks, first, last):
    """(edges, roots) over rounds first..last: what the strategies and utilities of a solve need;
    one round (first < 0): round last from the roots play reaches from round -first-1."""
    n = np.zeros(2, np.int64)
    for deck in decks:
        if first < 0:
            roots, rounds = roots_at(ctx, deck, -first - 1, last), [last]
        else:
            roots, rounds = first_roots(deck), range(first, last + 1)
        for r in rounds:
            t = ctx.pasur_build_round(deck, r, roots[0])
            q = t.pasur_unfold(roots[1], roots[2])
            n += q[1:].sum(), q[0]
            if r < last:
                roots = t.pasur_next_roots_nolinks()[:3]
            t.free()
    return n


def decks_within(ctx, deals, seed, first, last):
    """Suits for the deals that fit the result buffers, and those buffers."""
    key = (tuple(deals), first, last)
    if key not in ROOM:
        ROOM[key] = (room_needed(ctx, [deck_of(d) for d in deals], first, last) * 5 + 3) // 4
    room = ROOM[key]
    for again in range(100):
        decks = [deck_of(d, seed, again) for d in deals]
        if (room_needed(ctx, decks, first, last) <= room).all():
            break
    sigma, utility = (torch.zeros(int(n), dtype=torch.float32, device="cuda") for n in room)
    torch.cuda.synchronize()
    return np.stack(decks), sigma, utility


def first_roots(deck):
    return (np.array([sum(1 << int(c) for c in deck[:4])], np.uint64), np.array([0, 1], np.int64), np.zeros((1, 4), np.int16))


def roots_at(ctx, deck, first, rnd):
    """The roots play reaches at round rnd from the convention root of round `first`."""
    roots = first_roots(deck)
    for r in range(first, rnd):
        t = ctx.pasur_build_round(deck, r, roots[0])
        t.pasur_unfold(roots[1], roots[2])
        roots = t.pasur_next_roots_nolinks()[:3]
        t.free()
    return roots


def utilities(pools, soff, scores, g):
    """Next-round utilities as exact solves give them: the same for score slots of a pool that
    differ only in the inherited difference, +-7 with the clubs bonus, a lean to the player ahead
    in clubs."""
    pool = np.repeat(np.arange(len(pools)), np.diff(soff))
    sc = scores.astype(np.int64)
    key = ((pool * 16 + sc[:, 0]) * 16 + sc[:, 1]) * 4 + sc[:, 3]
    _, inv = np.unique(key, return_inverse=True)
    own = g.normal(0.0, 1.5, int(inv.max()) + 1)[inv] if len(inv) else np.zeros(0)
    u = g.normal(0.0, 3.0, len(pools))[pool] + own + 0.8 * (sc[:, 0] - sc[:, 1])
    return (u + 7.0 * (sc[:, 3] == 1) - 7.0 * (sc[:, 3] == 2)).astype(np.float32)


def feature_rows(ctx, n, g):
    """n surrogate input rows: round-4 roots that play reaches in seeded deals."""
    rows = []
    while sum(len(r) for r in rows) < n:
        deck = deck_of(int(g.integers(0, 41)), int(g.integers(1 << 30)))
        pools, soff, scores = roots_at(ctx, deck, 0, 3)
        rows.append(P.pasur_mlp_root_features(ctx, deck, 3, pools, soff, scores))
    x = np.concatenate(rows)
    return np.ascontiguousarray(x[g.permutation(len(x))[:n]])


def network(ctx, g, cap):
    p = np.zeros(P.N_MLP_PARAMS, np.float32)
    per = 256 * 256 + 256
    for l in range(3):
        p[l * per:l * per + 65536] = g.normal(0.0, 1.4 / 16.0, 65536)
        p[l * per + 65536:(l + 1) * per] = g.normal(0.0, 0.05, 256)
    p[3 * per:] = g.normal(0.0, 0.2, 257)
    mlp = P.Mlp(ctx, dataset_capacity=cap)
    mlp.set_params(p)
    return mlp, p


def batch_deals(case):
    return [DEALS[(case["deal"] + i) % len(DEALS)] for i in range(case["deals"])]


def prepare(case, seed):
    kind = case["kind"]
    g = np.random.default_rng([int(seed), 77])
    ctx = P.Ctx(0)
    s = dict(case=case, kind=kind, ctx=ctx, cfg=P.pasur_config_default(iters=ITERS, variant=case.get("variant", 0)))
    if kind == "round":
        first, rnd = case["first"], case["round"]
        decks, s["sigma"], s["utility"] = decks_within(ctx, [case["deal"]], seed, -first - 1, rnd)
        s["deck"] = decks[0]
        s["roots"] = roots_at(ctx, decks[0], first, rnd)
        s["next"] = None
        if rnd < 5:
            s["next"] = torch.from_numpy(utilities(*roots_at_after(ctx, decks[0], rnd, s["roots"]), g)).cuda()
    elif kind == "game":
        decks, s["sigma"], s["utility"] = decks_within(ctx, [case["deal"]], seed, case["first"], 5)
        s["deck"] = decks[0]
    elif kind == "batch":
        decks, s["sigma"], _ = decks_within(ctx, batch_deals(case), seed, case["first"], 5)
        s["batch"] = P.Batch(ctx, decks, case["first"], s["cfg"])
    elif kind == "forward":
        # the number of score slots depends on the clubs and the points: those keep their suits
        s["deck"] = other_suits(case["deal"], g)
    elif kind in ("response", "selfplay"):
        s["trees"], _ = forward(ctx, deck_of(case["deal"], seed), case["first"])
        solve(s["trees"], P.pasur_config_default(iters=50))
        s["seed"] = int(g.integers(1 << 40))
    elif kind == "predict":
        s["mlp"], _ = network(ctx, g, 0)
        s["x"] = torch.from_numpy(feature_rows(ctx, case["rows"], g).view(np.int16)).cuda()
        s["out"] = torch.zeros(case["rows"], dtype=torch.float32, device="cuda")
        torch.cuda.synchronize()
    elif kind == "train":
        s["mlp"], _ = network(ctx, g, case["rows"])
        x = feature_rows(ctx, case["rows"], g)
        w = g.normal(0.0, 0.6, 256).astype(np.float32)
        y = bf16_values(x) @ w + g.normal(0.0, 1.0, len(x)).astype(np.float32)
        s["mlp"].dataset_add_rows(x, np.ascontiguousarray(y, np.float32))
        s["seed"] = int(g.integers(1 << 40))
    return s


def other_suits(deal, g):
    to = np.arange(52)
    for r in range(13):
        if r != 9:
            to[4 * r + 1:4 * r + 4] = 4 * r + 1 + g.permutation(3)
    return to[P.pasur_deal(int(deal)).astype(np.int64)].astype(np.uint8)


def roots_at_after(ctx, deck, rnd, roots):
    t = ctx.pasur_build_round(deck, rnd, roots[0])
    t.pasur_unfold(roots[1], roots[2])
    after = t.pasur_next_roots_nolinks()[:3]
    t.free()
    return after


def bf16_values(x):
    return (x.astype(np.uint32) << 16).view(np.float32)


# ---- passes ------------------------------------------------------------------------------------


def forward(ctx, deck, first):
    """Every round's tree from `first` on, and the roots between them."""
    trees, between = [], []
    roots = first_roots(deck)
    for r in range(first, 6):
        t = ctx.pasur_build_round(deck, r, roots[0])
        t.pasur_unfold(roots[1], roots[2])
        trees.append(t)
        if r < 5:
            roots = t.pasur_next_roots_nolinks()[:3]
            between.append(roots)
    return trees, between


def solve(trees, cfg, sigma=None, utility=None):
    """The chain of rounds solved backward; where buffers are given, every round's strategies and
    utilities go into them, last round first."""
    nxt, e, q = None, 0, 0
    for t in reversed(trees):
        t.pasur_cfr_iterate(cfg, nxt)
        n = int(t.pasur_tree_sizes()[1][0])
        nxt = torch.empty(n, dtype=torch.float32, device="cuda") if utility is None else utility[q:q + n]
        t.pasur_round_utilities(nxt)
        if sigma is not None:
            m = t.n_edges()
            t.pasur_avg_strategy_async(sigma[e:e + m])
            e, q = e + m, q + n
    trees[0].ctx.pasur_sync()


def run(s):
    kind, case, ctx = s["kind"], s["case"], s["ctx"]
    if kind == "round":
        pools, soff, scores = s["roots"]
        t = ctx.pasur_build_round(s["deck"], case["round"], pools)
        t.pasur_unfold(soff, scores)
        if s["next"] is not None:
            t.n_next_roots()
        t.pasur_cfr_iterate(s["cfg"], s["next"])
        t.pasur_round_utilities(s["utility"])
        t.pasur_avg_strategy(s["sigma"])
        t.free()
        return dict(utility=s["utility"], sigma=s["sigma"])
    if kind == "game":
        trees, _ = forward(ctx, s["deck"], case["first"])
        solve(trees, s["cfg"], s["sigma"], s["utility"])
        for t in trees:
            t.free()
        return dict(utility=s["utility"], sigma=s["sigma"])
    if kind == "batch":
        b = s["batch"]
        utility, at = b.pasur_batch_solve(), 0
        for d in range(b.n_deals):
            for r in range(case["first"], 6):
                t = b.pasur_batch_tree(d, r)
                n = t.n_edges()
                t.pasur_avg_strategy_async(s["sigma"][at:at + n])
                at += n
        ctx.pasur_sync()
        return dict(utility=utility, sigma=s["sigma"])
    if kind == "forward":
        trees, between = forward(ctx, s["deck"], 0)
        out = dict(gt=np.stack([t.pasur_tree_sizes()[0] for t in trees]), fgt=np.stack([t.pasur_tree_sizes()[1] for t in trees]),
                   pools=[b[0].view(np.int64) for b in between], offsets=[b[1] for b in between], scores=[b[2] for b in between])
        for t in trees:
            t.free()
        return out
    if kind == "response":
        return dict(alex=P.chain_values(s["trees"], 1), bob=P.chain_values(s["trees"], 2))
    if kind == "selfplay":
        return dict(games=ctx.pasur_selfplay(s["trees"], case["games"], s["seed"]))
    if kind == "predict":
        return dict(utility=s["mlp"].forward(s["x"], s["out"]))
    losses = s["mlp"].train(1, case["batch"], 1e-3, shuffle_seed=s["seed"])
    return dict(losses=losses, params=s["mlp"].get_params())


# ---- necessary work ----------------------------------------------------------------------------

FLOPS_PER_EDGE = 15   # per swept edge and iteration: both passes' arithmetic on one child
MLP_MACS = 3 * 256 * 256 + 256


def round_work(t, iters):
    """Flops of the CFR on the solved slots' swept edges; bytes of the strategies and utilities
    written and of the trees' nodes (state, parent, move, root: 56 B) built."""
    gt, fgt = t.pasur_tree_sizes()
    swept = t.pasur_solved_sizes()[1]
    return dict(bytes=float(4 * fgt[1:].sum() + 4 * fgt[0] + 56 * gt.sum()), flops=float(FLOPS_PER_EDGE * swept * iters))


def work(case):
    kind = case["kind"]
    if kind in ("predict", "train"):
        n, k = case["rows"], 1 if kind == "predict" else 3
        return dict(bytes=float(n * (512 + 4) + 4 * P.N_MLP_PARAMS * (1 if k == 1 else 7)), flops=2.0 * k * n * MLP_MACS)
    ctx = P.Ctx(0)
    zero = P.pasur_config_default(iters=0)
    total = dict(bytes=0.0, flops=0.0)
    decks = [deck_of(d) for d in (batch_deals(case) if kind == "batch" else [case["deal"]])]
    first = case.get("first", 0)
    for deck in decks:
        if kind == "round":
            roots = roots_at(ctx, deck, first, case["round"])
            t = ctx.pasur_build_round(deck, case["round"], roots[0])
            t.pasur_unfold(roots[1], roots[2])
            trees = [t]
        else:
            trees, _ = forward(ctx, deck, first)
        nxt = None
        for t in reversed(trees):
            gt, fgt = t.pasur_tree_sizes()
            if kind in ("round", "game", "batch"):
                if t is trees[-1] and kind == "round" and case["round"] < 5:
                    nxt = np.zeros(t.n_next_roots(), np.float32)
                t.pasur_cfr_iterate(zero, nxt)
                w = round_work(t, ITERS)
                nxt = np.zeros(int(fgt[0]), np.float32)
            elif kind == "forward":
                # nodes written once, the score slots of every leaf read and ranked once
                w = dict(bytes=float(56 * gt.sum() + 16 * fgt[8]), flops=0.0)
            elif kind == "response":
                # strategies read and node values written once per player
                w = dict(bytes=2.0 * (4 * fgt[1:].sum() + 8 * fgt.sum()), flops=2.0 * 2 * fgt[1:].sum())
            else:
                # per game and ply: a node's child and slot offsets and its children's strategies
                w = dict(bytes=float(case["games"] * (8 * 36 + 2 / len(trees))), flops=0.0)
            total = {k: total[k] + w[k] for k in total}
        for t in trees:
            t.free()
    ctx.close()
    return total


# ---- 64-bit values -----------------------------------------------------------------------------


def exact(case, seed):
    if case["kind"] == "predict":
        g = np.random.default_rng([int(seed), 77])
        ctx = P.Ctx(0)
        mlp, p = network(ctx, g, 0)
        x = torch.from_numpy(bf16_values(feature_rows(ctx, case["rows"], g))).cuda().double()
        ctx.close()
        p = torch.from_numpy(p).cuda().double()
        per = 256 * 256 + 256
        for l in range(3):
            w, b = p[l * per:l * per + 65536].view(256, 256), p[l * per + 65536:(l + 1) * per]
            x = torch.nn.functional.gelu(x @ w.T + b)
        return dict(utility=x @ p[3 * per:-1] + p[-1])
    if case["kind"] == "round" and case["first"] == case["round"] == 5:
        ctx = P.Ctx(0)
        decks, sigma, utility = decks_within(ctx, [case["deal"]], seed, -case["first"] - 1, 5)
        ctx.close()
        return exact_final_round(decks[0], case["variant"], len(sigma), len(utility))
    return None


def captures():
    """Per numeric card, the sets of other numeric cards that complete it to 11, ascending."""
    by_sum = {0: [0]}
    for c in range(40):
        v = c // 4 + 1
        for s in sorted(by_sum, reverse=True):
            if s + v <= 10:
                by_sum.setdefault(s + v, []).extend([m | 1 << c for m in by_sum[s]])
    return [sorted(m for m in by_sum.get(10 - c // 4, []) if m and not m >> c & 1) for c in range(40)]


def exact_final_round(deck, variant, n_sigma, n_utility):
    """CFR of one final round from its convention root in 64 bits (None if the tree is large)."""
    table, numeric = captures(), (1 << 40) - 1
    jack_ace = 0xF | 0xF << 40
    points = lambda m: bin(m & jack_ace).count("1") + 2 * (m >> 4 & 1) + 3 * (m >> 37 & 1)  # noqa: E731
    clubs = lambda m: bin(m & 0x1111111111111).count("1")  # noqa: E731
    hands = [sum(1 << int(c) for c in deck[44 + 4 * p:48 + 4 * p]) for p in (0, 1)]
    # (hand0, hand1, pool, clubs0, clubs1, last picker, points difference)
    levels, first, count = [[(hands[0], hands[1], sum(1 << int(c) for c in deck[:4]), 0, 0, 0, 0)]], [], []
    for k in range(8):
        mv, nxt, cnt = k & 1, [], []
        for h0, h1, pool, c0, c1, last, diff in levels[-1]:
            n0 = len(nxt)
            hand = (h0, h1)[mv]
            for c in range(52):
                if not hand >> c & 1:
                    continue
                if c < 40:
                    picks = [m for m in table[c] if m & ~(pool & numeric) == 0] or [0]
                elif c < 44:
                    picks = [pool & (numeric | 0xF << 40)]
                else:
                    same = pool & (0xF << 44 if c < 48 else 0xF << 48)
                    picks = [1 << b for b in range(44, 52) if same >> b & 1] or [0]
                for m in picks:
                    a = [h0, h1]
                    a[mv] &= ~(1 << c)
                    if m:
                        got = m | 1 << c
                        cc = [c0, c1]
                        cc[mv] += clubs(got)
                        nxt.append((a[0], a[1], pool & ~m, cc[0], cc[1], mv + 1, diff + (points(got) if mv == 0 else -points(got))))
                    else:
                        nxt.append((a[0], a[1], pool | 1 << c, c0, c1, last, diff))
            cnt.append(len(nxt) - n0)
        if len(nxt) > 60000:
            return None
        count.append(np.array(cnt))
        first.append(np.concatenate([[0], np.cumsum(cnt)[:-1]]))
        levels.append(nxt)
    leaf = []
    for _, _, pool, c0, c1, last, diff in levels[8]:
        if last == 1:
            diff, c0 = diff + points(pool), c0 + clubs(pool)
        elif last == 2:
            diff, c1 = diff - points(pool), c1 + clubs(pool)
        leaf.append(diff + (7 if c0 >= 7 else -7 if c1 >= 7 else 0))
    value = [None] * 8 + [np.array(leaf, np.float64)]
    umax = float(np.abs(value[8]).max())
    up = [None] + [np.repeat(np.arange(len(c)), c) for c in count]
    R = [None] + [np.zeros(len(u)) for u in up[1:]]
    S = [None] + [np.zeros(len(u)) for u in up[1:]]
    total = 0.0
    for t in range(1, ITERS + 1):
        thr = float(np.float32(1e-6)) * t * umax
        reach = [(np.ones(1), np.ones(1))]  # own reach of Alex and Bob
        sig = [None] * 9
        for k in range(8):
            rp = np.where(R[k + 1] > thr, R[k + 1], 0.0)
            s = np.add.reduceat(rp, first[k])[up[k + 1]]
            sig[k + 1] = np.where(s > 0, rp / np.where(s > 0, s, 1.0), 1.0 / count[k][up[k + 1]])
            r = [x[up[k + 1]] for x in reach[k]]
            r[k & 1] = r[k & 1] * sig[k + 1]
            reach.append(tuple(r))
        for k in range(7, -1, -1):
            mv, u = k & 1, up[k + 1]
            value[k] = np.add.reduceat(sig[k + 1] * value[k + 1], first[k])
            inst = (1 if mv == 0 else -1) * reach[k][1 - mv][u] * (value[k + 1] - value[k][u])
            if variant == 1:
                a, b = (t - 1.0) ** 1.5, 1.0 if t > 1 else 0.0 ** 0.0
                R[k + 1] = R[k + 1] * np.where(R[k + 1] > 0, a / (a + 1), b / (b + 1)) + inst
                S[k + 1] = S[k + 1] * (1 - 1.0 / t) ** 2 + reach[k][mv][u] * sig[k + 1]
            else:
                R[k + 1] += inst
                S[k + 1] += reach[k][mv][u] * sig[k + 1]
        total += value[0][0]
    bar = []
    for k in range(8):
        s = np.add.reduceat(S[k + 1], first[k])[up[k + 1]]
        bar.append(np.where(s > 0, S[k + 1] / np.where(s > 0, s, 1.0), 1.0 / count[k][up[k + 1]]))
    pad = lambda x, n: np.concatenate([x, np.zeros(n - len(x))])  # noqa: E731
    return dict(utility=pad(np.array([total / ITERS]), n_utility), sigma=pad(np.concatenate(bar), n_sigma))
