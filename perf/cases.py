"""The work a user of this framework has it do, as cases that can be timed.

A case is a dict of plain values.  `prepare` makes what a program has in hand
before the call (a context, roots, a forest, a network, a server), `run` makes
one pass through the public entry points, `work` counts what the path cannot do
without, and `exact` gives the floating-point outputs in 64 bits from plain
torch.  Searches, playouts, determinizations and served decisions are whole
numbers: they are pure functions of the seeds and need no 64-bit counterpart.

Sizes are those of the framework's workloads (the batched benchmark, the
single tree, the uneven four-player forest, self-play moves, labelling,
training and the serving loop), shortened where a whole run takes seconds.
"""
import math

import numpy as np
import torch

import paper_2403_10720_gb300 as dvc
from paper_2403_10720_gb300 import autotune

# variant name: (players, tiles, deal, most draws before a root, most face-up tiles of a seat)
VARIANTS = {
    "2p24": (2, 24, 4, 10, 5),
    "3p24": (3, 24, 4, 6, 3),
    "4p24": (4, 24, 3, 8, 3),
    "2p26": (2, 26, 4, 10, 5),
    "3p26": (3, 26, 4, 6, 3),
    "4p26": (4, 26, 3, 8, 3),
}
# integer operations of one playout (about 104 per game step of a two-player
# game without jokers: the guess, its resolution, the draw and their random
# words; twice that with more seats or jokers)
PLAYOUT_OPS = {"2p24": 12.7 * 104, "3p24": 14 * 208, "4p24": 16 * 208, "2p26": 13 * 208, "3p26": 15 * 208,
               "4p26": 17 * 208}
FEATURES, HIDDEN = 640, 512
MACS = FEATURES * HIDDEN + 2 * HIDDEN * HIDDEN + 4 * HIDDEN  # one leaf's forward pass
NPARAMS = 855556


def listed():
    return [
        # the benchmark's batch: thousands of mid-game positions searched at
        # once, 256 playouts per leaf (a quarter of its iterations)
        dict(name="search_batch_2p24", kind="search", variant="2p24", trees=4096, lo=1024, hi=1024, playouts=256,
             value=False, full=False, tail=False, opening=False),
        # one turn of 2,000 self-play games under the full rules (a correct
        # guess keeps the turn, in the tree as in the game)
        dict(name="search_moves_full_2p24", kind="search", variant="2p24", trees=2000, lo=256, hi=256, playouts=32,
             value=False, full=True, tail=False, opening=True),
        # uneven four-player joker trees, log-uniform budgets, run to the end
        # of the longest under the library's schedule for such forests
        dict(name="search_uneven_4p26", kind="search", variant="4p26", trees=4096, lo=500, hi=10000, playouts=32,
             value=False, full=False, tail=True, opening=False),
        # one analysed position: one tree, one playout per leaf, and the whole
        # tree read back
        dict(name="search_single_2p24", kind="search", variant="2p24", trees=1, lo=10000, hi=10000, playouts=1,
             value=False, full=False, tail=False, opening=True),
        # the value-network agent's decisions on 4,096 positions
        dict(name="search_value_2p24", kind="search", variant="2p24", trees=4096, lo=256, hi=256, playouts=32,
             value=True, full=False, tail=False, opening=False),
        # one chunk of training labels: 16,384 states, 1,024 playouts each
        dict(name="rollout_labels_2p24", kind="rollout", variant="2p24", leaves=16384, playouts=1024),
        # a caller's own search scoring a few leaves: the smallest call
        dict(name="rollout_few_4p26", kind="rollout", variant="4p26", leaves=45, playouts=37),
        # deals consistent with a seat's view, for a caller's own search
        dict(name="determinize_4p26", kind="determinize", variant="4p26", roots=1000),
        # network inference on the workload's batch of leaves
        dict(name="value_eval_4p26", kind="eval", variant="4p26", rows=65536),
        # ... and on the leaves of a small forest
        dict(name="value_eval_few_3p24", kind="eval", variant="3p24", rows=333),
        # one training step, forward and backward, at the trainer's batch
        dict(name="value_train_2p24", kind="train", variant="2p24", rows=8192),
        # move queries of concurrent games of two variants, half of them in
        # value mode, through the server until all are answered
        dict(name="serve_mixed", kind="serve", queries=200, lo=200, hi=2000, playouts=32),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1))))))


def draw(rng):
    kind = rng.choice(["search", "search", "search", "rollout", "rollout", "determinize", "eval", "eval", "train",
                       "serve"])
    variant = rng.choice(sorted(VARIANTS))
    if kind == "search":
        value = rng.random() < 0.25
        trees = _log_int(rng, 1, 4096)
        hi = _log_int(rng, 64, 4096)
        playouts = 32 if value else _log_int(rng, 1, 256)
        most = 1 << 20 if value else int(1.2e12 / PLAYOUT_OPS[variant] / playouts)
        hi = max(16, min(hi, most // trees))
        tail = not value and rng.random() < 0.25
        return dict(kind=kind, variant=variant, trees=trees, lo=max(1, hi // 20) if tail else hi, hi=hi,
                    playouts=playouts, value=value, full=rng.random() < 0.25, tail=tail, opening=rng.random() < 0.3)
    if kind == "rollout":
        leaves = _log_int(rng, 1, 16384)
        return dict(kind=kind, variant=variant, leaves=leaves,
                    playouts=_log_int(rng, 1, max(1, min(1024, int(1.6e10 / PLAYOUT_OPS[variant] / leaves)))))
    if kind == "determinize":
        return dict(kind=kind, variant=variant, roots=_log_int(rng, 1, 1000))
    if kind == "eval":
        return dict(kind=kind, variant=variant, rows=_log_int(rng, 1, 65536))
    if kind == "train":
        return dict(kind=kind, variant=variant, rows=_log_int(rng, 100, 8192))
    lo = _log_int(rng, 50, 400)
    return dict(kind=kind, queries=_log_int(rng, 1, 200), lo=lo, hi=rng.randint(lo, 2000), playouts=32)


# ------------------------------------------------------------------ inputs

def _config(variant, playouts=1, full=False, opening=False):
    np_, nt, deal, predraw, revealed = VARIANTS[variant]
    return dvc.Config(nplayers=np_, ntiles=nt, deal=deal, max_predraw=0 if opening else predraw,
                      max_revealed=revealed, playouts=playouts, tree_continue=int(full))


def _budgets(case, seed, n):
    u = np.random.default_rng(seed).uniform(math.log(case["lo"]), math.log(case["hi"] + 1), size=n)
    return np.clip(np.floor(np.exp(u)), case["lo"], case["hi"]).astype(np.int32)


def _params(seed):
    """Network parameters as the library's flat FP32 array: Glorot-uniform
    matrices at BF16 values (the network's weight type), small biases."""
    rng = np.random.default_rng(seed)
    out = []
    for o, i in ((HIDDEN, FEATURES), (HIDDEN, HIDDEN), (HIDDEN, HIDDEN), (4, HIDDEN)):
        lim = math.sqrt(6.0 / (i + o))
        w = torch.from_numpy(rng.uniform(-lim, lim, size=(o, i)).astype(np.float32))
        out += [w.to(torch.bfloat16).to(torch.float32).reshape(-1),
                torch.from_numpy(rng.uniform(-0.05, 0.05, size=o).astype(np.float32))]
    return torch.cat(out)


def _positions(variant, n, seed):
    """n mid-game records (n x 32 uint8): a shuffled deal, further draws by
    the seats in turn, some tiles of every seat face up, the mover has drawn."""
    np_, nt, deal, predraw, revealed = VARIANTS[variant]
    rng = np.random.default_rng(seed)
    perm = rng.random((n, nt)).argsort(axis=1)
    draws = rng.integers(0, predraw + 1, size=n)
    cur = draws % np_
    slot = np.arange(nt)[None, :]
    # seat of the tile at each place of the shuffle: the deal, then the draws in turn, then the mover's draw
    seat = np.where(slot < np_ * deal, slot // deal, (slot - np_ * deal) % np_)
    held = slot < (np_ * deal + draws + 1)[:, None]
    is_drawn = slot == (np_ * deal + draws)[:, None]
    want = rng.integers(0, revealed + 1, size=(n, np_))
    up = np.zeros((n, nt), dtype=bool)
    score = rng.random((n, nt))
    for p in range(np_):
        mine = held & (seat == p) & ~is_drawn
        k = np.minimum(want[:, p], np.maximum(mine.sum(axis=1) - 1, 0))
        rank = np.where(mine, score, 2.0).argsort(axis=1).argsort(axis=1)
        up |= mine & (rank < k[:, None])
    bits = np.left_shift(np.uint32(1), perm.astype(np.uint32))
    hands = np.zeros((n, 4), dtype=np.uint32)
    for p in range(np_):
        hands[:, p] = np.where(held & (seat == p), bits, np.uint32(0)).sum(axis=1, dtype=np.uint32)
    rev = np.where(up, bits, np.uint32(0)).sum(axis=1, dtype=np.uint32)
    s = np.zeros((n, 32), dtype=np.uint8)
    s[:, :16] = hands.view(np.uint8)
    s[:, 16:20] = rev.reshape(n, 1).view(np.uint8)
    owner = np.full((n, 2), -1)
    numbered = np.zeros((n, 4), dtype=np.int64)
    for p in range(np_):
        numbered[:, p] = np.array([(hands[:, p] >> np.uint32(t)) & np.uint32(1) for t in range(24)]).sum(axis=0)
        for j in range(nt - 24):
            owner[(hands[:, p] >> np.uint32(24 + j)) & np.uint32(1) == 1, j] = p
    rows = np.arange(n)
    gap = np.zeros((n, 2), dtype=np.int64)
    for j in range(2):
        most = np.where(owner[:, j] >= 0, numbered[rows, np.maximum(owner[:, j], 0)], 0)
        gap[:, j] = np.floor(rng.random(n) * (most + 1)).astype(np.int64)
    white_first = (owner[:, 0] >= 0) & (owner[:, 0] == owner[:, 1]) & (gap[:, 0] == gap[:, 1]) & (rng.random(n) < 0.5)
    s[:, 20:22] = gap
    s[:, 22] = white_first
    s[:, 23] = cur
    s[:, 24] = perm[rows, np_ * deal + draws]
    s[:, 25] = (1 << np_) - 1
    s[:, 26] = np_
    s[:, 27] = nt
    s[:, 28] = 0xFF
    return s


def _labels(variant, n, seed):
    """Win fractions of 1,024 playouts per seat in play."""
    np_ = VARIANTS[variant][0]
    rng = np.random.default_rng(seed)
    y = np.zeros((n, 4), dtype=np.float32)
    y[:, :np_] = rng.multinomial(1024, rng.dirichlet(np.full(np_, 3.0), size=n)) / 1024.0
    return y


def _ids(n, seed):
    rng = np.random.default_rng(seed)
    return torch.from_numpy(rng.integers(0, 1 << 20, size=n).astype(np.int32)).cuda()


LEARNING_RATE = 1e-3


def prepare(case, seed):
    kind = case["kind"]
    if kind == "search":
        ctx = dvc.Context(_config(case["variant"], case["playouts"], case["full"], case["opening"]))
        if case["value"]:
            ctx.dvc_value_params(_params(seed).cuda())
        roots = ctx.dvc_init_states(seed, case["trees"])
        budgets = _budgets(case, seed, case["trees"])
        forest = dvc.Forest(ctx, roots, budgets, seed)
        forest.dvc_forest_count_work(False)  # instrumentation, off in a program that only searches
        return dict(case=case, ctx=ctx, roots=roots, budgets=budgets, forest=forest,
                    sms=torch.cuda.get_device_properties(0).multi_processor_count)
    if kind == "rollout":
        ctx = dvc.Context(_config(case["variant"]))
        n = case["leaves"]
        return dict(case=case, ctx=ctx, leaves=ctx.dvc_init_states(seed, n), seed=seed, trees=_ids(n, seed),
                    ids=_ids(n, seed + 1))
    if kind == "determinize":
        ctx = dvc.Context(_config(case["variant"]))
        n = case["roots"]
        return dict(case=case, ctx=ctx, roots=ctx.dvc_init_states(seed, n), seed=seed, trees=_ids(n, seed),
                    ids=_ids(n, seed + 1))
    if kind in ("eval", "train"):
        ctx = dvc.Context(_config(case["variant"]))
        ctx.dvc_value_params(_params(seed).cuda())
        state = dict(case=case, ctx=ctx, states=torch.from_numpy(_positions(case["variant"], case["rows"], seed)).cuda())
        if kind == "train":
            state["labels"] = torch.from_numpy(_labels(case["variant"], case["rows"], seed)).cuda()
            state["loss"] = torch.zeros(1, device="cuda")
        return state
    ctxs = [dvc.Context(_config(v, case["playouts"])) for v in ("2p24", "4p26")]
    for i, c in enumerate(ctxs):
        c.dvc_value_params(_params(seed + i).cuda())
    server = dvc.Server(ctxs, 512 << 20, 2000, value_share_pct=35, seed=seed)
    rng = np.random.default_rng(seed)
    n = case["queries"]
    roots = [c.dvc_init_states(seed + 7, n).cpu().numpy() for c in ctxs]
    budgets = _budgets(case, seed, n)
    modes = rng.integers(0, 2, size=n)
    return dict(case=case, ctxs=ctxs, server=server,
                queries=[(roots[i % 2][i], int(budgets[i]), int(modes[i]), i) for i in range(n)])


# --------------------------------------------------------------------- run

def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "search":
        f = state["forest"]
        f.dvc_forest_reset(state["roots"])
        if case["tail"]:
            # pipeline CTAs of one tree and one warp while many trees run (the
            # launch shape the tuner picks for such forests), then the tail
            autotune.step_with_tail(f, state["budgets"], (2, 1, 1, 8), state["sms"])
        else:
            f.dvc_mcts_step(case["hi"], dvc.DVC_MODE_VALUE if case["value"] else dvc.DVC_MODE_ROLLOUT)
        stats = f.dvc_root_stats()
        return (stats, f.dvc_tree_export(0)) if case["trees"] == 1 else stats
    if kind == "rollout":
        return state["ctx"].dvc_rollout_batch(state["leaves"], case["playouts"], state["seed"], state["trees"],
                                              state["ids"])
    if kind == "determinize":
        return state["ctx"].dvc_determinize(state["roots"], -1, state["seed"], state["trees"], state["ids"])
    if kind == "eval":
        return state["ctx"].dvc_value_eval(state["states"])
    if kind == "train":
        ctx = state["ctx"]
        ctx.dvc_value_train_step(state["states"], state["labels"], LEARNING_RATE, loss=state["loss"])
        return dict(loss=state["loss"].clone(), grads=ctx.dvc_value_grads(), params=ctx.dvc_value_params())
    sv, n = state["server"], case["queries"]
    out = np.zeros((n, 6), dtype=np.int32)
    for root, budget, mode, qid in state["queries"]:
        sv.dvc_server_submit(root, budget, mode, qid)
    got = 0
    while got < n:
        for r in sv.dvc_server_poll(256):
            out[r["query_id"]] = [r["best_action"], r["best_visits"], r["best_wins"], r["root_visits"],
                                  r["iterations"], r["mode"]]
            got += 1
    return out


# -------------------------------------------------------------------- work

def work(case):
    kind = case["kind"]
    if kind in ("search", "serve"):
        n = case["trees"] if kind == "search" else case["queries"]
        lo, hi = case["lo"], case["hi"]
        mean = hi if hi == lo else (hi - lo) / math.log(hi / lo)
        value = (1.0 if case["value"] else 0.0) if kind == "search" else 0.5
        ops = PLAYOUT_OPS[case["variant"]] if kind == "search" else 0.5 * (PLAYOUT_OPS["2p24"] + PLAYOUT_OPS["4p26"])
        return dict(bytes=64 * n + (2 * NPARAMS if value else 0),
                    flops=n * mean * (value * 2 * MACS + (1 - value) * case["playouts"] * ops))
    if kind == "rollout":
        return dict(bytes=case["leaves"] * (32 + 8 + 16),
                    flops=case["leaves"] * case["playouts"] * PLAYOUT_OPS[case["variant"]])
    if kind == "determinize":
        return dict(bytes=case["roots"] * (32 + 8 + 32), flops=0)
    if kind == "eval":
        return dict(bytes=case["rows"] * (32 + 16) + 2 * NPARAMS, flops=2 * MACS * case["rows"])
    # forward, and backward for weights and (but for the first layer) inputs; AdamW reads and writes its three
    # arrays and the gradient is written; the step's gradient and parameters are read back
    return dict(bytes=case["rows"] * (32 + 16) + NPARAMS * 4 * (7 + 4),
                flops=(6 * MACS - 2 * FEATURES * HIDDEN) * case["rows"])


# ------------------------------------------------------------------- exact

def _features64(s):
    """The network's 640 inputs of n records, in 64 bits: per tile the owner
    seat relative to the mover, face down / up, drawn this turn; per opponent
    slot the values it may hold given its face-up numbered neighbours and the
    tiles the mover cannot see."""
    n = s.shape[0]
    dev = s.device
    hand = s[:, :16].contiguous().view(torch.int32).long() & 0xFFFFFFFF
    rev = s[:, 16:20].contiguous().view(torch.int32).long()[:, 0] & 0xFFFFFFFF
    gaps, white = s[:, 20:22].long(), s[:, 22].long() & 1
    cur, drawn, nply, nt = s[:, 23].long(), s[:, 24].long(), s[:, 26].long(), s[:, 27].long()
    t = torch.arange(26, device=dev)
    bit = lambda x: ((x[:, None] >> t) & 1).bool()  # noqa: E731
    up = bit(rev)
    x = torch.zeros((n, FEATURES), dtype=torch.float64, device=dev)
    mine = bit(hand.gather(1, cur[:, None])[:, 0])
    unseen = (t[None, :] < nt[:, None]) & ~mine & ~up
    for r in range(4):
        live = r < nply
        q = torch.where(live, (cur + r) % nply.clamp(min=1), torch.zeros_like(cur))
        has = bit(hand.gather(1, q[:, None])[:, 0]) & live[:, None]
        for i in range(26):
            x[:, 7 * i + r] = has[:, i].double()
            x[:, 7 * i + 4] += (has[:, i] & ~up[:, i]).double()
            x[:, 7 * i + 5] += (has[:, i] & up[:, i]).double()
            x[:, 7 * i + 6] += (has[:, i] & (drawn == i)).double()
        if r == 0:
            continue
        num = has[:, :24]
        rank = num.long().cumsum(1) - num.long()  # numbered tiles of the row left of each tile
        j0, j1, g0, g1 = has[:, 24], has[:, 25], gaps[:, 0], gaps[:, 1]
        first1 = (g1 < g0) | ((g1 == g0) & (white == 1))  # the white joker stands left of the black one
        pos = torch.zeros((n, 26), dtype=torch.long, device=dev)
        pos[:, :24] = rank + (j0[:, None] & (g0[:, None] <= rank)).long() + (j1[:, None] & (g1[:, None] <= rank)).long()
        pos[:, 24] = g0 + (j1 & first1).long()
        pos[:, 25] = g1 + (j0 & ~first1).long()
        ids = torch.arange(24, device=dev)
        for i in range(26):
            left = (ids[None, :] < i) if i < 24 else (rank < (g0 if i == 24 else g1)[:, None])
            right = (ids[None, :] > i) if i < 24 else ~left
            lo = torch.where(num & up[:, :24] & left, ids[None, :], torch.full_like(rank, -1)).amax(1)
            hi = torch.where(num & up[:, :24] & right, ids[None, :], torch.full_like(rank, 24)).amin(1)
            fit = unseen[:, :24] & (ids[None, :] > lo[:, None]) & (ids[None, :] < hi[:, None])
            f = torch.zeros((n, 13), dtype=torch.float64, device=dev)
            f[:, :12] = (fit[:, 0::2] | fit[:, 1::2]).double()
            f[:, 12] = unseen[:, 24:].any(1).double()
            shown = torch.zeros(13, dtype=torch.float64, device=dev)
            shown[i // 2 if i < 24 else 12] = 1.0
            f = torch.where(up[:, i][:, None], shown[None, :], f)
            at = (has[:, i] & (pos[:, i] < 11)).nonzero()[:, 0]
            col = 182 + ((r - 1) * 11 + pos[at, i]) * 13
            for v in range(13):
                x[at, col + v] = f[at, v]
    return x


def _forward64(params, x):
    at, h = 0, x
    for k, (o, i) in enumerate(((HIDDEN, FEATURES), (HIDDEN, HIDDEN), (HIDDEN, HIDDEN), (4, HIDDEN))):
        w, b = params[at:at + o * i].view(o, i), params[at + o * i:at + o * i + o]
        at += o * i + o
        h = h @ w.T + b
        if k < 3:
            h = torch.nn.functional.gelu(h, approximate="tanh")
    return h


def exact(case, seed):
    if case["kind"] not in ("eval", "train"):
        return None
    s = torch.from_numpy(_positions(case["variant"], case["rows"], seed)).cuda()
    np_ = VARIANTS[case["variant"]][0]
    cur = s[:, 23].long()
    seats = (cur[:, None] + torch.arange(np_, device=s.device)[None, :]) % np_
    params = _params(seed).cuda().double()
    x = _features64(s)
    if case["kind"] == "eval":
        out = torch.zeros((case["rows"], 4), dtype=torch.float64, device=s.device)
        out.scatter_(1, seats, torch.softmax(_forward64(params, x)[:, :np_], dim=1))
        return out
    y = torch.from_numpy(_labels(case["variant"], case["rows"], seed)).cuda().double().gather(1, seats)
    params.requires_grad_(True)
    loss = -(y * torch.log_softmax(_forward64(params, x)[:, :np_], dim=1)).sum(1).mean()
    loss.backward()
    g = params.grad
    # the first AdamW step from zero moments: g / (|g| + eps), decay on the matrices
    decay, at = torch.zeros_like(g), 0
    for o, i in ((HIDDEN, FEATURES), (HIDDEN, HIDDEN), (HIDDEN, HIDDEN), (4, HIDDEN)):
        decay[at:at + o * i] = 1e-4
        at += o * i + o
    p = params.detach()
    return dict(loss=loss.detach().reshape(1), grads=g, params=p - LEARNING_RATE * (g / (g.abs() + 1e-8) + decay * p))
