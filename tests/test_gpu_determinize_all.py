"""Every determinization of a batch against the oracle, an output that equals its
root included: a root comes back undealt, with the error latched, only where
its view's counting table exceeds the capacity, counted here from the rows."""
import os
import sys

import numpy as np
import pytest
import torch

import oracle

sys.path.insert(0, os.path.dirname(os.path.abspath(__file__)))
from statefmt import decode, encode  # noqa: E402

pytestmark = pytest.mark.gpu

CAPACITY = 32768
GAMES = {
    "2p24": dict(nplayers=2, ntiles=24, deal=9, max_predraw=4, max_revealed=8),
    "2p26": dict(nplayers=2, ntiles=26, deal=5, max_predraw=12, max_revealed=6),
    "3p26_wide": dict(nplayers=3, ntiles=26, deal=6, max_predraw=0, max_revealed=6),
    "4p24": dict(nplayers=4, ntiles=24, deal=3, max_predraw=10, max_revealed=5),
    "4p26": dict(nplayers=4, ntiles=26, deal=4, max_predraw=8, max_revealed=5),
    "4p26_long": dict(nplayers=4, ntiles=26, deal=6, max_predraw=0, max_revealed=2),  # workspace tables
}


def _cells(state, observer):
    """Cells of a view's counting table: per unknown numbered tile (and once after
    them) the open slots of each opponent's gap times the unplaced jokers."""
    s = decode(state)
    obs = s["cur"] if observer < 0 else observer
    unknown = [t for t in range(s["T"]) if t not in s["hands"][obs] and t not in s["revealed"]]
    jokers, numbered = sum(t >= 24 for t in unknown), [t for t in unknown if t < 24]
    gaps, anchors = [], []
    for k in range(1, s["P"]):
        row, gap, size = s["hands"][(obs + k) % s["P"]], 0, [0]
        for t in row:
            if t not in s["revealed"]:
                size[-1] += 1
            elif t < 24:
                size.append(0)
        gaps.append(size)
        anchors.append([t for t in row if t < 24 and t in s["revealed"]])
    total = 0
    for u in numbered + [24]:
        n = jokers + 1
        for size, up in zip(gaps, anchors):
            n *= size[sum(a < u for a in up)] + 1
        total += n
    return total


def _over():
    """Two tiles against three rows of eight, all face down: 50,301 cells."""
    rest = [t for t in range(26) if t not in (3, 17)]
    np.random.default_rng(5).shuffle(rest)
    hands = [[3, 17]] + [sorted(rest[8 * k:8 * k + 8]) for k in range(3)]
    return encode(hands, set(), cur=0, ntiles=26)


def _u32(a):
    return torch.from_numpy(np.asarray(a, dtype=np.uint32).view(np.int32)).cuda()


@pytest.mark.parametrize("game", sorted(GAMES))
@pytest.mark.parametrize("n", [1, 2, 150, 530])
def test_every_output(game, n):
    import paper_2403_10720_gb300 as dvc
    kw = GAMES[game]
    cfg = oracle.OracleConfig(**kw)
    ctx = dvc.Context(dvc.Config(**kw), 0)
    roots = oracle.init_states(cfg, 67 + n, n)
    if game == "4p26_long":
        roots[n // 2] = _over()
    rng = np.random.default_rng(3)
    tree = rng.integers(0, 1 << 31, size=n).astype(np.uint32)
    it = rng.integers(0, 1 << 31, size=n).astype(np.uint32)
    for observer in range(-1, kw["nplayers"]):
        got = ctx.dvc_determinize(torch.from_numpy(roots).cuda(), observer, 5, _u32(tree), _u32(it)).cpu().numpy()
        latched = None
        try:
            ctx.dvc_check()
        except dvc.DvcError as e:
            latched = e.code
        over = [_cells(r, observer) > CAPACITY for r in roots]
        assert latched == (-5 if any(over) else None)
        assert sum(over) == (1 if game == "4p26_long" and observer <= 0 else 0)
        for i in range(n):
            want = roots[i] if over[i] else oracle.determinize(cfg, roots[i], observer, 5, int(tree[i]), int(it[i]))
            assert (got[i] == want).all(), (observer, i)
