"""Playouts at the edges of their two state forms, bit for bit against the
oracle: every player count with and without jokers, pools that run dry, leaves
that do not fill or straddle warps, may-stop and finished leaves, leaves of
another game than the context's, no continue coin."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu

GAMES = {
    "2p24": dict(nplayers=2, ntiles=24, deal=4, max_predraw=10, max_revealed=5),
    "2p24_dry": dict(nplayers=2, ntiles=24, deal=11, max_predraw=2, max_revealed=9),
    "2p26": dict(nplayers=2, ntiles=26, deal=4, max_predraw=10, max_revealed=5),
    "3p24": dict(nplayers=3, ntiles=24, deal=4, max_predraw=9, max_revealed=4),
    "3p26_dry": dict(nplayers=3, ntiles=26, deal=8, max_predraw=2, max_revealed=6),
    "4p24": dict(nplayers=4, ntiles=24, deal=3, max_predraw=8, max_revealed=3),
    "4p26": dict(nplayers=4, ntiles=26, deal=3, max_predraw=12, max_revealed=4),
    "4p26_dry": dict(nplayers=4, ntiles=26, deal=6, max_predraw=2, max_revealed=5),
}


def _u32(a):
    return torch.from_numpy(np.asarray(a, dtype=np.uint32).view(np.int32)).cuda()


def _leaves(game, n, seed):
    s = oracle.init_states(oracle.OracleConfig(**GAMES[game]), seed, n).copy()
    s[1::3, 22] |= 2  # may stop
    return s


@pytest.mark.parametrize("thr", [1 << 31, 0])
@pytest.mark.parametrize("context,leaves", [(g, (g,)) for g in sorted(GAMES)] + [("2p24", tuple(sorted(GAMES)))])
def test_rollouts(context, leaves, thr):
    import paper_2403_10720_gb300 as dvc
    ctx = dvc.Context(dvc.Config(**dict(GAMES[context], cont_thr=thr)), 0)
    each = 7 if len(leaves) > 1 else 40
    states = np.concatenate([_leaves(g, each, 19 + i) for i, g in enumerate(leaves)])
    if len(leaves) > 1:
        states = states[np.random.default_rng(4).permutation(len(states))]
    n = len(states)
    states[5, 28] = 0     # already won by seat 0
    states[6, 28] = 0xFE  # inactive: no credit
    tree, leaf = np.arange(n) * 5 + 3, np.arange(n) * 11 + 1
    for P in (1, 3, 31, 32, 33, 96):
        words = torch.zeros(1, dtype=torch.int64, device="cuda")
        got = ctx.dvc_rollout_batch(torch.from_numpy(states).cuda(), P, (9 << 32) + 77, _u32(tree), _u32(leaf),
                                    words=words).cpu().numpy()
        ctx.dvc_check()
        total = 0
        for i in range(n):
            if i == 5:
                assert got[i].tolist() == [P, 0, 0, 0]
                continue
            if i == 6:
                assert got[i].tolist() == [0, 0, 0, 0]
                continue
            cfg = oracle.OracleConfig(nplayers=int(states[i, 26]), ntiles=int(states[i, 27]), cont_thr=thr)
            want, w = oracle.rollout(cfg, states[i], P, (9 << 32) + 77, int(tree[i]), int(leaf[i]))
            assert (got[i] == want).all(), (P, i)
            total += w
        assert int(words.item()) == total


@pytest.mark.parametrize("game", ["2p24", "3p26_dry", "4p26"])
@pytest.mark.parametrize("P", [1, 7, 33, 150])
def test_pipeline_trees(game, P):
    """Leaves of one search that share warps, in the pipeline engine."""
    import paper_2403_10720_gb300 as dvc
    kw = dict(GAMES[game], playouts=P)
    ctx = dvc.Context(dvc.Config(**kw), 0)
    n, budget = 5, 66
    roots = ctx.dvc_init_states(31, n)
    forest = dvc.Forest(ctx, roots, [budget, budget, 3, budget, 0], 6)
    forest.dvc_forest_tune(2, 2, 0, 2)
    forest.dvc_mcts_step(budget)
    work = forest.dvc_forest_work().cpu().numpy()
    ctx.dvc_check()
    cfg = oracle.OracleConfig(**kw)
    states = roots.cpu().numpy()
    total = np.zeros(2, dtype=np.int64)
    for t, b in enumerate([budget, budget, 3, budget, 0]):
        nodes, _ = oracle.mcts(cfg, states[t], 6, t, b)
        assert (forest.dvc_tree_export(t).cpu().numpy()[:len(nodes)] == nodes).all(), t
        total += oracle.mcts_work(cfg, states[t], 6, t, b)
    assert (work == total).all()
    forest.close()
