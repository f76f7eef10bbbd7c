"""The fused engine's counts of random words and game steps over launches of
several stretches of 64 iterations, with trees that end inside them, and over
steps that take more than one launch: the oracle's."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

GAMES = {
    "2p24": dict(nplayers=2, ntiles=24, deal=4, max_predraw=10, max_revealed=5),
    "4p26": dict(nplayers=4, ntiles=26, deal=3, max_predraw=12, max_revealed=4),
}


@pytest.mark.parametrize("game", sorted(GAMES))
@pytest.mark.parametrize("kw,shape", [(dict(playouts=9), (1, 5, 2)), (dict(playouts=33), (1, 2, 16)),
                                      (dict(playouts=1, tree_continue=1), (1, 1, 1)),
                                      (dict(playouts=9, policy=1), (1, 5, 3)),
                                      (dict(playouts=9, vanilla=1), (1, 3, 4))])
def test_counts(game, kw, shape):
    import paper_2403_10720_gb300 as dvc
    kw = dict(GAMES[game], **kw)
    ctx = dvc.Context(dvc.Config(**kw), 0)
    budgets = [200, 64, 65, 0, 129]
    roots = ctx.dvc_init_states(31, len(budgets))
    f = dvc.Forest(ctx, roots, budgets, 6)
    f.dvc_forest_tune(*shape)
    f.dvc_mcts_step(170)
    first = f.dvc_forest_work().cpu().numpy()
    f.dvc_mcts_step(100)
    work = first + f.dvc_forest_work().cpu().numpy()
    ctx.dvc_check()
    f.close()
    cfg = oracle.OracleConfig(**kw)
    total = np.zeros(2, dtype=np.int64)
    for t, b in enumerate(budgets):
        total += oracle.mcts_work(cfg, roots.cpu().numpy()[t], 6, t, b)
    assert (work == total).all()
