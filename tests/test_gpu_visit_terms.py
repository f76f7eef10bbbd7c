"""UCB1 terms by visits: searches past the end of the table (2^17
backpropagations through a node, the root first) in both engines, and with 2^20
playouts a leaf, node by node against the oracle."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("playouts,engine", [(1, 1), (3, 2)])
def test_past_the_table(playouts, engine):
    import paper_2403_10720_gb300 as dvc
    kw = dict(nplayers=2, ntiles=24, deal=4, max_predraw=12, max_revealed=9, playouts=playouts)
    ctx, ocfg = dvc.Context(dvc.Config(**kw), 0), oracle.OracleConfig(**kw)
    roots, oroots = ctx.dvc_init_states(3, 2), oracle.init_states(ocfg, 3, 2)
    budgets = [(1 << 17) + 900, 1]
    f = dvc.Forest(ctx, roots, budgets, 8)
    f.dvc_forest_tune(engine, 0, 0, 0)
    f.dvc_mcts_step(budgets[0])
    ctx.dvc_check()
    for t in range(2):
        nodes, _ = oracle.mcts(ocfg, oroots[t], 8, t, budgets[t])
        assert np.array_equal(f.dvc_tree_export(t).cpu().numpy()[: len(nodes)], nodes)
    f.close()


def test_many_playouts_short_table():
    """2^20 playouts a leaf: 2,047 entries are all whose visits fit an int."""
    import paper_2403_10720_gb300 as dvc
    kw = dict(nplayers=2, ntiles=24, deal=11, max_predraw=2, max_revealed=9, playouts=1 << 20)
    ctx, ocfg = dvc.Context(dvc.Config(**kw), 0), oracle.OracleConfig(**kw)
    f = dvc.Forest(ctx, ctx.dvc_init_states(3, 1), [4], 8)
    f.dvc_mcts_step(4)
    ctx.dvc_check()
    nodes, _ = oracle.mcts(ocfg, oracle.init_states(ocfg, 3, 1)[0], 8, 0, 4)
    assert np.array_equal(f.dvc_tree_export(0).cpu().numpy()[: len(nodes)], nodes)
    f.close()
