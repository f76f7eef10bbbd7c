"""The default engine on both sides of its line (512 playouts per SM): the same
searches as either engine by name, counters and statistics bit for bit; and
value mode, whose default chain count changes with the forest's size."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kw", [dict(playouts=32), dict(playouts=5), dict(playouts=32, policy=1),
                                dict(playouts=32, vanilla=1), dict(playouts=5, tree_continue=1)])
@pytest.mark.parametrize("over", [0, 1])
def test_default_engine(kw, over):
    import paper_2403_10720_gb300 as dvc
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n = 512 * sms // max(kw["playouts"], 128 if kw.get("policy") else 16) + over
    ctx = dvc.Context(dvc.Config(nplayers=3, ntiles=26, deal=4, max_predraw=9, max_revealed=4, **kw), 0)
    roots = ctx.dvc_init_states(5, n)
    budgets = [6 + (7 * i) % 5 for i in range(n)]
    got = []
    for shape in (None, (1, 0, 0, 0), (2, 0, 0, 0)):
        f = dvc.Forest(ctx, roots, budgets, 11)
        if shape:
            f.dvc_forest_tune(*shape)
        f.dvc_mcts_step(7)
        f.dvc_mcts_step(10)
        got.append((f.dvc_root_stats().cpu(), f.dvc_forest_counters().cpu()))
        ctx.dvc_check()
        f.close()
    for s, c in got[1:]:
        assert torch.equal(s, got[0][0]) and torch.equal(c, got[0][1])


@pytest.mark.parametrize("over", [0, 1])
def test_value_chains(over):
    import paper_2403_10720_gb300 as dvc
    n = 16 * torch.cuda.get_device_properties(0).multi_processor_count + over
    ctx = dvc.Context(dvc.Config(max_predraw=10, playouts=4), 0)
    ctx.dvc_value_init(3)
    roots = ctx.dvc_init_states(5, n)
    got = []
    for chains in (0, 1, 8):
        f = dvc.Forest(ctx, roots, [40] * n, 11)
        if chains:
            f.dvc_forest_tune(0, 0, 0, chains)
        f.dvc_mcts_step(40, mode=dvc.DVC_MODE_VALUE)
        got.append((f.dvc_root_stats().cpu(), f.dvc_forest_counters().cpu()))
        ctx.dvc_check()
        f.close()
    for s, c in got[1:]:
        assert torch.equal(s, got[0][0]) and torch.equal(c, got[0][1])
