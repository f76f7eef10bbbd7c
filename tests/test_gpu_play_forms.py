"""Two-player playouts of the fused engine on both sides of the line between
their two forms: the pipeline engine's statistics and counters, bit for bit."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("per_sm,playouts,shape", [(0, 384, (1, 1, 12)), (0, 385, (1, 1, 13)), (0, 1100, (1, 1, 16)),
                                                   (12, 3, (1, 4, 4)), (13, 3, (1, 4, 4)), (14, 32, (1, 14, 14)),
                                                   (12, 32, (1, 12, 12)), (16, 32, (1, 4, 4)), (2, 64, (1, 2, 20)),
                                                   (2, 700, (1, 2, 32))])
@pytest.mark.parametrize("kw", [dict(), dict(vanilla=1), dict(tree_continue=1)])
def test_forms(per_sm, playouts, shape, kw):
    import paper_2403_10720_gb300 as dvc
    n = max(1, per_sm * torch.cuda.get_device_properties(0).multi_processor_count)
    ctx = dvc.Context(dvc.Config(max_predraw=10, playouts=playouts, **kw), 0)
    roots = ctx.dvc_init_states(5, n)
    got = []
    for s in (shape, (2, 0, 0, 0)):
        f = dvc.Forest(ctx, roots, [9] * n, 11)
        f.dvc_forest_tune(*s)
        f.dvc_mcts_step(9)
        got.append((f.dvc_root_stats().cpu(), f.dvc_forest_work().cpu()))
        ctx.dvc_check()
        f.close()
    assert torch.equal(got[0][0], got[1][0]) and torch.equal(got[0][1], got[1][1])
