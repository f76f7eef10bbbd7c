"""Value mode on both sides of the upper line of its chain count: the same search
as with the chain counts by name."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("over", [0, 1])
def test_upper_line(over):
    import paper_2403_10720_gb300 as dvc
    tiles = (torch.cuda.get_device_properties(0).multi_processor_count + 16) // 32
    n = 8 * 128 * tiles + over
    ctx = dvc.Context(dvc.Config(max_predraw=10, playouts=4), 0)
    ctx.dvc_value_init(3)
    roots = ctx.dvc_init_states(5, n)
    got = []
    for chains in (0, 1, 8):
        f = dvc.Forest(ctx, roots, [70] * n, 11)
        if chains:
            f.dvc_forest_tune(0, 0, 0, chains)
        f.dvc_mcts_step(70, mode=dvc.DVC_MODE_VALUE)
        got.append(f.dvc_root_stats().cpu())
        ctx.dvc_check()
        f.close()
    assert torch.equal(got[1], got[0]) and torch.equal(got[2], got[0])
