"""Launches that overlap the one before them: training steps and evaluations on
both sides of the line (a GEMM tile per SM), evaluations back to back into the
same buffers, and evaluations captured into a graph."""
import pytest
import torch

import test_gpu_train_edges as edges

pytestmark = pytest.mark.gpu


def _rows(over):
    """Rows that fill one 128 x 256 tile per SM (512 columns), or one more."""
    return torch.cuda.get_device_properties(0).multi_processor_count // 2 * 128 + over


@pytest.mark.parametrize("over", [0, 1])
def test_train_step(over):
    edges.test_gradients(_rows(over))


@pytest.mark.parametrize("over", [None, 0, 1])
def test_evaluations(over):
    import paper_2403_10720_gb300 as dvc
    n = 300 if over is None else _rows(over)
    ctx = dvc.Context(dvc.Config(**edges.KW), 0)
    ctx.dvc_value_init(13)
    sets = [ctx.dvc_init_states(s, n) for s in range(4)]
    want = [ctx.dvc_value_eval(s).cpu() for s in sets]  # one at a time
    batch = torch.cat([s[:64] for s in sets])
    assert torch.equal(ctx.dvc_value_eval(batch).cpu(), torch.cat([w[:64] for w in want]))
    got = [ctx.dvc_value_eval(s) for s in sets]  # back to back
    assert all(torch.equal(g.cpu(), w) for g, w in zip(got, want))
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        got = [ctx.dvc_value_eval(s) for s in sets]
    for _ in range(3):
        g.replay()
    torch.cuda.synchronize()
    ctx.dvc_check()
    assert all(torch.equal(g_.cpu(), w) for g_, w in zip(got, want))
