"""Search steps captured into a caller's CUDA graph: the forests whose size takes
the pipeline engine as well as those that take the fused one, steps of more and
fewer iterations than a chunk of the pipeline's own graph; replayed twice, the
statistics of the same steps launched plainly."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,kw", [(8, dict(playouts=16)), (400, dict(playouts=256)), (3, dict(playouts=40000)),
                                  (400, dict(playouts=256, policy=1)), (700, dict(playouts=120, vanilla=1))])
@pytest.mark.parametrize("iterations", [9, 70])
def test_captured_step(n, kw, iterations):
    import paper_2403_10720_gb300 as dvc
    ctx = dvc.Context(dvc.Config(max_predraw=10, **kw), 0)
    roots = ctx.dvc_init_states(3, n)
    budgets = [2 * iterations] * n

    def plain():
        f = dvc.Forest(ctx, roots, budgets, 5)
        f.dvc_mcts_step(iterations)
        f.dvc_mcts_step(iterations)
        s = f.dvc_root_stats().cpu()
        f.close()
        return s

    want = plain()
    f = dvc.Forest(ctx, roots, budgets, 5)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        f.dvc_mcts_step(iterations)
    g.replay()
    g.replay()
    assert torch.equal(f.dvc_root_stats().cpu(), want)
    ctx.dvc_check()
    del g
    f.close()
