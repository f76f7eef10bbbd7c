"""What dvc_determinize takes of the device's memory, and what it does without
its second half: calls of few roots hold 64 MB of tables, and a call of many
roots whose memory is spent, or that is being captured, gives the same records."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

KW = dict(nplayers=3, ntiles=26, deal=6, max_predraw=0, max_revealed=6)  # tables beyond shared memory


def _ids(n, seed):
    return torch.from_numpy(np.random.default_rng(seed).integers(0, 1 << 30, size=n).astype(np.int32)).cuda()


def _free():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def test_workspace():
    import paper_2403_10720_gb300 as dvc
    n = 700
    a = dvc.Context(dvc.Config(**KW), 0)
    roots, tree, it = a.dvc_init_states(9, n), _ids(n, 1), _ids(n, 2)
    out = torch.empty_like(roots)
    want = a.dvc_determinize(roots, -1, 5, tree, it).clone()  # both halves; the kernels are loaded
    b = dvc.Context(dvc.Config(**KW), 0)
    before = _free()
    b.dvc_determinize(roots[:200], -1, 5, tree[:200], it[:200], out=out[:200])
    assert before - _free() <= (64 << 20) + (4 << 20)
    assert torch.equal(out[:200], want[:200])
    # captured before a call has allocated the second half
    out.zero_()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        b.dvc_determinize(roots, -1, 5, tree, it, out=out)
    g.replay()
    assert torch.equal(out, want)
    out.zero_()
    before = _free()  # the capture took none of the second half, so the plain call does
    b.dvc_determinize(roots, -1, 5, tree, it, out=out)
    assert before - _free() >= 64 << 20
    assert torch.equal(out, want)
    a.dvc_check()
    b.dvc_check()
