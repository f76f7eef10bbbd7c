"""Network inference at batch sizes on both sides of its two paths (one launch
of clusters, layer by layer), with ragged tiles: the same bits for the same
state whatever batch it is in, rows beyond the batch untouched."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu

KW = dict(nplayers=4, ntiles=26, deal=3, max_predraw=8, max_revealed=3)


def test_batches_agree():
    import paper_2403_10720_gb300 as dvc
    ctx = dvc.Context(dvc.Config(**KW), 0)
    ctx.dvc_value_init(21)
    n = 20000
    other = [dict(nplayers=2, ntiles=24, deal=4, max_predraw=10, max_revealed=5),
             dict(nplayers=3, ntiles=26, deal=4, max_predraw=6, max_revealed=3)]
    states = oracle.init_states(oracle.OracleConfig(**KW), 5, n)
    for k, kw in enumerate(other):   # every variant in one batch
        states[k::3] = oracle.init_states(oracle.OracleConfig(**kw), 7 + k, n)[:len(states[k::3])]
    states = torch.from_numpy(states).cuda()
    whole = ctx.dvc_value_eval(states)   # layer by layer
    ctx.dvc_check()
    assert (whole.sum(1) - 1).abs().max().item() < 1e-5
    for size in (1, 31, 127, 128, 129, 333, 1000, 2944, 4096, 5000):
        for start in (0, 777):
            out = torch.full((size + 1, 4), -7.0, device="cuda")
            ctx.dvc_value_eval(states[start:start + size], out=out)
            ctx.dvc_check()
            assert torch.equal(out[:size], whole[start:start + size]), (size, start)
            assert bool((out[size] == -7.0).all())


def test_against_oracle():
    import paper_2403_10720_gb300 as dvc
    ctx = dvc.Context(dvc.Config(**KW), 0)
    ctx.dvc_value_init(8)
    p = ctx.dvc_value_params().cpu().to(torch.bfloat16).float()
    ctx.dvc_value_params(p.cuda())
    states = oracle.init_states(oracle.OracleConfig(**KW), 29, 200)
    got = ctx.dvc_value_eval(torch.from_numpy(states).cuda()).cpu().numpy()
    # three BF16 activation roundings (relative 2^-8 each) through 512-wide dot
    # products of O(1) terms and a softmax: the bound of the layer path's test
    for i in range(0, 200, 7):
        assert np.abs(got[i] - oracle.value_forward(p.numpy(), states[i])).max() < 1.5e-2, i
