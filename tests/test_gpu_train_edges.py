"""Training steps whose rows do not fill tiles or row splits: gradients and the
loss against a plain FP64 evaluation of the network on the same BF16 weights.

Each gradient element sums products of BF16-rounded factors (relative 2^-9);
the first layer's passes through up to six such roundings: sqrt(6) 2^-9 = 4.8e-3
relative per tensor; the bound is three times that, as for the oracle's check."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu

KW = dict(nplayers=3, ntiles=26, deal=4, max_predraw=6, max_revealed=3)
SHAPES = ((512, 640), (512, 512), (512, 512), (4, 512))


@pytest.mark.parametrize("n", [1, 64, 129, 300, 1000])
def test_gradients(n):
    import paper_2403_10720_gb300 as dvc
    ctx = dvc.Context(dvc.Config(**KW), 0)
    ctx.dvc_value_init(13)
    p = ctx.dvc_value_params().cpu().to(torch.bfloat16).float()
    ctx.dvc_value_params(p.cuda())
    states = torch.from_numpy(oracle.init_states(oracle.OracleConfig(**KW), 3, n)).cuda()
    y = torch.from_numpy(np.random.default_rng(n).dirichlet(np.ones(3), size=n))
    labels = torch.zeros((n, 4), dtype=torch.float32)
    labels[:, :3] = y.float()
    loss = torch.zeros(1, device="cuda")
    ctx.dvc_value_train_step(states, labels.cuda(), 0.0, loss=loss)
    got = ctx.dvc_value_grads().cpu().double()
    ctx.dvc_check()
    x = ctx.dvc_value_features(states).cpu().double()
    q = p.double().requires_grad_(True)
    at, h = 0, x
    for k, (o, i) in enumerate(SHAPES):
        h = h @ q[at:at + o * i].view(o, i).T + q[at + o * i:at + o * i + o]
        at += o * i + o
        if k < 3:
            h = torch.nn.functional.gelu(h, approximate="tanh")
    seats = (states[:, 23].cpu().long()[:, None] + torch.arange(3)) % 3
    want = -(labels.double().gather(1, seats) * torch.log_softmax(h[:, :3], dim=1)).sum(1).mean()
    want.backward()
    assert abs(loss.item() - want.item()) < 1e-2 * want.item()
    at = 0
    for o, i in SHAPES:
        for size in (o * i, o):
            g, w = got[at:at + size], q.grad[at:at + size]
            assert (g - w).norm() <= 1.5e-2 * w.norm(), (at, size)
            at += size
