"""A training step captured into a caller's CUDA graph when all that the process has
done before is one evaluation of as many rows: the parameters, gradients and
loss of the same step launched plainly, bit for bit.  In a process of its own,
since launch attributes outlast the calls that set them."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r'''
import torch
import paper_2403_10720_gb300 as dvc
n = 300
def context():
    c = dvc.Context(dvc.Config(nplayers=3, ntiles=26, deal=4, max_predraw=6, max_revealed=3), 0)
    c.dvc_value_init(13)
    return c
def result(c, loss):
    return [loss, c.dvc_value_params(), c.dvc_value_grads()]
a = context()
states = a.dvc_init_states(3, n)
labels = torch.zeros((n, 4), device="cuda")
labels[:, :3] = torch.rand((n, 3), device="cuda").softmax(1)
a.dvc_value_eval(states)
loss = torch.zeros(1, device="cuda")
torch.cuda.synchronize()
g = torch.cuda.CUDAGraph()
with torch.cuda.graph(g):
    a.dvc_value_train_step(states, labels, 1e-3, loss=loss)
g.replay()
got = result(a, loss)
b = context()
other = torch.zeros(1, device="cuda")
b.dvc_value_train_step(states, labels, 1e-3, loss=other)
for x, y in zip(got, result(b, other)):
    assert torch.equal(x, y)
a.dvc_check()
b.dvc_check()
print("same")
'''


def test_step_captured_after_an_evaluation():
    r = subprocess.run([sys.executable, "-c", SRC], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.split()[-1:] == ["same"], r.stderr[-2000:]
