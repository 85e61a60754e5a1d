"""The network's loss: no thread adds more than every 65,536th square in FP32,
whatever the shape of the outputs.  The sum bit for bit, from its order:
65,536 chains of fused multiply-adds, 256 trees of 256 chains, one tree."""
import numpy as np
import pytest

import problems
from tests.test_gpu_fp32_sums import _fma32

pytestmark = pytest.mark.gpu


def _tree(v):
    v = v.copy()
    while v.shape[-1] > 1:
        h = v.shape[-1] // 2
        v = v[..., :h] + v[..., h:]
    return v[..., 0]


@pytest.mark.parametrize("nout,batch", [(1, 70001), (16, 4096), (48, 8193), (81, 1000), (243, 257), (243, 4096)])
def test_loss_sum(nout, batch):
    import torch

    import paper_2606_12577_gb300 as cmg
    m = cmg.MLP(8, 16, nout, max_batch=batch, seed=1)
    m.set_params(np.zeros(m.nparam, np.float32))  # Y = 0: the errors are the targets
    T = problems.uniform(7, batch * nout).astype(np.float32)
    X = torch.zeros(batch, 8, device="cuda")
    loss, _ = m.gradients(X, torch.from_numpy(T).cuda().reshape(batch, nout))
    pad = np.zeros(-(-T.size // 65536) * 65536, np.float32)
    pad[:T.size] = T
    v = np.zeros(65536, np.float32)
    for row in pad.reshape(-1, 65536):
        v = _fma32(row, row, v)
    assert np.float32(loss) == _tree(_tree(v.reshape(256, 256))) / np.float32(T.size)
