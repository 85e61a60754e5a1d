"""Steps of 2x2-node blocks with several right-hand sides on a grid of more
than 65,535 block rows, the most that a launch grid's y counts, against the
single-column step of the same level."""
import numpy as np
import pytest

import problems
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,fp32", [(4, True), (8, True), (3, True), (2, True), (2, False), (1, False)])
def test_rhs_steps_of_a_tall_grid(m, fp32):
    import torch

    import paper_2606_12577_gb300 as cmg
    n = (5, 140001, 1)
    N = n[0] * n[1]
    offs = problems._star_offsets(2)
    c = np.full((5, N), -1.0)
    c[0] = 4.0 + problems.uniform01(2, N)
    A = problems.Stencil(2, n, offs, c)
    h = gu.gpu_hierarchy(A, block=2, max_levels=1)
    cas = cmg.setup_cascade(h, "additive", nu=1, lowp=True)
    dt = torch.float32 if fp32 else torch.float64
    B = torch.from_numpy(problems.uniform(31, N * m)).cuda().to(dt).reshape(N, m)
    X = torch.from_numpy(problems.uniform(32, N * m)).cuda().to(dt).reshape(N, m)
    out = torch.empty_like(X)
    cmg.sweep_rhs(h, cas, 0, 0, B, X, out, m)
    for r in range(m):
        one = torch.empty(N, dtype=dt, device="cuda")
        cmg.sweep(h, cas, 0, 0, B[:, r].contiguous(), X[:, r].contiguous(), one)
        # both sum five products and then four, in FP32 or FP64: a dozen roundings of terms of about 10
        assert float((out[:, r] - one).abs().max()) <= 120 * torch.finfo(dt).eps
