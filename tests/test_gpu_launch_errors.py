"""A launch that the runtime refuses is that call's error alone: the calls
after it run."""
import numpy as np
import pytest

import problems
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu


def test_call_after_a_refused_launch():
    import torch

    import paper_2606_12577_gb300 as cmg
    from paper_2606_12577_gb300 import _capi
    n = (5, 200001, 1)  # 66,667 block rows: more than a launch grid's y counts
    N = n[0] * n[1]
    offs = problems._star_offsets(2)
    c = np.full((5, N), -1.0)
    c[0] = 4.0
    h = gu.gpu_hierarchy(problems.Stencil(2, n, offs, c), block=3, max_levels=1)
    cas = cmg.setup_cascade(h, "additive", nu=1)
    B = torch.ones(N, 2, dtype=torch.float64, device="cuda")
    X, out = torch.zeros_like(B), torch.empty_like(B)
    with pytest.raises(_capi.CascadeError):
        cmg.sweep_rhs(h, cas, 0, 0, B, X, out, 2)
    one = torch.full((N,), np.nan, dtype=torch.float64, device="cuda")
    cmg.sweep(h, cas, 0, 0, B[:, 0].contiguous(), X[:, 0].contiguous(), one)
    assert bool((one > 0).all())
    gu.gpu_hierarchy(problems.poisson(2, 8))
