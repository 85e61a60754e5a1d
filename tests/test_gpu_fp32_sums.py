"""How many FP32 terms are added up before FP64 takes over: the squares of a
convergence norm, a CTA's nodes of one plane."""
import numpy as np
import pytest

import problems
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu


def test_convergence_norm_adds_planes_in_fp64():
    """r = b with values 4096 and 1 in planes of their own: squares 2^24 and 1.
    The sums of a plane's 256 equal squares are exact in FP32, and so are the
    norms in FP64; 2^24 + 1 is not an FP32 number."""
    import torch

    import paper_2606_12577_gb300 as cmg
    A = problems.poisson(3, 66)
    h = gu.gpu_hierarchy(A)
    c = cmg.setup_cascade(h, "additive", nu=1, lowp=True)
    for shift in range(4):
        iz = np.arange(A.N) // (66 * 66)
        b = torch.from_numpy(np.where(iz % 4 == shift, 4096.0, 1.0)).cuda()
        x = torch.zeros_like(b)
        info = cmg.solve(h, c, b, x, method="refine", precision="fp32", maxit=1, raise_on_error=False)
        assert info.history[0] == 1.0
