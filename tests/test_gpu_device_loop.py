"""Stationary solves whose loop runs on the device: one call equals two calls
that share its iterations, bit for bit, also beyond the history that the
device keeps, with host and device vectors; limits and finished systems."""
import numpy as np
import pytest

import problems
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,n,method,precision", [
    (2, 12, "stationary", "fp64"), (2, 40, "refine", "fp32"), (3, 17, "stationary", "fp64"), (2, 33, "refine", "bf16")])
def test_split_solves_agree(dim, n, method, precision):
    import torch

    import paper_2606_12577_gb300 as cmg
    A = problems.poisson(dim, n)
    h = gu.gpu_hierarchy(A)
    c = cmg.setup_cascade(h, "additive", nu=2, lowp=2 if precision == "bf16" else True)
    b = problems.uniform(5, A.N)

    def solve(x, maxit, tol=1e-30, host=False):
        bb = b if host else torch.from_numpy(b).cuda()
        return cmg.solve(h, c, bb, x, method=method, precision=precision, tol=tol, maxit=maxit, host_buffers=host,
                         raise_on_error=False)

    x1 = torch.zeros(A.N, dtype=torch.float64, device="cuda")
    one = solve(x1, 300)
    x2 = torch.zeros_like(x1)
    first, second = solve(x2, 130), solve(x2, 170)
    assert (one.iterations, first.iterations, second.iterations) == (300, 130, 170) and not one.converged
    assert len(one.history) == 301 and torch.equal(x1, x2)
    assert np.array_equal(one.history, np.concatenate([first.history, second.history[1:]]))
    x3 = np.zeros(A.N)
    assert solve(x3, 300, host=True).iterations == 300 and np.array_equal(x3, x1.cpu().numpy())
    done = solve(x1, 10, tol=1e-6)
    assert done.converged and done.iterations == 0 and torch.equal(x1, x2)
