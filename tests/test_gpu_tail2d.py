"""The small 2D levels of a cycle in one launch: FP64 cycles against the
oracle's and FP32 ones against FP64, on grids on both sides of the lines where
the launch starts (16^2 and 32^2 nodes), narrow ones, both kinds and orders,
without pre- or post-smoothing."""
import numpy as np
import pytest

import oracle
import problems
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,kind,nu", [
    ((5, 4), "additive", 2), ((16, 16), "multiplicative", 1), ((17, 16), "additive", 3), ((33, 31), "multiplicative", 3),
    ((64, 4), "additive", 4), ((3, 70), "multiplicative", 2), ((32, 32), "additive", 3), ((40, 65), "additive", 2)])
def test_cycles(n, kind, nu):
    import torch

    import paper_2606_12577_gb300 as cmg
    big = problems.variable_poisson(problems.random_coefficients(2, max(n), 3, -1.0, 1.0))
    c = big.coeff.reshape(5, big.n[1], big.n[0])[:, :n[1], :n[0]].reshape(5, -1).copy()
    A = problems.Stencil(2, (n[0], n[1], 1), big.offsets, c)
    ho = oracle.Hierarchy(A)
    co = oracle.Cascade(ho, kind, nu=nu)
    h = gu.gpu_hierarchy(A)
    cas = cmg.setup_cascade(h, kind, nu=nu, lowp=True)
    b = problems.rhs(A.N, 3)
    bd = torch.from_numpy(b).cuda()
    for pre, post, rf in ((1, 1, True), (2, 1, False), (1, 0, True), (0, 1, True)):
        ref = oracle.vcycle(ho, co, b, None, pre, post, rf)
        # FP64: the oracle's own tolerance; FP32: 30-odd roundings per level and step over O(10) levels and
        # steps; both relative to the largest value that a cycle without one of its smoothings may amplify
        for prec, tol in (("fp64", 1e-12), ("fp32", 1e-4)):
            x = torch.zeros(A.N, dtype=torch.float64, device="cuda")
            cmg.vcycle(h, cas, bd, x, mu_pre=pre, mu_post=post, order="RF" if rf else "FF", precision=prec)
            assert gu.rel_max(x.cpu().numpy(), ref) <= tol, (pre, post, rf, prec)
