"""Krylov columns of vectors that live in registers for a whole column and of
longer ones: the residual that the recurrence predicts is the true residual
only where the basis is orthonormal.  Sizes on both sides of the lines where a
thread holds more values, one CTA, and beyond the register file."""
import pytest

import problems
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu


# both figures are relative to |b|; they differ by the basis' loss of
# orthogonality, some 1e-14 times the condition of the preconditioned operator
# (below 10), and the cycles' own FP64 rounding
@pytest.mark.parametrize("n", [(9, 7), (278, 279), (280, 279), (394, 395), (395, 395), (1116, 1115), (1117, 1116)])
def test_predicted_residual(n):
    import torch

    import paper_2606_12577_gb300 as cmg
    A = problems.poisson(2, max(n))
    c = A.coeff.reshape(5, A.n[1], A.n[0])[:, :n[1], :n[0]].reshape(5, -1).copy()
    A = problems.Stencil(2, (n[0], n[1], 1), A.offsets, c)
    h = gu.gpu_hierarchy(A)
    cas = cmg.setup_cascade(h, "additive", nu=2)
    g = torch.Generator(device="cuda")
    g.manual_seed(7)
    b = torch.rand(A.N, generator=g, device="cuda", dtype=torch.float64) - 0.5
    for _ in range(2):
        x = torch.zeros_like(b)
        info = cmg.solve(h, cas, b, x, method="gmres_right", tol=1e-6, maxit=30, restart=30)
        assert info.converged and info.iterations >= 3
        assert abs(info.final_rel_residual - info.history[-1]) <= 1e-11
