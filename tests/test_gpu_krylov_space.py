"""The Krylov space that a cascade keeps between solves."""
import pytest

import problems
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu

HUGE = 700_000  # restart: 360 GB of basis vectors on 255^2 nodes, more than the device has


def _same(f, g):
    """Solves f and g give the same bits in the same number of steps, converged."""
    import torch
    (i, x), (j, y) = f(), g()
    assert i.converged and j.converged and i.iterations == j.iterations and torch.equal(x, y)
    return i


@pytest.mark.parametrize("method", ["gmres", "gmres_right"])
def test_solve_after_a_failed_allocation(method):
    import torch

    import paper_2606_12577_gb300 as cmg
    A = problems.poisson(2, 256)
    h = gu.gpu_hierarchy(A)
    b = torch.from_numpy(problems.rhs(A.N, 3)).cuda()

    def run(c, restart):
        x = torch.zeros_like(b)
        return cmg.solve(h, c, b, x, method=method, restart=restart, tol=1e-8, raise_on_error=False), x
    c = cmg.setup_cascade(h, "additive", nu=2)
    run(c, 30)
    info, _ = run(c, HUGE)
    assert not info.converged and info.status != 0
    _same(lambda: run(c, 10), lambda: run(cmg.setup_cascade(h, "additive", nu=2), 10))


def test_general_solve_after_a_failed_allocation():
    import torch

    import paper_2606_12577_gb300 as cmg
    u = problems.unstructured_q1(255, 3)
    h = cmg.gsetup_hierarchy(u["A"], u["Ps"], rscale=0.25)
    b = torch.from_numpy(problems.rhs(u["A"].shape[0], 3)).cuda()

    def run(c, restart):
        x = torch.zeros_like(b)
        return cmg.gsolve(h, c, b, x, restart=restart, tol=1e-8, raise_on_error=False), x
    c = cmg.gsetup_cascade(h, "additive", nu=2)
    run(c, 30)
    info, _ = run(c, HUGE)
    assert not info.converged and info.status != 0
    _same(lambda: run(c, 10), lambda: run(cmg.gsetup_cascade(h, "additive", nu=2), 10))


def test_right_solve_after_a_longer_left_one():
    """Z of a right solve of restart 4 does not serve one of restart 12 after a left solve of restart 30 made V longer."""
    import torch

    import paper_2606_12577_gb300 as cmg
    A = problems.variable_poisson(problems.random_coefficients(2, 120, 3, -1.5, 1.5))
    h = gu.gpu_hierarchy(A)
    b = torch.from_numpy(problems.rhs(A.N, 3)).cuda()

    def run(c, method, restart):
        x = torch.zeros_like(b)
        return cmg.solve(h, c, b, x, method=method, restart=restart, tol=1e-9, maxit=300), x
    c = cmg.setup_cascade(h, "additive", nu=1)
    run(c, "gmres_right", 4)
    run(c, "gmres", 30)
    info = _same(lambda: run(c, "gmres_right", 12), lambda: run(cmg.setup_cascade(h, "additive", nu=1), "gmres_right", 12))
    assert info.iterations > 4
