"""One application of a 2D point cascade in one launch: tiles with a halo as
wide as the number of steps.  Against the single steps (cs_sweep), bit for
bit, on grids narrower than a tile, at tile edges (the tiles' middles are 32 -
2 H and 64 - 2 H wide), above and below the size where the larger tiles start,
forward and reverse, 5- and 9-point levels, depths up to the widest halo."""
import pytest

import problems
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,kind,nu", [
    ((5, 7), "additive", 3), ((26, 53), "additive", 3), ((27, 25), "multiplicative", 2), ((61, 20), "multiplicative", 3),
    ((41, 33), "multiplicative", 4), ((300, 257), "multiplicative", 3), ((52, 1400), "multiplicative", 3),
    ((313, 290), "additive", 4), ((130, 129), "additive", 2)])
def test_application_equals_steps(n, kind, nu):
    import torch

    import paper_2606_12577_gb300 as cmg
    big = problems.variable_poisson(problems.random_coefficients(2, max(n), 3, -1.0, 1.0))
    c = big.coeff.reshape(5, big.n[1], big.n[0])[:, :n[1], :n[0]].reshape(5, -1).copy()
    A = problems.Stencil(2, (n[0], n[1], 1), big.offsets, c)
    h = gu.gpu_hierarchy(A)
    cas = cmg.setup_cascade(h, kind, nu=nu, lowp=True)
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    for l in range(min(2, h.nlevels - 1)):
        b = torch.rand(h.N(l), generator=g, device="cuda", dtype=torch.float64) - 0.5
        x0 = torch.rand(h.N(l), generator=g, device="cuda", dtype=torch.float64) - 0.5
        for reverse in (False, True):
            x = x0.clone()
            cmg.smooth(h, cas, l, b, x, reverse=reverse)
            y = x0.clone()
            for st in range(nu):
                lv = nu - 1 - st if reverse else st
                for col in (((1, 0) if reverse else (0, 1)) if kind == "multiplicative" else (-1,)):
                    out = torch.empty_like(y)
                    cmg.sweep(h, cas, l, lv, b, y, out, colour=col)
                    y = out
            assert torch.equal(x, y)
    # FP32: a cycle (which takes the launch) against the same cycle in FP64
    b = torch.rand(A.N, generator=g, device="cuda", dtype=torch.float64) - 0.5
    xs = []
    for prec in ("fp32", "fp64"):
        x = torch.zeros(A.N, dtype=torch.float64, device="cuda")
        cmg.vcycle(h, cas, b, x, mu_pre=2, mu_post=1, precision=prec)
        xs.append(x)
    # 30-odd FP32 roundings per level and step over O(10) levels and steps, relative to the largest value
    assert float((xs[0] - xs[1]).abs().max()) <= 1e-4 * float(xs[1].abs().max())
