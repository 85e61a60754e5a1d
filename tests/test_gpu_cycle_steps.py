"""Cycles on 2D point levels, where an application is one launch (FP32: tiles
of 64 x 48 above 256^2 nodes, 32 x 32 below; FP64: 16 x 16) and the small
levels are one launch in all, against the same cycle from single steps: bit
for bit."""
import pytest

import problems
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu


def _cycle(cmg, torch, h, c, l, b, kind, nu, pre, post, rf):
    """V(0, b) from level l in b's precision, step by step."""
    fp64 = b.dtype == torch.float64
    if l == h.nlevels - 1:
        xd = torch.empty(h.N(l), dtype=torch.float64, device="cuda")
        cmg.coarse_solve(h, b.double(), xd)
        return xd.to(b.dtype)
    x = torch.zeros_like(b)

    def smooth(x, reverse):
        for st in range(nu):
            lv = nu - 1 - st if reverse else st
            for col in (((1, 0) if reverse else (0, 1)) if kind == "multiplicative" else (-1,)):
                out = torch.empty_like(x)
                cmg.sweep(h, c, l, lv, b, x, out, colour=col)
                x = out
        return x

    for _ in range(pre):
        x = smooth(x, rf)
    rc = torch.empty(h.N(l + 1), dtype=b.dtype, device="cuda")
    cmg.residual_restrict(h, l, b, x, rc) if fp64 else cmg.residual_restrict_lowp(h, c, l, b, x, rc)
    xc = _cycle(cmg, torch, h, c, l + 1, rc, kind, nu, pre, post, rf)
    cmg.prolong_correct(h, l, xc, x) if fp64 else cmg.prolong_correct_lowp(h, c, l, xc, x)
    for _ in range(post):
        x = smooth(x, False)
    return x


# FP32: 6 and 8 steps deep; sides at a tile's middle (32 - 2 H, 64 - 2 H and 48 - 2 H), next to it, and narrow ones.
# FP64: up to 4 steps and 304 tiles, on levels of 5 points (the finest) and of 9.
@pytest.mark.parametrize("n,kind,nu,prec", [
    ((300, 257), "multiplicative", 3, "fp32"), ((52, 1400), "multiplicative", 3, "fp32"),
    ((313, 290), "multiplicative", 4, "fp32"), ((289, 289), "additive", 4, "fp32"), ((260, 253), "additive", 3, "fp32"),
    ((9, 8000), "multiplicative", 4, "fp32"), ((61, 20), "multiplicative", 3, "fp32"),
    ((41, 33), "multiplicative", 4, "fp32"), ((160, 159), "multiplicative", 2, "fp32"),
    ((136, 137), "multiplicative", 2, "fp64"), ((200, 190), "multiplicative", 1, "fp64"), ((135, 130), "additive", 4, "fp64"),
    ((24, 9), "multiplicative", 2, "fp64")])
def test_cycle_equals_steps(n, kind, nu, prec):
    import torch

    import paper_2606_12577_gb300 as cmg
    m = max(min(n), 300)
    big = problems.variable_poisson(problems.random_coefficients(2, m, 3, -1.0, 1.0))
    c = big.coeff.reshape(5, m, m)
    c = c[:, [y % m for y in range(n[1])]][:, :, [x % m for x in range(n[0])]].reshape(5, -1).copy()
    A = problems.Stencil(2, (n[0], n[1], 1), big.offsets, c)
    h = gu.gpu_hierarchy(A)
    cas = cmg.setup_cascade(h, kind, nu=nu, lowp=True)
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    dt = torch.float32 if prec == "fp32" else torch.float64
    b = torch.rand(A.N, generator=g, device="cuda", dtype=dt) - 0.5
    for pre, post, rf in ((1, 1, True), (2, 1, False)):
        x = torch.zeros(A.N, dtype=torch.float64, device="cuda")
        cmg.vcycle(h, cas, b.double(), x, mu_pre=pre, mu_post=post, order="RF" if rf else "FF", precision=prec)
        assert torch.equal(x.to(dt), _cycle(cmg, torch, h, cas, 0, b, kind, nu, pre, post, rf))
