"""How many FP32 terms are added up before FP64 takes over: the squares of a
convergence norm, a CTA's nodes of one plane; the products of a row in the
FP32 setup of large 27-point levels, none: they are summed as pairs."""
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


def _fma32(a, b, c):
    """fma(a, b, c) of FP32 values, correctly rounded: the product is exact in
    FP64, the sum is rounded to odd there and then to FP32."""
    p = a.astype(np.float64) * b.astype(np.float64)
    c = np.asarray(c, np.float64)
    s = p + c
    bb = s - p
    err = (p - (s - bb)) + (c - bb)
    even = (s.view(np.int64) & 1) == 0
    odd = np.where((err != 0) & even, np.nextafter(s, np.where(err > 0, np.inf, -np.inf)), s)
    return odd.astype(np.float32)


class _Pair:
    """A sum of products as a pair of FP32 numbers (Knuth's two-sum, products exact by fma)."""

    def __init__(self):
        self.s = self.e = np.float32(0)

    def add(self, a, b):
        p = a * b
        t = self.s + p
        v = t - self.s
        d = (self.s - (t - v)) + (p - v)
        self.e = self.e + (d + _fma32(a.reshape(1), b.reshape(1), -p.reshape(1))[0])
        self.s = t

    def value(self):
        return float(self.s) + float(self.e)


def _row_lambdas(a, nu):
    """Lambda of a row of the constant 27-point operator a (unit diagonal) far
    from the boundary, in the FP32 setup's arithmetic: a column of products
    over (sx, sy), inner products as pairs."""
    E = np.ones((1, 1, 1), np.float32)  # [z, y, x]
    lams = []
    for lev in range(nu):
        r, R = lev, lev + 1
        SC, SN = 2 * r + 1, 2 * R + 1
        acc = np.zeros((SN, SN, SN), np.float32)
        num, den = _Pair(), _Pair()
        for oy in range(-R, R + 1):
            for ox in range(-R, R + 1):
                col = np.zeros(SN, np.float32)
                for sy in range(max(-1, oy - r), min(1, oy + r) + 1):
                    for sx in range(max(-1, ox - r), min(1, ox + r) + 1):
                        e = E[:, oy - sy + r, ox - sx + r]
                        for u in range(SC):
                            col[u:u + 3] = _fma32(a[:, sy + 1, sx + 1], np.full(3, e[u]), col[u:u + 3])
                acc[:, oy + R, ox + R] = col
                mid = abs(ox) <= r and abs(oy) <= r
                for u in range(SN):
                    if mid and 1 <= u <= SC:
                        num.add(E[u - 1, oy + r, ox + r], col[u])
                    den.add(col[u], col[u])
        lams.append(num.value() / den.value())
        big = np.zeros((SN, SN, SN), np.float32)
        big[1:-1, 1:-1, 1:-1] = E
        E = _fma32(np.float32(-np.float32(lams[-1])) * np.ones_like(acc), acc, big)
    return lams


def test_fp32_setup_row_sums():
    """The repeated row of a constant 27-point level, bit for bit, to radius 4."""
    import paper_2606_12577_gb300 as cmg
    a = np.full((3, 3, 3), 0.0, np.float32)
    for z in range(3):
        for y in range(3):
            for x in range(3):
                a[z, y, x] = -(8 + x + 2 * y + 3 * z) / 512.0  # not symmetric
    a[1, 1, 1] = 1.0
    n = (51, 52, 50)  # 132,600 rows
    offs = [(x - 1, y - 1, z - 1) for z in range(3) for y in range(3) for x in range(3)]
    N = int(np.prod(n))
    A = problems.Stencil(3, n, offs, np.repeat(a.reshape(27, 1).astype(np.float64), N, axis=1))
    h = gu.gpu_hierarchy(A, max_levels=1)
    lam = cmg.export_lambda(cmg.setup_cascade(h, "additive", nu=4, setup_precision="fp32"), 0)
    centre = n[0] // 2 + n[0] * (n[1] // 2 + n[1] * (n[2] // 2))
    assert list(lam.reshape(4, N)[:, centre]) == _row_lambdas(a, 4)


# the same setup against the oracle on an operator without repeated rows, to
# the radii 3 and 4: FP32 products differ from the oracle's FP64 rows by a few
# u (u = 2^-24) of sums over up to 9^3 27 products: 1e-4, as for radius 2
def test_fp32_setup_rows_to_radius_4():
    import oracle
    import paper_2606_12577_gb300 as cmg
    n = (53, 50, 51)
    offs = [(x - 1, y - 1, z - 1) for z in range(3) for y in range(3) for x in range(3)]
    N = int(np.prod(n))
    c = np.stack([-0.05 - 0.02 * problems.uniform01(40 + s, N) for s in range(27)])
    c[13] = 2.0 + 0.4 * problems.uniform01(80, N)
    A = problems.Stencil(3, n, offs, c)
    ref = oracle.Cascade(oracle.Hierarchy(A), "additive", nu=4).lam(0)
    h = gu.gpu_hierarchy(A, max_levels=1)
    lam = cmg.export_lambda(cmg.setup_cascade(h, "additive", nu=4, setup_precision="fp32"), 0)
    for got, want in zip(np.reshape(lam, (4, N)), np.reshape(ref, (4, N))):
        assert gu.rel_max(got, want) <= 1e-4
