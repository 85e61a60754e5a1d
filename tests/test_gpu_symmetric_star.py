"""FP32 steps and residuals of 3D 7-point levels read a coupling once for both
of its rows only where the two are the same FP32 number: an operator whose
mirrored couplings differ, however little beside the larger of the two
diagonals, is read row by row."""
import numpy as np
import pytest

import problems
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [(34, 33, 31), (33, 34, 32)])  # pairs of nodes and single ones
def test_mirrored_couplings_of_unequal_rows(n):
    import torch

    import paper_2606_12577_gb300 as cmg
    big = problems.variable_poisson(problems.random_coefficients(3, max(n), 5, -1.0, 1.0))
    c = big.coeff.reshape(7, max(n), max(n), max(n))[:, :n[2], :n[1], :n[0]].copy()
    # rows of a large diagonal, whose neighbours' couplings to them are a half of theirs
    d = c[0].max()
    for x, y, z in ((10, 11, 12), (20, 21, 8), (7, 25, 20)):
        c[0, z, y, x] = 1e13 * d
        for s, q in ((1, (z, y, x + 1)), (2, (z, y, x - 1)), (3, (z, y + 1, x)), (4, (z, y - 1, x)), (5, (z + 1, y, x)),
                     (6, (z - 1, y, x))):
            c[(s, *q)] *= 0.5
    A = problems.Stencil(3, n, big.offsets, c.reshape(7, -1))
    h = gu.gpu_hierarchy(A, max_levels=2)
    cas = cmg.setup_cascade(h, "additive", nu=1, lowp=True)
    b, x = (problems.uniform(s, A.N).astype(np.float32).astype(np.float64) for s in (3, 4))
    lam = cmg.export_lambda(cas, 0).reshape(-1)[:A.N]
    r = gu.stencil_matvec(A, x) - b
    mag = gu.stencil_matvec(problems.Stencil(3, n, A.offsets, np.abs(A.coeff)), np.abs(x)) + np.abs(b)
    b32, x32 = (torch.from_numpy(v).cuda().float() for v in (b, x))
    out = torch.empty_like(x32)
    cmg.sweep(h, cas, 0, 0, b32, x32, out)
    # u = 2^-24: at most 9 roundings of a term of the row (coefficient, seven sums, b), 2 more of Lambda and its
    # product, one of the update
    err = np.abs(out.cpu().numpy() - (x - lam * r))
    assert (err <= 2.0 ** -24 * (14 * np.abs(lam) * mag + 2 * np.abs(x))).all()
    # the restricted residual: the same 9 in every fine value and 27 additions
    rc = torch.empty(h.N(1), device="cuda", dtype=torch.float32)
    cmg.residual_restrict_lowp(h, cas, 0, b32, x32, rc)
    R, M = (v.reshape(n[::-1]) for v in (r, mag))
    nc = [m // 2 for m in n]
    ref, lim = np.zeros(nc[::-1]), np.zeros(nc[::-1])
    for dz in range(3):
        for dy in range(3):
            for dx in range(3):
                w = 0.125 * np.prod([1.0 if q == 1 else 0.5 for q in (dx, dy, dz)])
                v, u = ([np.pad(F, ((0, 2), (0, 2), (0, 2)))[dz:dz + 2 * nc[2]:2, dy:dy + 2 * nc[1]:2, dx:dx + 2 * nc[0]:2]
                         for F in (R, M)])
                ref += w * v
                lim += w * u
    assert (np.abs(rc.cpu().numpy().reshape(ref.shape) - ref) <= 2.0 ** -24 * 39 * lim).all()
