"""Steps of 2x2-node block levels with several right-hand sides, a block per
thread: partial blocks on one side and on both, column counts for copies of
16, 8 and 4 bytes and for none, tensors off the copies' alignment, grids
smaller than a tile and of several, 5- and 9-point rows, both directions,
against the FP64 oracle's smoother column by column."""
import numpy as np
import pytest

import oracle
import problems
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu


def _operator(n, box):
    A = problems.q1_jittered(max(n), 11) if box else problems.variable_poisson(
        problems.random_coefficients(2, max(n), 5, -1.0, 1.0))
    c = A.coeff.reshape(A.nst, A.n[1], A.n[0])[:, :n[1], :n[0]].reshape(A.nst, -1).copy()
    return problems.Stencil(2, (n[0], n[1], 1), A.offsets, c)


# FP64: block products of a dozen terms on O(1) data, the setups' 1e-10 of
# nearly singular 9-point blocks on top; FP32: some forty roundings a step,
# 2e-5, times |Lambda||A| of about ten on the 9-point levels.
@pytest.mark.parametrize("n,box,kind,m,shift", [
    ((6, 5), False, "additive", 1, 0), ((5, 6), False, "additive", 2, 0), ((7, 7), False, "multiplicative", 3, 0),
    ((33, 9), False, "additive", 4, 1), ((33, 9), False, "multiplicative", 8, 2), ((20, 31), True, "additive", 6, 0),
    ((15, 12), True, "multiplicative", 4, 0), ((261, 7), False, "additive", 12, 0), ((9, 5), True, "additive", 5, 0),
    ((70, 30), False, "multiplicative", 32, 0), ((13, 41), False, "additive", 31, 0), ((40, 17), True, "additive", 28, 0)])
def test_rhs_steps_of_2d_blocks(n, box, kind, m, shift):
    import torch

    import paper_2606_12577_gb300 as cmg
    A = _operator(n, box)
    ho = oracle.Hierarchy(A, bs=2)
    co = oracle.Cascade(ho, kind, nu=2)
    h = gu.gpu_hierarchy(A, block=2)
    c = cmg.setup_cascade(h, kind, nu=2, lowp=True)
    B = problems.uniform(31, A.N * m).reshape(A.N, m)
    X = problems.uniform(32, A.N * m).reshape(A.N, m)
    cols = (0, 1) if kind == "multiplicative" else (-1,)
    for rev in (False, True):
        ref = np.stack([oracle.smooth(ho, co, 0, B[:, r], X[:, r], reverse=rev) for r in range(m)], axis=1)
        for dt, tol in ((torch.float64, 1e-9), (torch.float32, 2e-4 if box else 2e-5)):
            def dev(a):  # `shift` values off the allocation's alignment
                buf = torch.zeros(a.size + shift, dtype=dt, device="cuda")
                buf[shift:] = torch.from_numpy(a.reshape(-1)).to("cuda", dt)
                return buf[shift:]
            b, cur, oth = dev(B), dev(X), dev(np.zeros_like(X))
            for lv in ((1, 0) if rev else (0, 1)):
                for col in (cols[::-1] if rev else cols):
                    cmg.sweep_rhs(h, c, 0, lv, b, cur, oth, m, colour=col, transpose=rev)
                    cur, oth = oth, cur
            got = cur.cpu().numpy().astype(np.float64).reshape(A.N, m)
            assert gu.rel_max(got, ref) <= tol, f"reverse={rev} {dt}"
