"""FP32 block setups of levels with 4096 blocks and more: the products of the
FP32 rows are formed and summed in FP64.  The rows of these operators are FP32
numbers (unit diagonal, couplings of 24 bits), so the first step's Lambda is
the oracle's to FP64 accuracy."""
import numpy as np
import pytest

import oracle
import problems
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu


# 1e-12: the oracle's own tolerance (blocks of a diagonally dominant operator have cond(G) of about 10)
@pytest.mark.parametrize("n,bs,box", [((131, 129), 2, False), ((130, 133), 2, True), ((200, 197), 3, True),
                                      ((33, 35, 32), 2, False)])
def test_first_step_of_exact_rows(n, bs, box):
    import paper_2606_12577_gb300 as cmg
    dim = len(n)
    offs = [(a, b, 0) for b in (-1, 0, 1) for a in (-1, 0, 1)] if box else problems._star_offsets(dim)
    N = int(np.prod(n))
    c = np.stack([-problems.uniform(60 + s, N, 0.02, 0.1).astype(np.float32).astype(np.float64) for s in range(len(offs))])
    c[offs.index((0, 0, 0))] = 1.0
    A = problems.Stencil(dim, tuple(n) + (1,) * (3 - dim), offs, c)
    ref = oracle.Cascade(oracle.Hierarchy(A, bs=bs), "additive", nu=1).lam(0)
    h = gu.gpu_hierarchy(A, block=bs, max_levels=1)
    lam = cmg.export_lambda(cmg.setup_cascade(h, "additive", nu=1, setup_precision="fp32"), 0)
    assert gu.rel_max(lam, ref) <= 1e-12
