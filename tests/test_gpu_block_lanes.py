"""Block setups of levels with 4096 blocks and more, where the block products
and the E update run one block per lane, against the FP64 oracle: partial
blocks at the upper edges, block counts that leave a warp ragged, both
cascade kinds, 5-, 7- and 9-point operators, FP64 and FP32 products."""
import numpy as np
import pytest

import oracle
import problems
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu


def _ragged(A, nx, ny, nz=1):
    """The operator's rows on the first nx x ny x nz nodes (couplings that leave the box are dropped)."""
    n = A.n
    c = A.coeff.reshape(A.nst, n[2], n[1], n[0])[:, :nz, :ny, :nx].reshape(A.nst, -1).copy()
    return problems.Stencil(A.dim, (nx, ny, nz), A.offsets, c)


def _var(dim, n, seed):
    return problems.variable_poisson(problems.random_coefficients(dim, n, seed, -1.0, 1.0))


CASES = {
    "q1_3x3": (lambda: _ragged(problems.q1_jittered(200, 11), 200, 193), 3),
    "fv_2x2": (lambda: _ragged(_var(2, 131, 5), 129, 131), 2),
    "fv_2x2x2": (lambda: _ragged(_var(3, 35, 7), 35, 33, 32), 2),
}


# FP64: the oracle's own tolerance, 1e-12, for blocks with a regular Gram
# matrix; 3x3 blocks of 9-point operators have exactly null rows from the
# second step on, where two correct FP64 setups agree to a few 1e-12: 1e-10.
# FP32 products: about cond(G) (up to 1e2) times the products' 1e-6 to 1e-5.
@pytest.mark.parametrize("name,kind,nu,fp32,tol", [
    ("q1_3x3", "additive", 3, False, 1e-10), ("q1_3x3", "multiplicative", 1, False, 1e-10),
    ("fv_2x2", "additive", 2, False, 1e-12), ("fv_2x2", "multiplicative", 2, False, 1e-12),
    ("fv_2x2", "additive", 3, True, 1e-3), ("fv_2x2x2", "additive", 2, False, 1e-12),
    ("fv_2x2x2", "multiplicative", 1, False, 1e-12)])
def test_block_setup_of_large_levels(name, kind, nu, fp32, tol):
    import paper_2606_12577_gb300 as cmg
    make, bs = CASES[name]
    A = make()
    co = oracle.Cascade(oracle.Hierarchy(A, bs=bs), kind, nu=nu)
    h = gu.gpu_hierarchy(A, block=bs, max_levels=1)
    c = cmg.setup_cascade(h, kind, nu=nu, setup_precision="fp32" if fp32 else "fp64")
    lam = cmg.export_lambda(c, 0)
    assert np.isfinite(lam).all()
    assert gu.rel_max(lam, co.lam(0)) <= tol
