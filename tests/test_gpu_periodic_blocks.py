"""Block setups of periodic grids of 4096 blocks and more, against the FP64
oracle.  On a side that is no multiple of the block edge the last block is
partial and its next node is the first of block 0, so the blocks do not tile
the plane as a lattice; both such sides and whole ones, 2x2, 3x3 and 2x2x2
blocks, both cascade kinds, FP64 and FP32 products.

The operator is constant (and not symmetric), so a block's Lambda depends only
on where it lies beside the partial blocks, a few blocks away at most: the
oracle works on a small grid whose sides leave the same remainder, and every
block of the large one is compared with its image there."""
import numpy as np
import pytest

import oracle
import problems
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu

COUPLINGS = (5.0, -1.0, -0.7, -0.4, -1.3, -0.6, -0.9)


def _constant(n):
    dim = len(n)
    c = np.repeat(np.array(COUPLINGS[:2 * dim + 1])[:, None], int(np.prod(n)), axis=1)
    return problems.Stencil(dim, tuple(n) + (1,) * (3 - dim), problems._star_offsets(dim), c, periodic=True)


def _image(big, small):
    """Per block of a side of `big` blocks, the block of the side of `small`: the same distance from the last block
    near either end, the same parity in between."""
    assert (big - small) % 2 == 0
    half = small // 2
    return [b if b < half else b - (big - small) if b >= big - (small - half) else half - 1 + (b - half + 1) % 2
            for b in range(big)]


def _by_block(lam, n, bs, nu):
    """[step][block z, y, x] of the n_b x n_b values of the blocks, which lie one after the other."""
    sides = [[min(bs, m - bs * b) for b in range(-(-m // bs))] for m in n]
    size = np.array([[[(x * y * z) ** 2 for x in sides[0]] for y in sides[1]] for z in sides[2]])
    at = np.cumsum(size.ravel())[:-1]
    out = []
    for step in np.asarray(lam).reshape(nu, -1):
        part = np.empty(size.size, dtype=object)
        for b, v in enumerate(np.split(step, at)):
            part[b] = v
        out.append(part.reshape(size.shape))
    return out


# FP64: the oracle's own tolerance, 1e-12; the centre row of a 3x3 block of a
# 5-point operator is null from the second step on, where two correct FP64
# setups agree to a few 1e-12: 1e-10.  FP32 products: about cond(G) (up to
# 1e2) times the products' 1e-6 to 1e-5.
@pytest.mark.parametrize("n,small,bs,kind,nu,fp32,tol", [
    ((129, 129), (25, 25), 2, "additive", 2, False, 1e-12), ((129, 131), (25, 27), 2, "multiplicative", 2, False, 1e-12),
    ((131, 128), (27, 24), 2, "additive", 3, True, 1e-3), ((128, 132), (24, 28), 2, "additive", 2, False, 1e-12),
    ((200, 199), (32, 31), 3, "additive", 2, False, 1e-10), ((200, 199), (32, 31), 3, "multiplicative", 2, False, 1e-10),
    ((198, 195), (30, 33), 3, "additive", 2, False, 1e-10), ((33, 32, 33), (13, 12, 13), 2, "additive", 2, False, 1e-12),
    ((32, 33, 34), (12, 13, 14), 2, "multiplicative", 1, False, 1e-12)])
def test_periodic_block_setup(n, small, bs, kind, nu, fp32, tol):
    import paper_2606_12577_gb300 as cmg
    A, S = _constant(n), _constant(small)
    nb, ns = ([-(-v // bs) for v in B.n] for B in (A, S))
    assert np.prod(nb) >= 4096
    h = gu.gpu_hierarchy(A, block=bs, max_levels=1)
    lam = cmg.export_lambda(cmg.setup_cascade(h, kind, nu=nu, setup_precision="fp32" if fp32 else "fp64"), 0)
    ref = oracle.Cascade(oracle.Hierarchy(S, bs=bs), kind, nu=nu).lam(0)
    ix, iy, iz = (_image(p, q) for p, q in zip(nb, ns))
    for got, want in zip(_by_block(lam, A.n, bs, nu), _by_block(ref, S.n, bs, nu)):
        want = want[iz][:, iy][:, :, ix]
        assert gu.rel_max(np.concatenate(got.ravel()), np.concatenate(want.ravel())) <= tol
