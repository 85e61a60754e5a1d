"""Sweeps, residuals and restrictions of operators with repeated rows, which
take their coefficients and Lambda from the centre row (3D levels of 64^3 rows
and more march over planes), against the same handles built with reuse=False,
which read every row, and colour steps against the oracle on odd and even
widths.  Constant and partly constant operators, even and odd sides (an even
side cuts the coarse rows at the upper faces), planes that are no multiple of
the march."""
import numpy as np
import pytest

import oracle
import problems
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu


def _poisson(n):
    return problems.Stencil(len(n), tuple(n) + (1,) * (3 - len(n)), *_const(n))


def _const(n, w=1.0):
    """(offsets, coefficients) of the constant 5- / 7-point operator."""
    dim = len(n)
    offs = problems._star_offsets(dim)
    N = int(np.prod(n))
    c = np.full((len(offs), N), -w)
    c[0] = 2 * dim * w
    return offs, c


def _bump(n):
    """Constant, except for one row near a corner, one at an edge and one inside near a face."""
    A = _poisson(n)
    nx, ny = A.n[0], A.n[1]
    for k, (x, y, z) in enumerate([(1, 1, 1), (0, 0, A.n[2] // 2), (nx // 2, ny // 2, A.n[2] - 3)]):
        A.coeff[0, x + nx * (y + ny * z)] *= 1.5 + 0.25 * k
    return A


OPS = {"const": _poisson, "bump": _bump}


def _handles(A, kind, nu):
    import paper_2606_12577_gb300 as cmg
    out = []
    for reuse in (True, False):
        h = gu.gpu_hierarchy(A, reuse=reuse)
        out.append((h, cmg.setup_cascade(h, kind, nu=nu, lowp=True, reuse=reuse)))
    return out


# the same coefficients in the same order on both sides: equal bits, but for
# the FP64 norm's partial sums, which the march cuts differently
@pytest.mark.parametrize("op", ["const", "bump"])
@pytest.mark.parametrize("n,kind", [((66, 64, 65), "additive"), ((63, 65, 67), "additive"), ((64, 66, 65), "multiplicative"),
                                    ((129, 127), "multiplicative"), ((70, 64), "additive")])
def test_repeated_rows_change_no_bits(op, n, kind):
    import torch

    import paper_2606_12577_gb300 as cmg
    if op == "bump" and len(n) == 2:
        pytest.skip("3D rows")
    A = OPS[op](n)
    (h1, c1), (h0, c0) = _handles(A, kind, 2)
    g = torch.Generator(device="cuda")
    g.manual_seed(7)
    for l in range(min(2, h1.nlevels - 1)):
        N, Nc = h1.N(l), h1.N(l + 1)
        x = torch.rand(N, generator=g, device="cuda", dtype=torch.float64) - 0.5
        b = torch.rand(N, generator=g, device="cuda", dtype=torch.float64) - 0.5
        for dt in (torch.float64, torch.float32):
            xs, bs = x.to(dt), b.to(dt)
            got = []
            for h, c in ((h1, c1), (h0, c0)):
                r = []
                for step in range(2):
                    for colour in ((-1,) if kind == "additive" else (0, 1)):
                        o = torch.empty_like(xs)
                        cmg.sweep(h, c, l, step, bs, xs, o, colour=colour)
                        r.append(o)
                rc = torch.empty(Nc, device="cuda", dtype=dt)
                if dt == torch.float64:
                    cmg.residual_restrict(h, l, bs, xs, rc)
                    res = torch.empty_like(xs)
                    r += [rc, res]
                    norm = cmg.residual(h, l, bs, xs, res, norm=True)
                    assert abs(norm - float(res.norm())) <= 1e-13 * norm
                else:
                    cmg.residual_restrict_lowp(h, c, l, bs, xs, rc)
                    r.append(rc)
                got.append(r)
            for u, v in zip(*got):
                assert torch.equal(u, v)
    # whole cycles in both precisions
    b = torch.rand(A.N, generator=g, device="cuda", dtype=torch.float64) - 0.5
    for prec in ("fp64", "fp32"):
        xs = []
        for h, c in ((h1, c1), (h0, c0)):
            x = torch.zeros(A.N, dtype=torch.float64, device="cuda")
            cmg.vcycle(h, c, b, x, precision=prec)
            xs.append(x)
        assert torch.equal(*xs)


def test_colour_steps_match_oracle_on_ragged_widths():
    import torch

    import paper_2606_12577_gb300 as cmg
    for n in ((65, 33), (64, 31), (17, 16, 15)):
        A = _poisson(n)
        ho = oracle.Hierarchy(A)
        co = oracle.Cascade(ho, "multiplicative", nu=2)
        h = gu.gpu_hierarchy(A)
        c = cmg.setup_cascade(h, "multiplicative", nu=2)
        b = problems.rhs(A.N, 3)
        x = problems.uniform(5, A.N)
        xd = torch.tensor(x, device="cuda")
        cmg.smooth(h, c, 0, torch.tensor(b, device="cuda"), xd)
        xo = oracle.smooth(ho, co, 0, b, x)
        assert gu.rel_max(xd.cpu().numpy(), xo) <= 1e-12


# four rows per thread in the FP32 setup products (27-point levels of 128 k
# rows and more): Lambda against the oracle, whose FP64 rows differ from FP32
# products by a few u (u = 2^-24) of their sums over up to 3375 products: 1e-4,
# the bound of the row-per-thread form.  Quads that end early (sides no
# multiple of 4), with repeated rows and without.
@pytest.mark.parametrize("n,const", [((107, 106, 105), True), ((102, 104, 103), False)])
def test_fp32_setup_rows_of_large_27_point_levels(n, const):
    import paper_2606_12577_gb300 as cmg
    A = _poisson(n)
    if not const:
        A.coeff[0] *= 1.0 + 0.2 * problems.uniform01(9, A.N)
    # the finest operator itself as a 27-point one, the seven-point couplings and weak ones to the rest of the box
    offs = [(dx, dy, dz) for dz in (-1, 0, 1) for dy in (-1, 0, 1) for dx in (-1, 0, 1)]
    c = np.zeros((27, A.N))
    for s, o in enumerate(A.offsets):
        c[offs.index(o)] = A.coeff[s]
    for s, o in enumerate(offs):
        if o not in A.offsets:
            c[s] = -0.05
    c[13] += 1.2
    B = problems.Stencil(3, A.n, offs, c)
    co = oracle.Cascade(oracle.Hierarchy(B), "additive", nu=2)
    h = gu.gpu_hierarchy(B)
    cg = cmg.setup_cascade(h, "additive", nu=2, setup_precision="fp32")
    lam, ref = cmg.export_lambda(cg, 0), co.lam(0)
    assert gu.rel_max(lam, ref) <= 1e-4
