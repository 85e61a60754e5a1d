"""The network's products over the paths its shapes take: K splits and their
reduction, one wave of tiles and the persistent form, results in float4 rows
and in single columns, hidden widths that leave the packed operands padded,
one row.  Forward pass and gradients against FP64 arithmetic on BF16 weights
(plain torch).  FP32 factors enter as BF16 pairs, so every product carries
about 2^-16 relative: 1e-4 of the largest entry over three layers.  A
pre-activation within that distance of zero may fall on either side of the
ReLU's kink, which adds or drops its row's whole contribution to the
gradients: the bound of a gradient entry adds the magnitudes of those
contributions, |d| |h| summed over the undecided units."""
import math

import pytest

pytestmark = pytest.mark.gpu

SHAPES = [(225, 256, 243, 1), (225, 256, 243, 4096), (20, 52, 30, 77), (64, 64, 64, 129), (33, 130, 7, 300),
          (225, 128, 244, 20001)]


def _reference(p, X, T):
    """Y, loss, gradients, and per gradient entry the most that undecided ReLUs can change it by."""
    import torch
    W = [t.to(torch.bfloat16).double() if t.dim() == 2 else t.double() for t in p]
    X = X.double()
    Z1 = X @ W[0].T + W[1]
    H1 = Z1.clamp(min=0)
    Z2 = H1 @ W[2].T + W[3]
    H2 = Z2.clamp(min=0)
    Y = H2 @ W[4].T + W[5]
    E = Y - T.double()
    dY = 2 * E / E.numel()
    dH2 = dY @ W[4]
    dZ2 = dH2 * (Z2 > 0)
    dH1 = dZ2 @ W[2]
    dZ1 = dH1 * (Z1 > 0)
    g = [dZ1.T @ X, dZ1.sum(0), dZ2.T @ H1, dZ2.sum(0), dY.T @ H2, dY.sum(0)]
    u2 = dH2.abs() * (Z2.abs() <= 1e-4 * Z2.abs().max())
    u1 = (dH1.abs() + u2 @ W[2].abs()) * (Z1.abs() <= 1e-4 * Z1.abs().max()) + (u2 @ W[2].abs()) * (Z1 > 0)
    s = [u1.T @ X.abs(), u1.sum(0), u2.T @ H1, u2.sum(0), 0 * g[4], 0 * g[5]]
    return Y, float((E * E).mean()), g, s


@pytest.mark.parametrize("nin,nhid,nout,B", SHAPES)
def test_forward_and_gradients(nin, nhid, nout, B):
    import torch

    import paper_2606_12577_gb300 as cmg
    g = torch.Generator(device="cuda")
    g.manual_seed(5)

    def rnd(*s):
        return torch.rand(*s, generator=g, device="cuda") * 2 - 1
    p = []
    for r, c in ((nhid, nin), (nhid, nhid), (nout, nhid)):
        p += [rnd(r, c) * math.sqrt(6.0 / c), 0.05 * rnd(r)]
    X, T = rnd(B, nin), rnd(B, nout)
    net = cmg.MLP(nin, nhid, nout, max_batch=max(B, 64))
    net.set_params(torch.cat([t.reshape(-1) for t in p]).cpu().numpy())
    Y, loss, grad, slacks = _reference(p, X, T)
    assert float((net.forward(X).double() - Y).abs().max()) <= 1e-4 * float(Y.abs().max())
    lg, gg = net.gradients(X, T)
    assert abs(lg - loss) <= 1e-4 * loss
    at = 0
    for ref, slack in zip(grad, slacks):  # each parameter's gradient against its own largest entry
        got = torch.tensor(gg[at:at + ref.numel()], device="cuda").double().reshape(ref.shape)
        assert bool(((got - ref).abs() <= 3e-4 * ref.abs().max() + slack).all())
        at += ref.numel()
    # the same pass after a smaller one leaves nothing of it behind
    net.forward(X[: max(1, B // 3)].contiguous())
    assert float((net.forward(X).double() - Y).abs().max()) <= 1e-4 * float(Y.abs().max())
