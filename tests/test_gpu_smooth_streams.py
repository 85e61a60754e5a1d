"""Red-black applications on a 5-point level work in place, on b and x alone:
calls of one cascade may overlap on two streams."""
import pytest

import problems
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [20, 120, 500])
def test_in_place_applications_overlap(n):
    import torch

    import paper_2606_12577_gb300 as cmg
    A = problems.variable_poisson(problems.random_coefficients(2, n, 3, -1.0, 1.0))
    h = gu.gpu_hierarchy(A)
    c = cmg.setup_cascade(h, "multiplicative", nu=2)
    g = torch.Generator(device="cuda")
    g.manual_seed(5)
    b, x0 = (torch.rand(2, A.N, generator=g, device="cuda", dtype=torch.float64) - 0.5 for _ in range(2))
    ref = x0.clone()
    for k in range(2):
        for _ in range(60):
            cmg.smooth(h, c, 0, b[k], ref[k])
    x = x0.clone()
    streams = [torch.cuda.Stream() for _ in range(2)]
    torch.cuda.synchronize()
    for _ in range(60):
        for k, s in enumerate(streams):
            cmg.smooth(h, c, 0, b[k], x[k], stream=s)
    torch.cuda.synchronize()
    assert torch.equal(x, ref)
