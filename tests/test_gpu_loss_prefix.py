"""The composed loss on rows of one sign, where row prefixes grow to the length
of the row: its gradient is no further from 64 bits than that of the separate
calls whose scans carry a float64 between tiles (variant 0, and 5 where rows
are aligned)."""
import numpy as np
import pytest

from helpers import forced, skel
from test_gpu_loss import separate

pytestmark = pytest.mark.gpu


def stencil(x):
    import torch
    p = torch.nn.functional.pad(x[None, None], (1, 1, 1, 1), mode="replicate")[0, 0]
    w = [1, 2, 1]
    return sum(w[a] * w[b] / 16 * p[a:a + x.shape[0], b:b + x.shape[1]] for a in range(3) for b in range(3))


def exact_gradient(x):
    """In 64 bits; the stencil's adjoint by torch's own differentiation."""
    import torch
    with torch.enable_grad():
        v = x.double().requires_grad_(True)
        t = torch.tanh(v)
        loss = stencil(t).square().sum() + t.cumsum(1).square().sum() / x.numel()
        return torch.autograd.grad(loss, v)[0]


@pytest.mark.parametrize("high", [0.02, 1.0])
@pytest.mark.parametrize("shape,variant", [((2048, 8191), 0), ((512, 2050), 0), ((64, 8192), 5)])
def test_gradient_on_rows_of_one_sign(shape, variant, high):
    import torch
    from paper_1405_2915_gb300.autograd import composed_loss
    sk = skel()
    g = torch.Generator(device="cuda").manual_seed(7)
    x = torch.rand(shape, device="cuda", generator=g) * high
    ref = exact_gradient(x)
    xt = x.clone().requires_grad_(True)
    (gx,) = torch.autograd.grad(composed_loss(xt), xt)
    with forced("scan", variant):
        _, gs = separate(sk, x, None, "clamp", 1.0)
    error = lambda v: float((v.double() - ref).norm() / ref.norm())
    fused, calls = error(gx), error(torch.from_numpy(gs).cuda())
    assert fused <= calls, (fused, calls)
