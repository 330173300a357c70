"""BlendFunction without materialised gradients: an image that nothing below
differentiates still gives zero gradients of the inputs' shapes."""
import pytest
import torch

from paper_2604_02120_gb300 import gs

pytestmark = pytest.mark.gpu


class _NoGrad(torch.autograd.Function):
    @staticmethod
    def forward(ctx, x):
        return x.sum()

    @staticmethod
    def backward(ctx, _):
        return None


@pytest.mark.parametrize("variant", ["fp32", "fp16_split"])
def test_undefined_image_gradient_gives_zeros(variant):
    n, w, h = 5, 40, 24
    f = lambda *v: torch.rand(*v, device="cuda").requires_grad_()  # noqa: E731
    leaves = (f(n, 2), f(n, 3), f(n), f(n, 3))
    ranges = torch.zeros(2 * gs.num_tiles(w, h), dtype=torch.int32, device="cuda")
    ids = torch.zeros(1, dtype=torch.int32, device="cuda")
    image, T, nc = gs.BlendFunction.apply(*leaves, ranges, ids, w, h, gs.make_opts(variant))
    assert not T.requires_grad and not nc.requires_grad
    _NoGrad.apply(image).backward()
    for x in leaves:
        assert x.grad is None or (x.grad.shape == x.shape and not x.grad.any())
