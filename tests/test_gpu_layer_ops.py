"""The kernels around a layer's weight gradient in the native autograd node: GELU derivative, bias gradient, rounded weight gradient."""
import pytest
import torch
import torch.nn.functional as F

pytestmark = pytest.mark.gpu

U = 2.0 ** -8      # half a unit in the last place of bf16, relative


def _run(M, Ca, Cz, scale, bias, device, nd=2):
    from paper_2202_13808_b200.nn import DropITGeluLinear
    g = torch.Generator().manual_seed(7 + M + Ca)
    x = (torch.randn(M, Ca, generator=g) * scale).to(torch.bfloat16).to(device)
    if nd == 3:
        x = x.reshape(1, M, Ca)
    lin = DropITGeluLinear(Ca, Cz, bias=bias, gamma=0.5, device=device, dtype=torch.bfloat16).train()
    dz = torch.randn(*x.shape[:-1], Cz, generator=g).to(torch.bfloat16).to(device)
    x.requires_grad_(True)
    lin(x).backward(dz)
    return lin, x, dz


# Widths: one column group and a partial last one, more than one; lengths: fewer rows than a cluster takes at once, ragged, many.
# Scales: inside the derivative's table, far above it (its tails) and far below it.
@pytest.mark.parametrize("M, Ca, Cz, scale, bias", [(1, 64, 8, 1.0, True), (37, 72, 72, 1.0, True), (257, 200, 136, 8.0, True),
                                                    (1031, 328, 64, 1e-4, True), (3152, 768, 200, 2.0, True), (300, 96, 64, 1.0, False),
                                                    (37, 37, 8, 1.0, True)])
def test_gradients_around_the_weight_gradient(cuda_device, M, Ca, Cz, scale, bias):
    lin, x, dz = _run(M, Ca, Cz, scale, bias, cuda_device, nd=2 + M % 2)
    dz2, x2 = dz.reshape(-1, Cz), x.detach().reshape(-1, Ca)
    # dx: the rounded dy that the layer forms, times the derivative in fp64; one rounding, and the derivative's own fp32 error (erff 2 ulp,
    # expf 2 ulp, the constants' rounding times |x| <= 13 before it vanishes: below 1e-5).
    dy = torch.matmul(dz2, lin.weight.detach()).double()
    xd = x2.double()
    deriv = 0.5 * torch.erfc(-xd / 2 ** 0.5) + xd * torch.exp(-0.5 * xd * xd) / (2 * torch.pi) ** 0.5
    want = dy * deriv
    assert bool(((x.grad.reshape(-1, Ca).double() - want).abs() <= U * want.abs() + 1e-5 * dy.abs() + 1e-37).all())
    if bias:        # fp32 sum of M terms, then one rounding
        want = dz2.double().sum(0)
        bound = U * want.abs() + M * 2.0 ** -24 * dz2.double().abs().sum(0) * (1 + U) + 1e-37
        assert bool(((lin.bias.grad.double() - want).abs() <= bound).all())
    # dW: the public entry point's fp32 result for the same kept elements, rounded once (its fp32 sums may run in another order)
    from paper_2202_13808_b200 import api
    y, prep = api.dropit_produce(x2.contiguous(), 0.5, "gelu")
    cache = api.dropit_compress_prepared(y, 0.5, prep)
    full = api.dropit_weight_grad(dz2.contiguous(), cache).double()
    bound = U * full.abs() + 2 * M * 2.0 ** -24 * (dz2.double().abs().t() @ F.gelu(xd).abs()) * (1 + U) + 1e-37
    assert bool(((lin.weight.grad.double() - full).abs() <= bound).all())
