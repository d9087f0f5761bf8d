"""The native autograd node of GELU + Linear where an ordinary backward pass does not lead: errors, gradients of other forms."""
import pytest
import torch

import paper_2202_13808_b200 as dropit
from paper_2202_13808_b200.nn import DropITGeluLinear

pytestmark = pytest.mark.gpu


def _layer(M, Ca, Cz, device, bias=True):
    g = torch.Generator().manual_seed(M + Ca + Cz)
    lin = DropITGeluLinear(Ca, Cz, bias=bias, gamma=0.5, device=device, dtype=torch.bfloat16).train()
    x = torch.randn(M, Ca, generator=g).to(torch.bfloat16).to(device).requires_grad_(True)
    dz = torch.randn(M, Cz, generator=g).to(torch.bfloat16).to(device)
    return lin, x, dz


# The gradient of a torch.cat along the tokens is a contiguous slice that starts anywhere; the weight gradient takes aligned buffers.
@pytest.mark.parametrize("Cz", [10, 100])
def test_an_error_in_the_backward_pass_reaches_the_caller(cuda_device, Cz):
    lin, x, dz = _layer(37, 64, Cz, cuda_device)
    slice_of = torch.cat([dz.new_zeros(1), dz.reshape(-1)])[1:].view_as(dz)
    assert slice_of.is_contiguous() and slice_of.data_ptr() % 16
    with pytest.raises(dropit.DropITError) as error:
        lin(x).backward(slice_of)
    assert error.value.code == 1 and "dropit_weight_grad" in str(error.value)
    lin(x).backward(dz)                      # nothing is left behind
    dropit.check_device_status(cuda_device)
    assert bool(torch.isfinite(lin.weight.grad).all())


def test_a_gradient_penalty_reaches_the_weight(cuda_device):
    """dx = (dz W) GELU'(x) can be differentiated again: the gradients of |dx|^2 with respect to W and dz."""
    lin, x, dz = _layer(37, 64, 24, cuda_device)
    dz.requires_grad_(True)
    dx, = torch.autograd.grad(lin(x), x, dz, create_graph=True)
    dW, ddz = torch.autograd.grad((dx.double() ** 2).sum(), (lin.weight, dz))
    W, z, xd = lin.weight.detach().double(), dz.detach().double(), x.detach().double()
    g = 0.5 * torch.erfc(-xd / 2 ** 0.5) + xd * torch.exp(-0.5 * xd * xd) / (2 * torch.pi) ** 0.5
    inner, size = 2 * (z @ W) * g * g, 2 * (z.abs() @ W.abs()) * g * g      # d|dx|^2 / d(dz W), and what it is summed from
    # bf16 roundings on the way, half a unit (2^-8) each: dz W, dx, its gradient, that times GELU'(x), and the result
    for got, want, bound in ((dW, z.t() @ inner, z.abs().t() @ size), (ddz, inner @ W.t(), size @ W.t().abs())):
        assert bool(((got.double() - want).abs() <= 6 * 2.0 ** -8 * bound).all())


def test_a_bias_gradient_can_be_differentiated(cuda_device):
    lin, x, dz = _layer(37, 64, 24, cuda_device)
    dz.requires_grad_(True)
    _, db = torch.autograd.grad(lin(x), (lin.weight, lin.bias), dz, create_graph=True)
    back, = torch.autograd.grad(db.float().sum(), dz)
    assert torch.equal(back, torch.ones_like(dz))


# Widths that the kernel for the bias gradient and the rounding of dW does not take, a gradient that is expanded, not stored, one that
# has gaps between its rows, and a weight that is not trained.
@pytest.mark.parametrize("Cz", [8, 10, 100, 200])
@pytest.mark.parametrize("form", ["stored", "expanded", "sliced", "frozen"])
def test_gradients_of_other_forms(cuda_device, Cz, form):
    M, Ca = 61, 72
    lin, x, dz = _layer(M, Ca, Cz, cuda_device)
    if form == "expanded":
        dz = dz[0, 0].expand(M, Cz)
    elif form == "sliced":
        dz = torch.cat([dz, dz], 1)[:, Cz // 2:Cz // 2 + Cz]
    lin.weight.requires_grad_(form != "frozen")
    lin(x).backward(dz)
    dropit.check_device_status(cuda_device)
    z, xd, W = dz.double(), x.detach().double(), lin.weight.detach().double()
    u, eps = 2.0 ** -8, M * 2.0 ** -24
    g = 0.5 * torch.erfc(-xd / 2 ** 0.5) + xd * torch.exp(-0.5 * xd * xd) / (2 * torch.pi) ** 0.5
    # bf16 roundings of dz W and of dx; one rounding of an fp32 sum of M terms for the others
    assert bool(((x.grad.double() - (z @ W) * g).abs() <= 2.1 * u * (z.abs() @ W.abs()) * g.abs() + 1e-5 * (z.abs() @ W.abs())).all())
    assert bool(((lin.bias.grad.double() - z.sum(0)).abs() <= u * z.sum(0).abs() + 2 * eps * z.abs().sum(0)).all())
    if form == "frozen":
        assert lin.weight.grad is None
        return
    y, prep = dropit.dropit_produce(x.detach(), 0.5, "gelu")
    kept = dropit.dropit_decompress(dropit.dropit_compress_prepared(y, 0.5, prep)).double()
    want, size = z.t() @ kept, z.abs().t() @ kept.abs()
    assert bool(((lin.weight.grad.double() - want).abs() <= u * want.abs() + 2 * eps * size).all())


def test_refusals_read_as_torch_writes_types(cuda_device):
    x = torch.randn(8, 16, device=cuda_device)
    with pytest.raises(TypeError, match=r"x: dtype torch\.float16 is not supported"):
        dropit.dropit_compress(x.half(), 0.5)
    cache = dropit.dropit_compress(x.bfloat16(), 0.5)
    with pytest.raises(TypeError, match=r"dy dtype torch\.float32 != cache dtype torch\.bfloat16"):
        dropit.dropit_weight_grad(x, cache)
    with pytest.raises(IndexError):
        dropit.dropit_weight_grad(x[0, 0].bfloat16(), cache)
