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
