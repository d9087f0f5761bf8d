"""Coordinate caches are complete without their seek table: calls that read one take them with a table, an unaligned one or none."""
import ctypes
from dataclasses import replace

import pytest
import torch

import dropit_inputs as di
import paper_2202_13808_b200 as dropit
from paper_2202_13808_b200 import _lib


def test_binding_takes_a_cache_without_a_table():
    """(On CPU tensors, which the call refuses only after it has taken its arguments.)"""
    cache = dropit.DropITCache(torch.zeros(2), torch.zeros(2, dtype=torch.int32), None, 4, 2, (2, 2), torch.float32, dropit.FMT_INDEX32, 0.5)
    with pytest.raises(ValueError, match="CUDA tensor"):
        dropit.dropit_weight_grad(torch.zeros(2, 2), cache)
    with pytest.raises(ValueError, match="CUDA tensor"):
        dropit.dropit_conv_weight_grad(torch.zeros(1, 2, 2, 2), replace(cache, shape=(1, 1, 2, 2)), (1, 1))


@pytest.mark.gpu
@pytest.mark.parametrize("dtype", ["bf16", "f32"])
def test_gradients_do_not_depend_on_the_table(cuda_device, dtype):
    case = di.small_linear(300, 72, 40, dtype, 0.7)
    dy = di.make_dy(case).to(cuda_device)
    cache = dropit.dropit_compress(di.make_x(case).to(cuda_device), case.gamma, "index32")
    assert torch.equal(dropit.dropit_weight_grad(dy, replace(cache, offsets=None)), dropit.dropit_weight_grad(dy, cache))
    conv = di.small_conv(2, 5, 9, 11, 6, 3, 3, 1, 1, dtype, 0.7)
    dy = di.make_dy(conv).to(cuda_device)
    cache = dropit.dropit_compress(di.make_x(conv).to(cuda_device), conv.gamma, "index32")
    assert torch.equal(dropit.dropit_conv_weight_grad(dy, replace(cache, offsets=None), (3, 3), 1, 1),
                       dropit.dropit_conv_weight_grad(dy, cache, (3, 3), 1, 1))
    dropit.check_device_status(cuda_device)


@pytest.mark.gpu
@pytest.mark.parametrize("shift", [1, 2, 4])     # bytes
def test_decompression_with_an_unaligned_table(cuda_device, shift):
    x = torch.randn(5000, generator=torch.Generator().manual_seed(shift)).to(torch.bfloat16).to(cuda_device)
    cache = dropit.dropit_compress(x, 0.6, "index32")
    dense, out = dropit.dropit_decompress(cache), torch.full_like(x, 7.0)
    table = torch.zeros(cache.offsets.numel() * 4 + 16, dtype=torch.uint8, device=cuda_device)
    table[shift:shift + cache.offsets.numel() * 4] = cache.offsets.view(torch.uint8)
    status = _lib.load().dropit_decompress(
        ctypes.c_void_p(cache.values.data_ptr()), ctypes.c_void_p(cache.meta.data_ptr()), ctypes.c_void_p(table.data_ptr() + shift),
        cache.n, cache.k, dropit.BF16, dropit.FMT_INDEX32, ctypes.c_void_p(out.data_ptr()),
        ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert status == 0 and torch.equal(out, dense)
