"""Conv2d weight gradient straight from a bitmask cache: against the oracle where its bands and tiles can go wrong."""
import pytest
import torch

import dropit_inputs as di
import oracle
import paper_2202_13808_b200 as dropit
from _parity import conv_weight_grad_f64, max_rel_err, oracle_cache

pytestmark = pytest.mark.gpu

CASES = [
    di.small_conv(1, 1, 3, 3, 1, 3, 3, 1, 0, "bf16", 0.5),        # one output pixel, one channel
    di.small_conv(5, 17, 7, 7, 65, 3, 3, 1, 1, "bf16", 0.8),      # several images in a band, an odd number of 8-pixel groups
    di.small_conv(3, 9, 9, 9, 64, 1, 1, 1, 0, "bf16", 0.8),       # a flattened plane that is no multiple of 8 pixels
    di.small_conv(2, 33, 27, 21, 129, 2, 3, 1, 2, "bf16", 0.0),   # two output tiles, nothing dropped, padding wider than the filter needs
    di.small_conv(2, 300, 11, 40, 20, 3, 3, 1, 1, "bf16", 0.9),   # many channel blocks
    di.small_conv(3, 24, 19, 23, 40, 1, 1, 2, 0, "bf16", 0.8),    # every other row and column only
    di.small_conv(3, 24, 20, 33, 72, 3, 2, 2, 1, "bf16", 0.8),    # stride 2, even and odd columns
    di.small_conv(2, 16, 130, 5, 16, 3, 1, 2, 1, "bf16", 0.5),    # tall and narrow: several bands per image, one plane
    di.small_conv(3, 40, 64, 64, 24, 3, 3, 1, 1, "bf16", 0.95),   # rows of whole mask words
]


@pytest.mark.parametrize("case", CASES, ids=lambda c: c.name)
def test_fused_conv_weight_grad_matches_oracle(cuda_device, case):
    x, dy = di.make_x(case), di.make_dy(case)
    bits, dt, keep, _ = oracle_cache(x, case.gamma)
    dyb, _ = oracle.to_bits(dy)
    ref = oracle.conv_weight_grad(dyb, bits, keep, case.B, case.Ca, case.H, case.W, case.Cz, case.R, case.S, case.stride,
                                  case.pad, dt)
    cache = dropit.dropit_compress(x.to(cuda_device), case.gamma, "bitmask")
    args = (dy.to(cuda_device), cache, (case.R, case.S), case.stride, case.pad)
    dw = dropit.dropit_conv_weight_grad(*args)
    # exact bf16 products, fp32 sums: the bound that the other bf16 gradients are held to
    assert max_rel_err(dw.cpu().numpy(), ref) <= 2e-4
    twice = dropit.dropit_conv_weight_grad(*args, out=dw.clone(), accumulate=True)
    dropit.check_device_status(cuda_device)
    assert torch.equal(twice, dw + dw)      # the same sums in the same order


def test_fused_conv_waits_give_up_and_recover(cuda_device, monkeypatch):
    case = di.small_conv(16, 64, 56, 56, 64, 3, 3, 1, 1, "bf16", 0.8)
    cache = dropit.dropit_compress(di.make_x(case).to(cuda_device), case.gamma, "bitmask")
    dy = di.make_dy(case).to(cuda_device)
    good = dropit.dropit_conv_weight_grad(dy, cache, (3, 3), 1, 1)
    dropit.check_device_status(cuda_device)
    monkeypatch.setenv("DROPIT_TEST_SPIN_LIMIT", "1")
    dropit.dropit_conv_weight_grad(dy, cache, (3, 3), 1, 1)          # must return
    with pytest.raises(dropit.DropITError):
        dropit.check_device_status(cuda_device)
    monkeypatch.delenv("DROPIT_TEST_SPIN_LIMIT")
    again = dropit.dropit_conv_weight_grad(dy, cache, (3, 3), 1, 1)
    dropit.check_device_status(cuda_device)
    assert torch.equal(again, good)


# strided 1 x 1 filters with many outputs: the most work that is inflated per block of outputs, and the first that takes dense copies
@pytest.mark.parametrize("batch", [56, 64])
def test_strided_pointwise_either_side_of_the_line(cuda_device, batch):
    B, Ca, side, Cz = batch, 512, 27, 1024 + 8
    inflated = -(-Cz // 128) * B * Ca * ((side + 1) // 2) * 64
    assert (inflated >= 240_000_000) == (batch == 64)
    x = torch.randn(B, Ca, side, side, generator=torch.Generator().manual_seed(batch)).to(torch.bfloat16).to(cuda_device)
    cache = dropit.dropit_compress(x, 0.9)
    dy = torch.randn(B, Cz, 14, 14, device=cuda_device).to(torch.bfloat16)
    before = dropit.dropit_launch_count()
    dw = dropit.dropit_conv_weight_grad(dy, cache, (1, 1), 2, 0)
    launches = dropit.dropit_launch_count() - before
    dropit.check_device_status(cuda_device)
    assert (launches == 2) == (batch == 56)               # product and reduction, without decompression and gathered copies
    a = dropit.dropit_decompress(cache)[:, :, ::2, ::2].double()
    ref = torch.einsum("njyx,ncyx->jc", dy.double(), a)
    assert float((dw[:, :, 0, 0].double() - ref).abs().max()) <= 2e-4 * float(ref.abs().max())


# The forms of the reduction with more splits than a warp takes at once: three taps (all filters that have them in threes), nine taps, 16
# channels of a 1 x 1 filter, one tap.  (case, columns of a tile's sums in chunks of 32, tiles, splits at least)
SPLITS = [
    (di.small_conv(64, 120, 28, 28, 120, 3, 3, 1, 1, "bf16", 0.8), 14, 3, 33),
    (di.small_conv(64, 300, 9, 9, 100, 1, 3, 1, 1, "bf16", 0.8), 15, 2, 33),
    (di.small_conv(64, 300, 9, 9, 100, 3, 1, 1, 1, "bf16", 0.8), 8, 4, 25),
    (di.small_conv(64, 300, 9, 9, 100, 2, 3, 1, 1, "bf16", 0.8), 15, 4, 25),
    (di.small_conv(64, 300, 9, 9, 100, 3, 2, 2, 1, "bf16", 0.8), 15, 4, 25),
    (di.small_conv(24, 250, 14, 14, 250, 3, 3, 1, 1, "bf16", 0.8), 14, 12, 9),
    (di.small_conv(64, 250, 15, 15, 600, 1, 1, 1, 0, "bf16", 0.8), 8, 5, 17),
    (di.small_conv(64, 60, 28, 28, 60, 3, 3, 1, 1, "bf16", 0.8), 9, 2, 33),
]


@pytest.mark.parametrize("case,chunks,tiles,splits", SPLITS, ids=lambda v: getattr(v, "name", str(v)))
def test_many_splits_are_added_up(cuda_device, case, chunks, tiles, splits):
    size = dropit.dropit_conv_weight_grad_workspace(case.B, case.Ca, case.H, case.W, case.Cz, case.R, case.S, case.stride, case.pad, dropit.BF16,
                                                    dropit.FMT_BITMASK, cuda_device)
    assert size % (chunks * 32 * 128 * 4 * tiles) == 0 and size // (chunks * 32 * 128 * 4 * tiles) >= splits
    cache = dropit.dropit_compress(di.make_x(case).to(cuda_device), case.gamma, "bitmask")
    dy = di.make_dy(case).to(cuda_device)
    ref = conv_weight_grad_f64(dy, dropit.dropit_decompress(cache), (case.R, case.S), case.stride, case.pad)
    args = (dy, cache, (case.R, case.S), case.stride, case.pad)
    dw = dropit.dropit_conv_weight_grad(*args)
    assert float((dw.double() - ref).abs().max()) <= 2e-4 * float(ref.abs().max())
    twice = dropit.dropit_conv_weight_grad(*args, out=dw.clone(), accumulate=True)
    dropit.check_device_status(cuda_device)
    assert torch.equal(twice, dw + dw)
