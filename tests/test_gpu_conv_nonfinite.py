"""Infinities and NaN among the retained values of a convolution's input reach exactly the taps that see them."""
import numpy as np
import pytest
import torch

import dropit_inputs as di
import oracle
import paper_2202_13808_b200 as dropit
from _parity import max_rel_err, oracle_cache

pytestmark = pytest.mark.gpu

# rows that end inside an 8-pixel group, an odd number of such groups in a band, several images in a band, two blocks of
# outputs, a padded tap at every side, stride 2 with even and odd columns; rows of whole groups for comparison
CASES = [
    di.small_conv(2, 17, 14, 14, 65, 3, 3, 1, 1, "bf16", 0.5),
    di.small_conv(3, 16, 7, 7, 130, 3, 3, 1, 1, "bf16", 0.5),
    di.small_conv(1, 16, 56, 56, 16, 3, 3, 1, 1, "bf16", 0.5),
    di.small_conv(2, 16, 12, 20, 24, 3, 3, 1, 0, "bf16", 0.5),
    di.small_conv(2, 20, 14, 14, 40, 3, 3, 2, 1, "bf16", 0.5),
    di.small_conv(2, 16, 16, 16, 16, 3, 3, 1, 1, "bf16", 0.5),
    di.small_conv(2, 16, 15, 15, 16, 1, 1, 1, 0, "bf16", 0.5),
]


def _places(h, w):
    return [(y, x) for y in (0, h // 2, h - 1) for x in (0, w // 2, w - 2, w - 1)]


@pytest.mark.parametrize("case", CASES, ids=lambda c: c.name)
def test_nonfinite_values_stay_where_they_are_seen(cuda_device, case):
    dy = di.make_dy(case)
    dyb, _ = oracle.to_bits(dy)
    for i, (y, x) in enumerate(_places(case.H, case.W)):
        a = di.make_x(case)
        a[case.B - 1, 3, y, x] = (float("inf"), float("-inf"), float("nan"))[i % 3]
        a[0, case.Ca - 1, (y + 5) % case.H, (x + 3) % case.W] = float("inf")
        bits, dt, keep, _ = oracle_cache(a, case.gamma)
        with np.errstate(invalid="ignore"):
            ref = oracle.conv_weight_grad(dyb, bits, keep, case.B, case.Ca, case.H, case.W, case.Cz, case.R, case.S, case.stride,
                                          case.pad, dt)
        cache = dropit.dropit_compress(a.to(cuda_device), case.gamma, "bitmask")
        dw = dropit.dropit_conv_weight_grad(dy.to(cuda_device), cache, (case.R, case.S), case.stride, case.pad)
        dropit.check_device_status(cuda_device)
        got = dw.cpu().numpy()
        finite = np.isfinite(ref)
        assert (~finite).any() and (np.isfinite(got) == finite).all(), (y, x)
        assert (got[np.isinf(ref)] == ref[np.isinf(ref)]).all() and (np.isnan(got) == np.isnan(ref)).all(), (y, x)
        # exact bf16 products, fp32 sums: the bound that the other bf16 gradients are held to
        assert max_rel_err(got[finite], ref[finite]) <= 2e-4


# the reduction's forms: all nine taps of four channels per block, three taps, 16 channels of a 1 x 1 filter; ragged in both channel counts
@pytest.mark.parametrize("case", [
    di.small_conv(2, 299, 6, 6, 250, 3, 3, 1, 1, "bf16", 0.5),
    di.small_conv(2, 61, 6, 9, 250, 3, 3, 1, 1, "bf16", 0.5),
    di.small_conv(2, 300, 5, 5, 500, 1, 1, 1, 0, "bf16", 0.5),
], ids=lambda c: c.name)
def test_every_form_of_the_reduction(cuda_device, case):
    cache = dropit.dropit_compress(di.make_x(case).to(cuda_device), case.gamma, "bitmask")
    args = (di.make_dy(case).to(cuda_device), cache, (case.R, case.S), case.stride, case.pad)
    dw = dropit.dropit_conv_weight_grad(*args)
    assert torch.equal(dropit.dropit_conv_weight_grad(*args, out=dw.clone(), accumulate=True), dw + dw)
    test_nonfinite_values_stay_where_they_are_seen(cuda_device, case)
