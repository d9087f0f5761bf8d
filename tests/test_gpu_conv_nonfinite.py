"""Infinities and NaN among the retained values of a convolution's input reach exactly the taps that see them."""
import numpy as np
import pytest
import torch

import dropit_inputs as di
import oracle
import paper_2202_13808_b200 as dropit
from _parity import conv_weight_grad_f64, max_rel_err, oracle_cache

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


def _layer(device, B, Ca, side, Cz, R, stride, pad):
    gen = torch.Generator(device=device).manual_seed(Ca + side)
    x = torch.relu(torch.randn(B, Ca, side, side, generator=gen, device=device)).to(torch.bfloat16)
    out = (side + 2 * pad - R) // stride + 1
    return x, torch.randn(B, Cz, out, out, generator=gen, device=device).mul_(0.02).to(torch.bfloat16)


# nine taps, three taps, one tap per block, 16 channels of a 1 x 1 filter; more pixels than one round of them, images for every warp
@pytest.mark.parametrize("shape", [(20, 250, 14, 250, 3, 1, 1), (20, 120, 13, 120, 3, 2, 1), (12, 24, 20, 40, 3, 1, 1), (20, 250, 7, 600, 1, 1, 0)],
                         ids=lambda s: "x".join(map(str, s)))
def test_nonfinite_values_among_many_images(cuda_device, shape):
    x, dy = _layer(cuda_device, *shape)
    B, Ca, side, Cz, R, stride, pad = shape
    x[B - 1, 3, side - 1, side - 2] = float("inf")                # two channels of one block, one of another
    x[2, 0, 0, 1] = float("nan")
    x[B // 2, Ca - 1, side // 2, side // 2] = float("-inf")
    cache = dropit.dropit_compress(x, 0.8)
    ref = conv_weight_grad_f64(dy, dropit.dropit_decompress(cache), (R, R), stride, pad)
    finite = torch.isfinite(ref)
    for bad in (None, float("nan"), float("inf")):
        rows = torch.arange(Cz, device=cuda_device)
        if bad is not None:                                       # ... and a row of dY, which turns all of its sums
            dy[1, Cz - 2, 1, 0] = bad
            rows = rows[rows != Cz - 2]
        got = dropit.dropit_conv_weight_grad(dy, cache, (R, R), stride, pad)
        dropit.check_device_status(cuda_device)
        if bad is not None:
            clean = torch.tensor([c for c in range(Ca) if c not in (0, 3, Ca - 1)], device=cuda_device)
            assert not torch.isfinite(got[Cz - 2, clean]).any()
        for c in range(0, Ca, 64):
            g, r, f = (t[rows][:, c:c + 64] for t in (got, ref, finite))
            assert (torch.isfinite(g) == f).all() and (g[~f].double().nan_to_num(nan=7.0) == r[~f].nan_to_num(nan=7.0)).all()
            assert float((g[f].double() - r[f]).abs().max()) <= 2e-4 * float(ref[finite].abs().max())


def test_one_odd_value_costs_a_look_at_its_channels(cuda_device):
    B, Ca, side, Cz = 64, 256, 14, 256
    x, dy = _layer(cuda_device, B, Ca, side, Cz, 3, 1, 1)
    workspace = torch.empty(dropit.dropit_conv_weight_grad_workspace(B, Ca, side, side, Cz, 3, 3, 1, 1, dropit.BF16, dropit.FMT_BITMASK, cuda_device),
                            dtype=torch.uint8, device=cuda_device)
    out = torch.empty(Cz, Ca, 3, 3, device=cuda_device)

    def microseconds(x, dy):
        cache = dropit.dropit_compress(x, 0.8)
        best = float("inf")
        for _ in range(5):
            start, end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            start.record()
            for _ in range(20):
                dropit.dropit_conv_weight_grad(dy, cache, (3, 3), 1, 1, out=out, workspace=workspace)
            end.record()
            torch.cuda.synchronize()
            best = min(best, start.elapsed_time(end) * 50)
        return best

    odd_x, odd_dy = x.clone(), dy.clone()
    odd_x[B // 2, 3, 2, 3] = float("inf")
    odd_dy[B // 2, 5, 2, 3] = float("nan")
    plain = microseconds(x, dy)
    # 34, 40 and 297 us; 359 and 1369 us when each tap searched the channels and summed by itself
    assert microseconds(x, odd_dy) < 4 * plain
    assert microseconds(odd_x, dy) < 20 * plain
