"""fp32 weight gradients and bf16 shapes that the tensor cores do not take, and caches in coordinate format: at the edges
of tiles, token stages and 1024-element steps."""
import pytest
import torch

import dropit_inputs as di
import oracle
import paper_2202_13808_b200 as dropit
from _parity import max_rel_err, oracle_cache

pytestmark = pytest.mark.gpu

CASES = [
    di.small_linear(1, 1, 1, "f32", 0.0, dy_std=1.0),
    di.small_linear(33, 65, 31, "f32", 0.5, dy_std=1.0),          # narrow tiles, ragged everywhere
    di.small_linear(31, 772, 836, "f32", 0.5, dy_std=1.0),        # wide tiles, one partial stage, rows of whole vectors
    di.small_linear(97, 770, 834, "f32", 0.9, dy_std=1.0),        # wide tiles, rows that start anywhere
    di.small_linear(200, 704, 100, "bf16", 0.8),                  # classifier with 100 classes
    di.small_linear(513, 1023, 10, "bf16", 0.9),
    di.small_linear(64, 192, 1000, "bf16", 0.9),                  # few tokens: the tensor cores are not worth setting up
    di.small_linear(65, 192, 1000, "bf16", 0.9),                  # ... and one more, where they are
]


@pytest.mark.parametrize("fmt", ["bitmask", "index32"])
@pytest.mark.parametrize("case", CASES, ids=lambda c: c.name)
def test_ffma_weight_grad_matches_oracle(cuda_device, case, fmt):
    x, dy = di.make_x(case), di.make_dy(case)
    bits, dt, keep, _ = oracle_cache(x, case.gamma)
    dyb, _ = oracle.to_bits(dy)
    ref = oracle.fc_weight_grad(dyb, bits, keep, case.M, case.Ca, case.Cz, dt)
    cache = dropit.dropit_compress(x.to(cuda_device), case.gamma, fmt)
    dense = dropit.dropit_decompress(cache)
    assert torch.equal(dense.cpu(), torch.where(torch.from_numpy(keep.astype(bool)).reshape(x.shape), x, torch.zeros_like(x)))
    dw = dropit.dropit_weight_grad(dy.to(cuda_device), cache)
    assert max_rel_err(dw.cpu().numpy(), ref) <= 1e-5      # products exact or rounded to fp32, fp32 sums of at most 513 terms
    twice = dropit.dropit_weight_grad(dy.to(cuda_device), cache, out=dw.clone(), accumulate=True)
    dropit.check_device_status(cuda_device)
    assert torch.equal(twice, dw + dw)
