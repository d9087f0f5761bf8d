"""Selection where the sampled band of keys is about as wide as the per-warp histograms hold, a little less and more; zeros in the sample."""
import pytest
import torch

import paper_2202_13808_b200 as dropit
from _parity import assert_cache_matches_oracle, oracle_cache

pytestmark = pytest.mark.gpu

N = (1 << 20) + 517          # sampled path, a ragged last super-block


# |x| log-uniform over `octaves`: 128 * octaves keys with the same mass, of which the band at gamma 0.5 holds about a tenth: 38 to 180 keys
@pytest.mark.parametrize("octaves", [3, 5, 6, 7, 8, 14])
def test_band_widths(cuda_device, octaves):
    g = torch.Generator().manual_seed(octaves)
    x = (torch.exp2(torch.rand(N, generator=g) * octaves - 4) * torch.randn(N, generator=g).sign()).to(torch.bfloat16)
    _check(x, 0.5, cuda_device)


# all but the retained share (and a little more, and less) exact zeros: the band reaches the lowest key
@pytest.mark.parametrize("zeros", [0.0, 0.5, 0.895, 0.9, 0.905, 1.0])
def test_zeros_in_the_sample(cuda_device, zeros):
    g = torch.Generator().manual_seed(5)
    x = torch.randn(N, generator=g)
    x[torch.rand(N, generator=g) < zeros] = 0.0
    _check(x.to(torch.bfloat16), 0.9, cuda_device)


def _check(x, gamma, device):
    bits, dt, keep, k = oracle_cache(x, gamma)
    cache = dropit.dropit_compress(x.to(device), gamma, "bitmask")
    dropit.check_device_status(device)
    assert_cache_matches_oracle(cache, bits, dt, keep, k, "bitmask")
