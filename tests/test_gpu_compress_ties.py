"""Selection where one run of the tensor holds the end of the tie quota and all others decide by a single threshold."""
import pytest
import torch

import paper_2202_13808_b200 as dropit
from _parity import assert_cache_matches_oracle, oracle_cache

pytestmark = pytest.mark.gpu

N = (1 << 20) + 517          # sampled path, a ragged last super-block


def _tensor(kind):
    g = torch.Generator().manual_seed(3)
    x = torch.randn(N, generator=g).to(torch.bfloat16)
    if kind == "levels":         # the threshold is one of three keys: ties in every run
        x = torch.randint(0, 3, (N,), generator=g).to(torch.bfloat16)
    elif kind == "nan":          # the threshold among NaN and Inf patterns
        bits = torch.randint(0x7F70, 0x7FFF, (N,), generator=g, dtype=torch.int16)
        x = bits.view(torch.bfloat16)
    elif kind == "subnormal":
        x = (torch.randn(N, generator=g) * 1e-39).to(torch.bfloat16)
    return x


@pytest.mark.parametrize("gamma", [0.95, 0.84, 0.5, 0.02])       # sparse and dense words, both sides of the line between them
@pytest.mark.parametrize("kind", ["normal", "levels", "nan", "subnormal"])
def test_tie_quota_and_thresholds(cuda_device, kind, gamma):
    x = _tensor(kind)
    bits, dt, keep, k = oracle_cache(x, gamma)
    for fmt in ("bitmask", "index32"):
        cache = dropit.dropit_compress(x.to(cuda_device), gamma, fmt)
        dropit.check_device_status(cuda_device)
        assert_cache_matches_oracle(cache, bits, dt, keep, k, fmt)
