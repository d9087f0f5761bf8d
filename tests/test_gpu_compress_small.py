"""One-cluster selection (tensors of up to 2^19 elements): bit-exact against the oracle where its work partition changes."""
import numpy as np
import pytest
import torch

import paper_2202_13808_b200 as dropit
from _parity import assert_cache_matches_oracle, oracle_cache

pytestmark = pytest.mark.gpu

# one CTA / two CTAs / the full cluster, its last element and the first size that another kernel takes; ragged in between
SIZES = [8 * 1024, 8 * 1024 + 1, 16 * 8 * 1024, 16 * 8 * 1024 + 1023, 300_007, (1 << 19) - 1, 1 << 19, (1 << 19) + 1]


def _draw(n, law, dtype):
    g = torch.Generator().manual_seed(n)
    if law == "normal":
        return torch.randn(n, generator=g).to(dtype)
    if law == "relu":        # half zeros: the threshold falls inside the ties at gamma = 0.3
        return torch.relu(torch.randn(n, generator=g)).to(dtype)
    return torch.randint(0, 3, (n,), generator=g).to(dtype)     # three levels: every digit round ends in one bin


@pytest.mark.parametrize("fmt", ["bitmask", "index32"])
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32], ids=["bf16", "f32"])
@pytest.mark.parametrize("n", SIZES)
def test_small_tensors_match_the_oracle(cuda_device, n, dtype, fmt):
    for law, gamma in (("normal", 0.9), ("relu", 0.3), ("levels", 0.5)):
        x = _draw(n, law, dtype)
        bits, dt, keep, k = oracle_cache(x, gamma)
        cache = dropit.dropit_compress(x.to(cuda_device), gamma, fmt)
        dropit.check_device_status(cuda_device)
        assert_cache_matches_oracle(cache, bits, dt, keep, k, fmt)


# fp32 keys that share their upper 15 bits: up to 1024 of them are ranked from a list, more by counting their lower digits in turn
@pytest.mark.parametrize("matching", [1, 37, 1023, 1024, 1025, 4095, 4096, 4097, 9000])
@pytest.mark.parametrize("front", [0, 20000])
def test_keys_that_match_in_their_upper_bits(cuda_device, matching, front):
    gen = torch.Generator().manual_seed(matching + front)
    low = torch.randint(0, 1 << 16, (matching,), generator=gen)
    low[::5] = low[0]                                          # ties, at the threshold too for some of the counts below
    same = (low + (0x3F80 << 16)).to(torch.int32)              # 1.0 .. 1.0078
    others = torch.where(torch.rand(front, generator=gen) < 0.5, 0.25, -3.0).view(torch.int32)
    bits = torch.cat([others, same])[torch.randperm(matching + front, generator=gen)]
    x = bits.view(torch.float32)
    above = int((others.view(torch.float32).abs() > 1).sum())
    for kept in {above + 1, above + (matching + 1) // 2, above + matching}:
        gamma = 1.0 - kept / x.numel()
        xb, dt, keep, k = oracle_cache(x, gamma)
        cache = dropit.dropit_compress(x.to(cuda_device), gamma)
        assert_cache_matches_oracle(cache, xb, dt, keep, k, "bitmask")


def test_few_matching_keys_take_no_longer_than_many(cuda_device):
    """Keys that match in their upper bits and lie side by side: as many as are ranked from a list, or almost, cost no more than as many as
    certainly are counted."""
    n, gen = 196608, torch.Generator(device=cuda_device).manual_seed(5)

    def microseconds(matching):
        x = torch.randn(n, generator=gen, device=cuda_device)
        x = torch.where((x.abs() >= 1) & (x.abs() < 1.0079), x * 1.05, x)
        x[:matching] = 1.0 + torch.rand(matching, generator=gen, device=cuda_device) * 0.0077
        gamma = 1.0 - (int((x.abs() >= 1.0079).sum()) + matching / 2) / n             # the threshold is one of them
        workspace = torch.empty(max(16, dropit.dropit_cache_sizes(n, gamma, dropit.F32, dropit.FMT_BITMASK)[3]), dtype=torch.uint8,
                                device=cuda_device)
        stream = torch.cuda.Stream()
        with torch.cuda.stream(stream):
            dropit.dropit_compress(x, gamma, workspace=workspace)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            for _ in range(20):
                dropit.dropit_compress(x, gamma, workspace=workspace)
        best = float("inf")
        for _ in range(10):
            start, end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            start.record()
            graph.replay()
            end.record()
            torch.cuda.synchronize()
            best = min(best, start.elapsed_time(end) * 50)
        return best

    many = microseconds(4200)
    for matching in (1024, 2000, 4000):
        # 13.6, 14.8 and 15.8 us against 16; a list of 4000 took 21 us
        assert microseconds(matching) < 1.15 * many, matching
