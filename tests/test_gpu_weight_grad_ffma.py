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


# Either side of every line between the kernel's forms: tiles per SM, tokens, rows that are read by the element.
FORMS = [
    di.small_linear(8, 768, 768, "f32", 0.5, dy_std=1.0),         # a tile per SM: few tokens, less than a stage
    di.small_linear(48, 772, 708, "f32", 0.5, dy_std=1.0),        # ... the most tokens of that form, ragged tiles
    di.small_linear(49, 772, 708, "f32", 0.5, dy_std=1.0),        # ... one more
    di.small_linear(80, 772, 1000, "f32", 0.9, dy_std=1.0),       # more tiles than SMs
    di.small_linear(81, 772, 1000, "f32", 0.9, dy_std=1.0),
    di.small_linear(112, 770, 1001, "bf16", 0.9),                 # ... rows by the element
    di.small_linear(113, 770, 1001, "bf16", 0.9),
    di.small_linear(130, 1031, 1155, "bf16", 0.95),               # ... and more tiles than two per SM
    di.small_linear(1, 1031, 1155, "f32", 0.0, dy_std=1.0),
]


@pytest.mark.parametrize("case", FORMS, ids=lambda c: c.name)
def test_every_form_matches_oracle(cuda_device, case):
    test_ffma_weight_grad_matches_oracle(cuda_device, case, "bitmask")


def test_few_tokens_cost_little_more_than_the_output(cuda_device):
    """An fp32 gradient of a few tokens is a write of its output; it must not pay for the stages and sums of many tokens."""
    M, Ca, Cz = 8, 1024, 4096
    cache = dropit.dropit_compress(torch.randn(M, Ca, device=cuda_device), 0.5)
    dy = torch.randn(M, Cz, device=cuda_device)
    out, other = torch.empty(Cz, Ca, device=cuda_device), torch.randn(Cz, Ca, device=cuda_device)
    workspace = torch.empty(dropit.dropit_weight_grad_workspace(M, Ca, Cz, dropit.F32, cache.fmt, cuda_device), dtype=torch.uint8,
                            device=cuda_device)

    def microseconds(call):
        stream = torch.cuda.Stream()
        with torch.cuda.stream(stream):
            call()
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            for _ in range(10):
                call()
        best = float("inf")
        for _ in range(10):
            start, end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            start.record()
            graph.replay()
            end.record()
            torch.cuda.synchronize()
            best = min(best, start.elapsed_time(end) * 100)
        return best

    gradient = microseconds(lambda: dropit.dropit_weight_grad(dy, cache, out=out, workspace=workspace))
    copy = microseconds(lambda: out.copy_(other))       # one read and one write of as many bytes
    assert gradient < 2.5 * copy, (gradient, copy)      # 8 us and 4 us; 23 us with one CTA per SM and its sums over four groups
