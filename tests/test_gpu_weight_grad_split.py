"""How the token blocks of few output tiles are shared out among CTA pairs: whole ranges per pair with tickets, or evenly with
pairs that cross from one tile into the next."""
import pytest
import torch

import dropit_inputs as di
import oracle
import paper_2202_13808_b200 as dropit
from _parity import max_rel_err, oracle_cache

pytestmark = pytest.mark.gpu

CASES = [
    di.small_linear(145, 264, 136, "bf16", 0.9),       # two token blocks, one of them nearly empty
    di.small_linear(9000, 256, 768, "bf16", 0.9),      # three tiles for all pairs: even split, many pairs per tile
    di.small_linear(10007, 200, 520, "bf16", 0.95),    # ... ragged tiles and a ragged last block
    di.small_linear(7000, 520, 776, "bf16", 0.95),     # twelve tiles: pairs cross tile boundaries at uneven places
    di.small_linear(12000, 800, 2304, "bf16", 0.97),   # 36 tiles, whole ranges only
    di.small_linear(9300, 776, 2056, "bf16", 0.97),    # 36 ragged tiles
    di.small_linear(11000, 768, 2304, "bf16", 0.97),   # 27 tiles: two ranges per tile with tickets
    di.small_linear(7001, 1032, 2000, "bf16", 0.97),   # 40 tiles: one range per tile and the rests
    di.small_linear(700, 768, 768, "bf16", 0.9),       # a few blocks: no split
    di.small_linear(4000, 1536, 384, "bf16", 0.95),    # 12 tiles: six pairs each, none of which crosses into the next
]


@pytest.mark.parametrize("case", CASES, ids=lambda c: c.name)
def test_split_weight_grad_matches_oracle(cuda_device, case):
    x, dy = di.make_x(case), di.make_dy(case)
    bits, dt, keep, _ = oracle_cache(x, case.gamma)
    dyb, _ = oracle.to_bits(dy)
    ref = oracle.fc_weight_grad(dyb, bits, keep, case.M, case.Ca, case.Cz, dt)
    cache = dropit.dropit_compress(x.to(cuda_device), case.gamma)
    dyd = dy.to(cuda_device)
    dw = dropit.dropit_weight_grad(dyd, cache)
    assert max_rel_err(dw.cpu().numpy(), ref) <= 2e-4      # exact bf16 products, fp32 sums: the bound of the other bf16 gradients
    assert torch.equal(dropit.dropit_weight_grad(dyd, cache), dw)                                     # fixed order
    assert torch.equal(dropit.dropit_weight_grad(dyd, cache, out=dw.clone(), accumulate=True), dw + dw)
    dropit.check_device_status(cuda_device)


# The way that the plan takes, as it shows outside: the even split adds up in a launch of its own, and the workspace holds a plane of
# whole tiles per range.
WAYS = [
    (di.small_linear(700, 768, 768, "bf16", 0.9), 2, 0),       # no split
    (di.small_linear(2000, 768, 2304, "bf16", 0.97), 2, 2),    # two ranges with tickets
    (di.small_linear(3001, 1024, 1536, "bf16", 0.97), 2, 3),   # three
    (di.small_linear(4000, 1536, 384, "bf16", 0.95), 3, 6),    # even split, whole ranges of equal length
    (di.small_linear(9000, 256, 768, "bf16", 0.9), 3, 24),     # ... of many pairs
    (di.small_linear(7001, 1032, 2000, "bf16", 0.97), 3, 3),   # ... one range per tile, the rests shared out by pairs that cross tiles
    (di.small_linear(13001, 768, 2304, "bf16", 0.98), 3, 4),   # ... two ranges per tile and the rests
]


@pytest.mark.parametrize("case, launches, planes", WAYS, ids=lambda v: getattr(v, "name", None))
def test_every_way_to_split_is_taken_and_matches_oracle(cuda_device, case, launches, planes):
    size = dropit.dropit_weight_grad_workspace(case.M, case.Ca, case.Cz, dropit.BF16, dropit.FMT_BITMASK, cuda_device)
    tiles = 2 * -(-case.Cz // 256) * -(-case.Ca // 256)
    assert (size - case.M * case.Ca * 2) // (tiles * 128 * 256 * 4) == planes
    cache = dropit.dropit_compress(di.make_x(case).to(cuda_device), case.gamma)
    dy = di.make_dy(case).to(cuda_device)
    before = dropit.dropit_launch_count()
    dropit.dropit_weight_grad(dy, cache)
    assert dropit.dropit_launch_count() - before == launches
    test_split_weight_grad_matches_oracle(cuda_device, case)


def test_even_split_waits_give_up_and_recover(cuda_device, monkeypatch):
    case = di.small_linear(9000, 256, 768, "bf16", 0.9)
    cache = dropit.dropit_compress(di.make_x(case).to(cuda_device), case.gamma)
    dy = di.make_dy(case).to(cuda_device)
    good = dropit.dropit_weight_grad(dy, cache)
    dropit.check_device_status(cuda_device)
    monkeypatch.setenv("DROPIT_TEST_SPIN_LIMIT", "1")
    dropit.dropit_weight_grad(dy, cache)                    # must return
    with pytest.raises(dropit.DropITError):
        dropit.check_device_status(cuda_device)
    monkeypatch.delenv("DROPIT_TEST_SPIN_LIMIT")
    again = dropit.dropit_weight_grad(dy, cache)
    dropit.check_device_status(cuda_device)
    assert torch.equal(again, good)
