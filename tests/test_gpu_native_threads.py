"""The native calls let other Python threads run."""
import sys
import threading
import time

import pytest
import torch

import paper_2202_13808_b200 as dropit
from paper_2202_13808_b200 import api

pytestmark = pytest.mark.gpu


def test_calls_release_the_interpreter(cuda_device):
    M, C = 8192, 2048
    dy = torch.randn(M, C, device=cuda_device).to(torch.bfloat16)
    cache = dropit.dropit_compress(dy, 0.9)
    out = torch.empty(C, C, device=cuda_device)
    workspace = torch.empty(dropit.dropit_weight_grad_workspace(M, C, C, dropit.BF16, dropit.FMT_BITMASK, cuda_device), dtype=torch.uint8,
                            device=cuda_device)
    weight_grad = api._native().weight_grad
    args = (dy, cache.values, cache.meta, cache.offsets, cache.n, C, cache.k, cache.fmt, out, False, workspace, False)
    weight_grad(*args)
    turns, done = 0, False

    def other():
        nonlocal turns
        while not done:
            turns += 1
            time.sleep(0)

    thread = threading.Thread(target=other)
    interval = sys.getswitchinterval()
    sys.setswitchinterval(1000.0)             # no thread is interrupted: the other one runs when this one lets it
    try:
        thread.start()
        before = turns
        for _ in range(2000):                 # more launches than a stream's queue takes: later ones wait for their turn
            weight_grad(*args)
        after = turns
    finally:
        sys.setswitchinterval(interval)
        done = True
        thread.join()
    assert after > before
    dropit.check_device_status(cuda_device)
