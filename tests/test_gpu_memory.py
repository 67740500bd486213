"""Device memory that a call holds at its peak, by polling the free memory while it runs."""
import threading

import pytest
import torch

from gpu_util import lib, need_gpu

pytestmark = pytest.mark.gpu


def _peak(call):
    call()  # first use: caches
    torch.cuda.synchronize()
    base = torch.cuda.mem_get_info()[0]
    low, stop = [base], threading.Event()

    def poll():
        while not stop.is_set():
            low[0] = min(low[0], torch.cuda.mem_get_info()[0])

    t = threading.Thread(target=poll)
    t.start()
    call()
    stop.set()
    t.join()
    return base - low[0]


def test_build_keeps_no_screen_scratch():
    """A build holds its largest set of buffers in the merge: 4.17 GB at 1M x 128; with the order's
    scratch and the columns' operand image kept until its end it was 4.55 GB."""
    need_gpu()
    cng = lib()
    X = torch.randn(1_000_000, 128, device="cuda", generator=torch.Generator(device="cuda").manual_seed(1))

    def build():
        idx, _ = cng.cng_build(X, alpha=1.2, R=32, L=128, connect_L=-1)
        cng.cng_free(idx)

    assert _peak(build) < 4.35e9
