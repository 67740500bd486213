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


def test_gradient_of_the_largest_batch():
    """2^22 samples: 0.70 GB of partial gradients and the activations of 131,072 samples (0.14 GB), not
    of all of them (4.6 GB)."""
    need_gpu()
    cng = lib()
    gen = torch.Generator(device="cuda").manual_seed(2)
    B = 1 << 22
    P = 0.1 * torch.randn(5313, device="cuda", generator=gen)
    x = torch.randn(B, 16, device="cuda", generator=gen)
    y = (torch.rand(B, device="cuda", generator=gen) < 0.5).float()
    assert _peak(lambda: cng.cng_mlp_grad(P, x, y)) < 1.0e9


def test_gradient_over_several_chunks():
    """A batch of two chunks of 131,072 samples and a rest: the sample-weighted mean of the parts'
    gradients.  Tolerance: three FP32 means whose entries are sums of up to 2,049 partials, each within
    (128 + 2,049 + 1) * 2^-24 of the sum of the terms' magnitudes, of which the largest entry is taken
    as a tenth: 2 * 2178 * 2^-24 * 10 < 3e-3 of the largest entry."""
    need_gpu()
    cng = lib()
    gen = torch.Generator(device="cuda").manual_seed(3)
    B = 2 * 131_072 + 77
    P = 0.1 * torch.randn(5313, device="cuda", generator=gen)
    x = torch.randn(B, 16, device="cuda", generator=gen)
    y = (torch.rand(B, device="cuda", generator=gen) < 0.5).float()
    loss, g = cng.cng_mlp_grad(P, x, y)
    ref, ref_loss = torch.zeros(5313, dtype=torch.double, device="cuda"), 0.0
    for part in (slice(0, 131_072), slice(131_072, 262_144), slice(262_144, B)):
        w = (min(part.stop, B) - part.start) / B
        li, gi = cng.cng_mlp_grad(P, x[part].contiguous(), y[part].contiguous())
        ref += w * gi.double()
        ref_loss += w * float(li)
    assert abs(float(loss) - ref_loss) <= 1e-4 * ref_loss
    assert (g.double() - ref).abs().max() <= 3e-3 * ref.abs().max()
