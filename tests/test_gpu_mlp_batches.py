"""Batch gradients of the stop model at the edges of the kernels' tiles (32 samples per forward CTA,
128 per partial gradient), against the FP64 oracle.  Tolerance: each entry is a chain of FP32 FMAs over
at most 128 samples, then over the groups, of terms no larger than a few times the largest entry:
(128 + 33 + 64) * 2^-24 * 4 < 1e-4 of the largest entry."""
import numpy as np
import pytest

from gpu_util import host, lib, need_gpu, tensor
from oracle import mlp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B", [1, 31, 33, 127, 128, 129, 4096, 4225])
def test_gradient_at_tile_edges(B):
    need_gpu()
    cng = lib()
    rng = np.random.default_rng(B)
    P = mlp.init(5).astype(np.float32)
    X = rng.standard_normal((B, 16)).astype(np.float32)
    y = (rng.random(B) < 0.6).astype(np.float32)
    loss, g = cng.cng_mlp_grad(tensor(P), tensor(X), tensor(y))
    ref_loss, ref_g = mlp.loss_and_grad(P.astype(np.float64), X.astype(np.float64),
                                        y.astype(np.float64))
    assert abs(float(loss.item()) - ref_loss) <= 1e-5 * abs(ref_loss)
    err = np.abs(host(g).astype(np.float64) - ref_g)
    assert err.max() <= 1e-4 * np.abs(ref_g).max() + 1e-7
