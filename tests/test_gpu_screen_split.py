"""Screens whose few row blocks are split over the columns: one row, less than a block, one block and
one row more, several blocks, self lists of several blocks; long and short lists.  Ids equal the
oracle's, distances to FP32 rounding (d additions of relative 2^-24 each)."""
import numpy as np
import pytest

import oracle
from paper_2510_05975_gb300 import synth

from gpu_util import host, lib, need_gpu, tensor

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,n,d,m,k", [("sift", 60_007, 128, 1, 100), ("deep", 90_000, 96, 255, 1),
                                          ("gauss", 50_021, 20, 257, 256), ("bigann16", 30_011, 200, 1500, 33),
                                          ("gauss", 9_999, 12, 0, 64), ("sift", 20_001, 64, 0, 200)])
def test_split_lists(kind, n, d, m, k):
    need_gpu()
    cng = lib()
    X = synth.generate(kind, n, d, seed=51)
    Q = synth.generate(kind, m, d, seed=52, centre_seed=51) if m else None
    ids, ds, st = cng.cng_knn(tensor(X), k, rows=tensor(Q) if m else None)
    ref, rd = oracle.knn(X, k, rows=Q)
    assert st["screen_used"] == 1 and st["cert_fail_rows"] == 0
    assert np.array_equal(host(ids), ref)
    assert np.allclose(host(ds), rd, rtol=2e-5)


def test_split_certifies_clustered_rows():
    """All of a row's nearest columns in one split's tiles: tight clusters of one tile's width, so a
    split's share of a row's list is all or nothing.  Every list certifies."""
    need_gpu()
    cng = lib()
    rng = np.random.default_rng(53)
    X = np.repeat(rng.normal(size=(400, 24)) * 10, 96, axis=0) + 0.1 * rng.normal(size=(38_400, 24))
    X = X.astype(np.float32)
    Q = X[::311] + np.float32(0.01)
    ids, _, st = cng.cng_knn(tensor(X), 96, rows=tensor(Q))
    assert st["cert_fail_rows"] == 0
    assert np.array_equal(host(ids), oracle.knn(X, 96, rows=Q)[0])
