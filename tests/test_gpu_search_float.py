"""The register-queue search on FP32 and FP16 rows where its order is hardest to get right: queues
filled exactly, by one less and one more than their registers hold, and points whose distances tie
to the last FP32 bits (duplicates, jittered copies), against the oracle's FP64 order; the
near-ties of candidate lists on the same data."""
import numpy as np
import pytest

import oracle
from paper_2510_05975_gb300 import synth

from gpu_util import host, lib, need_gpu, tensor
from test_gpu_search import _search_check

pytestmark = pytest.mark.gpu


def _tied(kind, n, d, seed, dtype="float32"):
    """n rows: a third of them copies, a third jittered by a few units in the last place."""
    X = synth.generate(kind, n, d, seed=seed, dtype=dtype).astype(np.float32)
    rng = np.random.default_rng(seed)
    m = n // 3
    X[m:2 * m] = X[:m]
    X[2 * m:3 * m] = X[:m] * (1 + 2.0 ** -22 * rng.integers(-3, 4, (m, d)))
    return X.astype(dtype)


# widths 1 .. 960: one chunk per lane and several, with and without a rest; queues of 32 QS - 1,
# 32 QS and 32 QS + 1 entries
@pytest.mark.parametrize("kind,d,L,dtype", [
    ("gauss", 8, 31, "float32"), ("gauss", 24, 32, "float32"), ("deep", 96, 33, "float32"),
    ("gauss", 40, 64, "float32"), ("deep", 130, 128, "float32"), ("gauss", 24, 256, "float32"),
    ("gist", 960, 65, "float32"), ("bigann16", 64, 32, "float16"), ("bigann16", 128, 64, "float16"),
    ("bigann16", 200, 129, "float16"),
])
def test_tied_distances(kind, d, L, dtype):
    need_gpu()
    cng = lib()
    X = _tied(kind, 2400, d, 51, dtype)
    Q = synth.generate(kind, 150, d, seed=52, centre_seed=51)
    Q[:40] = X[:40].astype(np.float32)  # zero distances
    idx, st = cng.cng_build(tensor(X), alpha=1.2, R=20, L=60, repair_slots=24, connect_L=64, keep_lists=True)
    cand = host(cng.cng_lists(idx)[0])
    assert np.array_equal(cand, oracle.knn(X.astype(np.float32), 60)[0])
    _search_check(X.astype(np.float32), Q, idx, cng, min(10, L), L)
    cng.cng_free(idx)


# row strides of 33 to 96 slots: a hop's new points in one, two and three batches
@pytest.mark.parametrize("R,slots", [(25, 8), (64, 1), (64, 32)])
def test_wide_rows(R, slots):
    need_gpu()
    cng = lib()
    X = synth.generate("gauss", 4000, 20, seed=53)
    Q = synth.generate("gauss", 100, 20, seed=54)
    idx, _ = cng.cng_build(tensor(X), alpha=2.0, R=R, L=128, repair_slots=slots)
    for L in (16, 100):
        _search_check(X, Q, idx, cng, 10, L)
    cng.cng_free(idx)
