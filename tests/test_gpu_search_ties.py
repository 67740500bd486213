"""Searches on float rows with many exactly tied distances (coordinates from few levels): whole groups
of points tie at the end of the queue, among them points that a hop drops.  Ids and hops equal the
FP64 oracle's on the same graph."""
import numpy as np
import pytest

from gpu_util import lib, need_gpu, tensor
from test_gpu_search import _search_check

pytestmark = pytest.mark.gpu


# queues that fill their registers exactly (32, 64, 128, 256) and others; two levels: equal distances
# are equal sums; more levels: equal up to the rounding of the coordinates
@pytest.mark.parametrize("levels,d,L,dtype", [
    (2, 24, 32, "float32"), (2, 64, 32, "float32"), (2, 64, 64, "float32"), (2, 96, 64, "float32"),
    (2, 96, 128, "float32"), (2, 24, 256, "float32"), (2, 64, 64, "float16"), (2, 96, 61, "float32"),
    (3, 64, 32, "float32"), (5, 48, 64, "float32"), (16, 24, 128, "float32"), (3, 100, 64, "float16"),
])
def test_points_of_few_levels(levels, d, L, dtype):
    need_gpu()
    cng = lib()
    rng = np.random.default_rng(101)
    grid = (np.arange(levels) - (levels - 1) / 2).astype(np.float32) * np.float32(0.2)
    X = grid[rng.integers(0, levels, (2400, d))].astype(dtype).astype(np.float32)
    Q = grid[rng.integers(0, levels, (120, d))].astype(dtype).astype(np.float32)
    Q[60:] += 0.05 * rng.standard_normal((60, d)).astype(np.float32)  # and queries off the levels
    idx, st = cng.cng_build(tensor(X.astype(dtype)), alpha=1.2, R=24, L=64, repair_slots=32, connect_L=128)
    assert st["exact_int"] == 0
    _search_check(X, Q, idx, cng, min(10, L), L)
    cng.cng_free(idx)


def test_copies_cost_no_fp64_sums():
    """Every point stored twice: the pairs' order is their ids', found without FP64 sums.  Searches
    take at most 20 times those of single points (2 measured; with every tied pair of the queue
    compared in FP64 after each hop it was 330 times)."""
    need_gpu()
    cng = lib()
    rng = np.random.default_rng(103)
    X = rng.standard_normal((8000, 96)).astype(np.float32)
    Q = tensor(rng.standard_normal((1000, 96)).astype(np.float32))
    ms = []
    for rows in (X, np.tile(X[:4000], (2, 1))):
        idx, _ = cng.cng_build(tensor(rows), alpha=1.2, R=24, L=64, repair_slots=32, connect_L=64)
        runs = [cng.cng_search(idx, Q, k=10, L=128, warps_per_block=4, with_stats=True)["stats"]["ms"]
                for _ in range(4)]
        ms.append(min(runs))
        cng.cng_free(idx)
    assert ms[1] <= 20 * ms[0], ms
