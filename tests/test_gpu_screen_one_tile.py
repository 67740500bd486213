"""Row blocks against a single column tile: every block of a resident screen CTA then uses one of its
two accumulator buffers in turn, and several blocks follow one another on each SM.  Ids equal the
oracle's."""
import numpy as np
import pytest

import oracle
from paper_2510_05975_gb300 import synth

from gpu_util import host, lib, need_gpu, tensor

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,d,m", [(96, 24, 160_001), (60, 128, 100_000), (64, 250, 80_000), (97, 24, 80_000)])
def test_many_rows_against_one_tile(n, d, m):
    need_gpu()
    cng = lib()
    X = synth.generate("gauss", n, d, seed=91)
    Q = synth.generate("gauss", m, d, seed=92)
    ids, _, st = cng.cng_knn(tensor(X), 5, rows=tensor(Q))
    assert st["screen_used"] == 1
    assert np.array_equal(host(ids), oracle.knn(X, 5, rows=Q)[0])
