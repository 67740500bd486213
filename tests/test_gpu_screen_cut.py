"""Lists of the resident screen that overflow inside a part of the sweep and are cut there (the cut
reads what 32 lanes have just appended): short and long lists, every operand width class, capacities
of 384 to 768 entries.  Ids equal the oracle's."""
import numpy as np
import pytest

import oracle
from paper_2510_05975_gb300 import synth

from gpu_util import host, lib, need_gpu, tensor

pytestmark = pytest.mark.gpu


# n below 1/64 x 4 tiles: the first part has 1/16 or all of the columns, several times a capacity
@pytest.mark.parametrize("n,d,k", [(3000, 24, 10), (3000, 128, 128), (20_000, 24, 100), (20_000, 150, 192),
                                   (9000, 230, 256)])
def test_cut_lists(n, d, k):
    need_gpu()
    cng = lib()
    X = synth.generate("gauss", n, d, seed=81)
    ids, _, st = cng.cng_knn(tensor(X), k)
    assert st["screen_used"] == 1 and st["cert_fail_rows"] == 0
    assert np.array_equal(host(ids), oracle.knn(X, k)[0])
