"""FP16 collections of small norm through the tensor-core screen: the screen's FP16 pieces of the
column norms resolve an absolute 2^-24, so unscaled operands with coordinates below about 1e-3 gave
lists that were certified and wrong.  Candidate lists equal the oracle's at every magnitude."""
import numpy as np
import pytest

import oracle
from paper_2510_05975_gb300 import synth

from gpu_util import host, lib, need_gpu, tensor

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,d,amax", [("bigann16", 128, 1e-2), ("bigann16", 128, 1e-3), ("bigann16", 128, 5e-4),
                                         ("bigann16", 128, 3e-4), ("bigann16", 250, 4e-4), ("gauss", 96, 5e-4),
                                         ("gauss", 128, 4.5e-4)])
def test_lists_of_small_fp16_rows(kind, d, amax):
    need_gpu()
    cng = lib()
    X = synth.generate(kind, 6000, d, seed=71).astype(np.float32)
    X = (X * (amax / np.abs(X).max())).astype(np.float16)
    idx, st = cng.cng_build(tensor(X), alpha=1.2, R=16, L=128, margin=32, keep_lists=True, connect_L=-1)
    cand = host(cng.cng_lists(idx)[0])
    cng.cng_free(idx)
    assert st["screen_used"] == 1
    assert np.array_equal(cand, oracle.knn(X.astype(np.float32), 128)[0])
