"""Which kernels a call launches, where its results cannot tell: by the library's launch counter."""
import numpy as np
import pytest

import oracle
from paper_2510_05975_gb300 import synth

from gpu_util import lib, need_gpu, tensor

pytestmark = pytest.mark.gpu


def _launches(cng, call):
    call()  # first use: launch shapes are timed
    before = cng.lib().cngx_launches()
    call()
    return cng.lib().cngx_launches() - before


def test_beam_candidates_of_byte_rows_use_the_register_queue():
    """Candidate searches on a graph of at most 96 neighbours launch the 8-bit register-queue kernel
    and the general one (which finds nothing to do); wider graphs the general one alone."""
    need_gpu()
    cng = lib()
    X = synth.generate("sift", 2000, 64, seed=111)
    G0 = oracle.knn(X, 97)[0].astype(np.int32)
    counts = []
    for K in (96, 97):
        g0, pts = tensor(G0[:, :K]), tensor(X)

        def build():
            idx, _ = cng.cng_build(pts, alpha=1.2, R=16, L=40, connect_L=-1, candidates=cng.CNG_CAND_BEAM,
                                   beam_L=48, knn_graph=g0)
            cng.cng_free(idx)

        counts.append(_launches(cng, build))
    assert counts[0] == counts[1] + 1


def test_column_splits_stop_at_one_unit_per_sm():
    """k-NN of up to 76 row blocks of 256 splits the columns (one more launch, which merges the splits'
    lists); from 77 row blocks on a split would give an SM two units in turn, which is slower."""
    need_gpu()
    cng = lib()
    rng = np.random.default_rng(112)
    X, Q = tensor(rng.standard_normal((1_000_000, 16)).astype(np.float32)), rng.standard_normal((60_000, 16))
    counts = {}
    for m in (1, 1000, 10_000, 20_000, 39_000, 60_000):
        rows = tensor(Q[:m].astype(np.float32))
        counts[m] = _launches(cng, lambda: cng.cng_knn(X, 10, rows=rows))
    assert counts[1] == counts[1000] == counts[10_000] == counts[60_000] + 1
    assert counts[20_000] == counts[39_000] == counts[60_000]
