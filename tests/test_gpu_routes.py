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
