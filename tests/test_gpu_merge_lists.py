"""Phase 3 on float rows with merged sets on both sides of each route's limit: kept rows (up to R),
the Gram tile (FP16, up to 128), the all-pairs kernel (up to 256) and the whole-CTA merge above, with
the near-tied orders of copied points; graphs against the oracle."""
import numpy as np
import pytest

import oracle
from paper_2510_05975_gb300 import synth

from gpu_util import host, lib, need_gpu, tensor

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,dtype", [(72, "float32"), (200, "float32"), (64, "float16"), (128, "float16"),
                                     (90, "float16")])
def test_merged_sets_of_every_size(d, dtype):
    need_gpu()
    cng = lib()
    rng = np.random.default_rng(61)
    X = synth.generate("gauss", 4500, d, seed=61)
    # hubs: points near the centre, in the candidate lists of most others, at graded radii
    X[:40] *= np.linspace(0.3, 1.0, 40, dtype=np.float32)[:, None]
    X[4400:] = X[100:200]  # copies: tied orders
    X = X.astype(dtype)[rng.permutation(4500)]
    R, L = 12, 64
    G = oracle.build_graph(X.astype(np.float32), 1.1, 0.0, R, L, connect_L=0)
    merged = np.bincount(G.fwd[G.fwd >= 0], minlength=4500) + G.fdeg  # |V'| before duplicates leave
    for lo, hi in ((1, R), (R, 128), (128, 256), (256, 4500)):
        assert ((merged > lo) & (merged <= hi)).any()
    idx, st = cng.cng_build(tensor(X), alpha=1.1, R=R, L=L, connect_L=-1)
    adj, deg, _, entry = cng.cng_graph(idx)
    assert st["merge_max_list"] == merged.max() and entry == G.entry
    assert np.array_equal(host(deg), G.deg) and np.array_equal(host(adj)[:, :R], G.adj)
    cng.cng_free(idx)
