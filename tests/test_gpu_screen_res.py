"""The resident tensor-core screen (rows of up to 250 coordinates: operands in TMEM, the columns'
norms folded into the product, sampled column order) at the edges of its operand widths, column
tiles and sample parts: raw scores against the same arithmetic in FP64, lists against the oracle."""
import numpy as np
import pytest

import oracle
from paper_2510_05975_gb300 import synth

from gpu_util import host, lib, need_gpu, tensor
from test_gpu_tc import _scores_f16

pytestmark = pytest.mark.gpu


# operand widths 16, 32, 48 .. 256 (the coordinates and six norm pieces), tiles of 96, 80 and 64
# columns filled exactly, by one less and one more; 251 coordinates take the streamed kernel
@pytest.mark.parametrize("m,n,d", [(256, 96, 10), (1, 95, 11), (257, 97, 26), (300, 193, 122),
                                   (130, 160, 123), (40, 161, 186), (300, 129, 187), (513, 64, 250),
                                   (64, 200, 251)])
def test_scores_at_operand_edges(m, n, d):
    need_gpu()
    cng = lib()
    R = synth.generate("gauss", m, d, seed=41)
    C = synth.generate("gauss", n, d, seed=42)
    got = _scores_f16(cng, R, C, 1024.0)
    rh = (R * np.float32(1024)).astype(np.float16).astype(np.float64)
    ch = (C * np.float32(1024)).astype(np.float16).astype(np.float64)
    nb = (ch * ch).sum(1)[None, :]
    ref = nb - 2.0 * rh @ ch.T
    # d + 6 products and one norm, each addition within 2^-22 of the magnitudes summed
    bound = (d + 16) * 2.0 ** -22 * ((np.abs(rh) @ np.abs(ch).T) * 2 + nb)
    assert np.all(np.abs(got - ref) <= bound + 1e-6)


# self lists: a tile less one, exactly, more; n that activates one, two and three sample parts
@pytest.mark.parametrize("kind,n,d,k", [("gauss", 2, 8, 1), ("gauss", 95, 16, 20), ("sift", 96, 128, 95),
                                        ("gauss", 97, 200, 33), ("sift", 1700, 100, 100),
                                        ("sift", 7001, 123, 64), ("gauss", 26_003, 12, 10)])
def test_self_lists(kind, n, d, k):
    need_gpu()
    cng = lib()
    X = synth.generate(kind, n, d, seed=43)
    ids, ds, st = cng.cng_knn(tensor(X), k)
    ref, rd = oracle.knn(X, k)
    assert st["screen_used"] == 1 and st["cert_fail_rows"] == 0
    assert np.array_equal(host(ids), ref)
    assert np.allclose(host(ds), rd, rtol=2e-6)


# separate rows: fewer and more than a block, lists of 1 and 256 (L' = 33 and 288)
@pytest.mark.parametrize("kind,n,d,m,k", [("sift", 30_011, 128, 1, 256), ("gauss", 30_011, 24, 700, 100),
                                          ("deep", 4099, 96, 257, 1), ("bigann16", 9001, 250, 300, 200)])
def test_row_lists(kind, n, d, m, k):
    need_gpu()
    cng = lib()
    X = synth.generate(kind, n, d, seed=44)
    Q = synth.generate(kind, m, d, seed=45, centre_seed=44)
    ids, ds, st = cng.cng_knn(tensor(X), k, rows=tensor(Q))
    ref, rd = oracle.knn(X, k, rows=Q)
    assert st["screen_used"] == 1 and st["cert_fail_rows"] == 0
    assert np.array_equal(host(ids), ref)
    assert np.allclose(host(ds), rd, rtol=2e-6)


def test_clustered_ids_are_sampled_fairly():
    """Points sorted by cluster, 64 tight clusters of 128: a row's 100 nearest are consecutive ids.
    The sample of the column order is chosen by a hash of the id, so no row's threshold is set too
    low by it (every list certifies)."""
    need_gpu()
    cng = lib()
    rng = np.random.default_rng(46)
    X = (np.repeat(rng.normal(size=(64, 20)) * 10, 128, axis=0) + 0.1 * rng.normal(size=(8192, 20)))
    X = X.astype(np.float32)
    ids, _, st = cng.cng_knn(tensor(X), 100)
    assert st["cert_fail_rows"] == 0
    assert np.array_equal(host(ids), oracle.knn(X, 100)[0])


def test_norms_beyond_the_pieces():
    """FP16 points whose squared norms exceed what the norm pieces hold take the streamed kernel;
    the candidate lists are the oracle's."""
    need_gpu()
    cng = lib()
    X = (synth.generate("gauss", 3000, 192, seed=47) * 9000).astype(np.float16)
    assert (X.astype(np.float64) ** 2).sum(1).max() > 2 * 4 * 65504 * 32768
    idx, st = cng.cng_build(tensor(X), alpha=1.2, R=16, L=48, keep_lists=True)
    cand = host(cng.cng_lists(idx)[0])
    cng.cng_free(idx)
    assert st["screen_used"] == 1
    assert np.array_equal(cand, oracle.knn(X.astype(np.float32), 48)[0])
