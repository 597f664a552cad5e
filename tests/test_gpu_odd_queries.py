"""Queries whose norm leaves FP32's range, infinities and NaN among ordinary ones: every
probed list is one of the index's (or none), the ordinary queries get the answer that
they get alone, and the odd ones valid ids.  A larger batch goes first, so that the
workspace holds its data."""
import numpy as np
import pytest
import torch

import paper_2510_00566_gb300 as pano

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
NLIST, N, NQ = 37, 3_000, 70
ODD = {3: 3e19, 4: np.inf, 20: np.nan, 41: -np.inf, 69: 1e20}


def _data(d):
    rng = np.random.default_rng(d)
    X = rng.standard_normal((N, d)).astype(np.float32)
    Q = rng.standard_normal((NQ, d)).astype(np.float32)
    bad = Q.copy()
    for i, v in ODD.items():
        bad[i] = v
    bad[41] = Q[41]
    bad[41, 5] = -np.inf
    bad[69] = Q[69]
    bad[69, 7] = 1e20
    big = torch.from_numpy(rng.standard_normal((4_000, d)).astype(np.float32)).to(DEV)
    t = pano.panorama_transform_import(np.eye(d), np.zeros(d), np.ones(d))
    return X, torch.from_numpy(Q).to(DEV), torch.from_numpy(bad).to(DEV), big, t


def _check(good, bad, n):
    keep = np.setdiff1d(np.arange(NQ), list(ODD))
    for a, b in zip(good, bad):
        assert torch.equal(a[keep], b[keep])
    ids = bad[0].cpu().numpy()
    assert ids.min() >= -1 and ids.max() < n
    for i in ODD:
        got = ids[i][ids[i] >= 0]
        assert len(set(got.tolist())) == len(got)


@pytest.mark.parametrize("prec,d", [(pano.PANO_FP32, 64), (pano.PANO_FP32, 66),
                                    (pano.PANO_BF16, 64), (pano.PANO_FP8, 64)])
@pytest.mark.parametrize("nprobe", [5, NLIST])
def test_search_and_probe(prec, d, nprobe):
    X, Q, bad, big, t = _data(d)
    idx = pano.panorama_build_ivf(t, torch.from_numpy(X).to(DEV), NLIST, level_widths=[d // 2] * 2,
                                  precision=prec, centroids=X[:NLIST].copy())
    idx.search(big, nprobe, 10)
    lists = pano.panorama_probe(idx, bad, nprobe).cpu().numpy()
    assert lists.min() >= -1 and lists.max() < NLIST
    for row in lists:
        assert len(set(row[row >= 0].tolist())) == np.count_nonzero(row >= 0)
    for k in (10, 100):
        _check(idx.search(Q, nprobe, k), idx.search(bad, nprobe, k), N)


@pytest.mark.parametrize("d", [64, 66])
def test_a_centroid_beyond_the_range_comes_last(d):
    X, Q, _, big, t = _data(d)
    C = X[:NLIST].copy()
    C[5] = 1e20
    idx = pano.panorama_build_ivf(t, torch.from_numpy(X).to(DEV), NLIST, level_widths=[d // 2] * 2,
                                  centroids=C)
    idx.search(big, NLIST, 10)
    lists = pano.panorama_probe(idx, Q, NLIST).cpu().numpy()
    e = ((Q.cpu().numpy().astype(np.float64)[:, None] - C[None]) ** 2).sum(2)
    assert np.array_equal(lists, e.argsort(1))
    ids, _ = idx.search(Q, NLIST, 10)
    x = ((Q.cpu().numpy().astype(np.float64)[:, None] - X[None]) ** 2).sum(2)
    assert np.array_equal(ids.cpu().numpy(), x.argsort(1)[:, :10])


@pytest.mark.parametrize("nprobe", [5, NLIST])
def test_search_pq(nprobe):
    X, Q, bad, big, t = _data(64)
    idx = pano.panorama_build_ivfpq(t, X, NLIST, 32, 8, centroids=X[:NLIST].copy())
    idx.search_pq(big, nprobe, 10)
    for k in (10, 100):
        for mode in (0, 1):
            _check(idx.search_pq(Q, nprobe, k, mode=mode), idx.search_pq(bad, nprobe, k, mode=mode), N)
