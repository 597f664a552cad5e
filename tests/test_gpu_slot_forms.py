"""More than 40 results on both sides of the rule that chooses between sorted slots (few
queries) and unsorted ones: the same answer, bit for bit, as from the largest batch,
which is the oracle's, with database rows (id 0 at distance 0 among them) as queries."""
import numpy as np
import pytest
import torch

import oracle
import paper_2510_00566_gb300 as pano
import synth
from parity import check_topk

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("prec", [pano.PANO_FP32, pano.PANO_BF16, pano.PANO_FP8])
@pytest.mark.parametrize("k", [41, 100, 128, 129, 300, -1])
def test_slot_forms_agree(prec, k):
    w = synth.generate(synth.scaled(1, n=9_001, n_queries=40, nlist=2, n_clusters=0))
    X = w.X.numpy()
    Q = np.concatenate([X[:260], w.Q.numpy()])
    C = synth.initial_centroids(w.X, 2, seed=31).numpy()
    idx = pano.panorama_build_ivf(pano.panorama_fit_transform(X, n_levels=2), w.X.to(DEV), 2,
                                  level_widths=[64, 64], precision=prec, centroids=C)
    q = torch.from_numpy(Q).to(DEV)
    ks = np.full(len(Q), k, np.int32) if k > 0 else np.resize([41, 1, 129, 40, 100, 0, 300], len(Q)).astype(np.int32)
    kd, k_max = torch.from_numpy(ks).to(DEV), int(ks.max())
    ids, dist = idx.search(q, 2, kd, k_max=k_max)
    ref = oracle.ivf_search(X, Q, C, 2, k_max, lists_of_vector=idx.assignment())
    check_topk(X, Q, ids.cpu().numpy(), dist.cpu().numpy(), ref["ids"], ref["dists"], ks)
    rows = np.arange(260)[ks[:260] > 0]
    assert np.array_equal(ids.cpu().numpy()[rows, 0], rows) and not dist.cpu().numpy()[rows, 0].any()
    for m in (1, 15, 16, 31, 32, 127, 128, 255, 256):
        a, b = idx.search(q[:m], 2, kd[:m], k_max=k_max)
        assert torch.equal(a, ids[:m]) and torch.equal(b, dist[:m])


@pytest.mark.parametrize("prec", [pano.PANO_FP32, pano.PANO_BF16, pano.PANO_FP8])
@pytest.mark.parametrize("k", [100, 300])
def test_relaxed_bound_with_unsorted_slots(prec, k):
    # The seeds enter sorted, verification enters them again into unsorted slots: no id
    # may come twice.  A row's relaxed bound against itself is at most 0.04 of its tail
    # energy (epsilon 0.98), far below its k-th neighbour's distance: it is found.
    w = synth.generate(synth.scaled(1, n=9_001, n_queries=1, nlist=2, n_clusters=0))
    X = w.X.numpy()
    Q = X[:300]
    C = synth.initial_centroids(w.X, 2, seed=31).numpy()
    idx = pano.panorama_build_ivf(pano.panorama_fit_transform(X, n_levels=2), w.X.to(DEV), 2,
                                  level_widths=[64, 64], precision=prec, centroids=C)
    ids, dist = idx.search(torch.from_numpy(Q).to(DEV), 2, k, epsilon=0.98)
    ids, dist = ids.cpu().numpy(), dist.cpu().numpy()
    assert np.array_equal(ids[:, 0], np.arange(300)) and not dist[:, 0].any()
    for i in range(300):
        got = ids[i][ids[i] >= 0]
        assert len(set(got.tolist())) == len(got) >= 0.9 * k
        e = ((X[got].astype(np.float64) - Q[i]) ** 2).sum(1)
        assert np.allclose(dist[i, :len(got)], e, rtol=1e-5, atol=0)
        assert np.all(np.diff(dist[i, :len(got)]) >= 0)
