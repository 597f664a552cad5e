"""Top-k insertion at the k where it changes: up to 40 sorted slots are kept by
atomic chains, more stay unsorted and a new key replaces the largest (up to 128
slots in registers, more in rounds), mixed in one batch, with many work items
competing for each query's slots."""
import numpy as np
import pytest
import torch

import oracle
import paper_2510_00566_gb300 as pano
import synth
from parity import check_topk

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("precision", [pano.PANO_FP32, pano.PANO_BF16, pano.PANO_FP8])
def test_mixed_k_at_the_insertion_edges(precision):
    s = synth.scaled(1, n=9_001, n_queries=96, nlist=2, n_clusters=0)
    w = synth.generate(s)
    X, Q = w.X.numpy(), w.Q.numpy()
    C = synth.initial_centroids(w.X, 2, seed=31).numpy()
    t = pano.panorama_fit_transform(X, n_levels=2)
    idx = pano.panorama_build_ivf(t, w.X.to(DEV), nlist=2, level_widths=[64, 64],
                                  precision=precision, centroids=C)
    k = np.resize([1, 16, 33, 40, 41, 64, 127, 128, 129, 300, 1024, 0], len(Q)).astype(np.int32)
    ids, d = idx.search(torch.from_numpy(Q).to(DEV), 2, torch.from_numpy(k).to(DEV), k_max=1024)
    lists, _ = oracle.assign(X, C)
    ref = oracle.ivf_search(X, Q, C, 2, 1024, lists_of_vector=lists)
    check_topk(X, Q, ids.cpu().numpy(), d.cpu().numpy(), ref["ids"], ref["dists"], k)
