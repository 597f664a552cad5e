"""The tensor-core verify kernel at its edges: level widths of every panel form
(less than a panel, one, several), query groups around 16, 32 and 64, segments
of one to four chunks with a ragged end, rows longer than the staged split, a
schedule that tests every level and one that leaves levels out."""
import numpy as np
import pytest
import torch

import oracle
import paper_2510_00566_gb300 as pano
import synth
from parity import check_topk

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
CASES = [
    (pano.PANO_BF16, [16, 16, 32, 64, 128]),
    (pano.PANO_BF16, [128, 128]),
    (pano.PANO_BF16, [16]),
    (pano.PANO_BF16, [64] * 25),
    (pano.PANO_FP8, [32, 32, 64, 128, 256]),
    (pano.PANO_FP8, [128] * 13),
    (pano.PANO_FP8, [32]),
]


@pytest.mark.parametrize("precision,widths", CASES)
def test_panels_groups_and_segments(precision, widths):
    d = sum(widths)
    s = synth.scaled(1, n=1_500, n_queries=130, nlist=3, n_clusters=0, d=d, n_levels=1, decay=8.0 / d)
    w = synth.generate(s)
    X, Q = w.X.numpy(), w.Q.numpy()
    C = synth.initial_centroids(w.X, 3, seed=17).numpy()
    t = pano.panorama_fit_transform(X, identity=True)
    idx = pano.panorama_build_ivf(t, w.X.to(DEV), nlist=3, level_widths=widths,
                                  precision=precision, centroids=C)
    lists, _ = oracle.assign(X, C)
    ref = oracle.ivf_search(X, Q, C, 3, 10, lists_of_vector=lists)
    for nq in (1, 16, 17, 33, 64, 65, 130):
        for te in (0, 1):
            ids, dist = idx.search(torch.from_numpy(Q[:nq]).to(DEV), 3, 10, test_every=te,
                                   collect_stats=True)
            assert pano.last_stats().device_error == 0
            check_topk(X, Q[:nq], ids.cpu().numpy(), dist.cpu().numpy(), ref["ids"][:nq],
                       ref["dists"][:nq], 10)
