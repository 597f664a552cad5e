"""Refinement at the edges of its eight-lane groups: dimensions and levels that
are no multiples of 4 or 32, one level, lists shorter than a warp's four groups,
longer than the seeded prefix, and k above the candidates."""
import numpy as np
import pytest
import torch

import oracle
import paper_2510_00566_gb300 as pano
import synth
from parity import check_topk

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("widths", [[4], [33], [3, 5, 7, 85], [32, 32, 32, 4], [60] * 5])
@pytest.mark.parametrize("kprime,k", [(1, 1), (5, 10), (37, 3), (2_500, 40)])
def test_refine_groups(widths, kprime, k):
    d = sum(widths)
    s = synth.scaled(1, n=3_000, n_queries=9, nlist=1, n_clusters=0, d=d, n_levels=1, decay=4.0 / d)
    w = synth.generate(s)
    X, Q = w.X.numpy(), w.Q.numpy()
    idx = pano.panorama_build_flat(pano.panorama_fit_transform(X), w.X.to(DEV), level_widths=widths)
    rng = np.random.default_rng(5)
    cand = np.stack([rng.permutation(len(X))[:kprime] for _ in range(len(Q))]).astype(np.int64)
    ids, dist = idx.refine(torch.from_numpy(Q).to(DEV), torch.from_numpy(cand).to(DEV), k)
    want_i, want_d = np.full((len(Q), k), -1, np.int64), np.full((len(Q), k), np.inf)
    for i in range(len(Q)):
        e = ((X[cand[i]].astype(np.float64) - Q[i]) ** 2).sum(1)
        o = np.lexsort((cand[i], e))[:k]
        want_i[i, :len(o)], want_d[i, :len(o)] = cand[i][o], e[o]
    check_topk(X, Q, ids.cpu().numpy(), dist.cpu().numpy(), want_i, want_d, k)
