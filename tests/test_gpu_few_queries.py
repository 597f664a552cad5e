"""Small batches: the transform of up to eight queries by a warp per output row, the
seeds of fewer than 152 queries by sixteen warps, and segments that shrink with the
batch give the answers of the same queries in a large batch, bit for bit."""
import numpy as np
import pytest
import torch

import paper_2510_00566_gb300 as pano
import synth

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("prec,widths,nlist", [("fp32", [31, 31, 37], 1), ("fp32", [33], 20),
                                               ("fp32", [16] * 8, 20), ("bf16", [64, 64], 20),
                                               ("fp8", [32, 64], 20)])
def test_small_batches_answer_as_large_ones(prec, widths, nlist):
    d, nq = sum(widths), 330
    s = synth.scaled(1, n=9_001, n_queries=nq, nlist=1, n_clusters=0, d=d, n_levels=1, decay=4.0 / d)
    w = synth.generate(s)
    X, Q = w.X.numpy(), w.Q.to(DEV)
    P = {"fp32": pano.PANO_FP32, "bf16": pano.PANO_BF16, "fp8": pano.PANO_FP8}[prec]
    idx = pano.panorama_build_ivf(pano.panorama_fit_transform(X), w.X.to(DEV), nlist,
                                  level_widths=widths, precision=P, centroids=X[:nlist].copy())
    for k in (1, 10, 100):
        ids, dist = idx.search(Q, min(4, nlist), k)
        for m in (1, 7, 8, 9, 151, 152):
            i, v = idx.search(Q[:m].contiguous(), min(4, nlist), k)
            assert np.array_equal(torch.as_tensor(i).cpu().numpy(), torch.as_tensor(ids[:m]).cpu().numpy())
            assert np.array_equal(torch.as_tensor(v).cpu().numpy(), torch.as_tensor(dist[:m]).cpu().numpy())
