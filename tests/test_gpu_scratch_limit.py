"""The fixed scratch of the allocation-free search: a batch is not refused where a larger
one on the same index is accepted.  (Small FP32 batches split long lists into shorter
segments, whose work items need more of the scratch.)"""
import numpy as np
import pytest
import torch

import paper_2510_00566_gb300 as pano

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def test_a_smaller_batch_is_accepted_where_a_larger_one_is():
    rng = np.random.default_rng(8)
    n, d, nlist = 1_000_000, 8, 27_000
    # one long list at the origin; the other centroids are far from every vector
    C = rng.standard_normal((nlist, d)).astype(np.float32)
    C *= 100 / np.linalg.norm(C, axis=1, keepdims=True)
    C[0] = 0
    X = torch.from_numpy(rng.standard_normal((n, d)).astype(np.float32)).to(DEV)
    t = pano.panorama_transform_import(np.eye(d), np.zeros(d), np.ones(d))
    idx = pano.panorama_build_ivf(t, X, nlist, level_widths=[8], centroids=C)
    assert np.all(idx.assignment() == 0)
    Q = torch.from_numpy(rng.standard_normal((640, d)).astype(np.float32)).to(DEV)
    stream = torch.cuda.current_stream().cuda_stream

    def accepted(nq, k_max):
        ids = torch.empty((nq, k_max), dtype=torch.int64, device=DEV)
        dist = torch.empty((nq, k_max), dtype=torch.float32, device=DEV)
        rc = pano.lib().panorama_search_noalloc(idx.handle, Q.data_ptr(), nq, None, 1, None, 1,
                                                k_max, ids.data_ptr(), dist.data_ptr(), stream)
        if rc == 0:
            want, _ = idx.search(Q[:nq].contiguous(), 1, 1)
            assert torch.equal(ids[:, 0], want[:, 0])
        return rc == 0

    # (an unused slot of a query's k_max takes 8 bytes: a fine step in size)
    for large in (560, 572, 590, 640):
        lo, hi = 0, 1024  # the largest k_max that the batch of `large` queries may have
        while lo < hi:
            mid = (lo + hi + 1) // 2
            lo, hi = (mid, hi) if accepted(large, mid) else (lo, mid - 1)
        if not lo:
            continue
        for nq in (large - 1, large - 2, large - 5, large - 20, 300, 30, 1):
            assert accepted(nq, lo), (nq, large, lo)
