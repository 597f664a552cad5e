"""IVFPQ residuals whose energy leaves FP32's range at either end, whose tails are zero,
and ordinary ones: the pruned search equals the plain scan bit for bit."""
import numpy as np
import pytest
import torch

import paper_2510_00566_gb300 as pano

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("scale", [1.0, 1.5e18, 1e-25])
def test_ivfpq_residuals_beyond_the_range(scale):
    # (at 1.5e18 a residual's energy may leave FP32's range where the query's own does
    # not; at 1e-25 every square underflows)
    rng = np.random.default_rng(13)
    n, d = 4_000, 64
    X = (rng.standard_normal((n, d)) * scale).astype(np.float32)
    Q = (rng.standard_normal((12, d)) * scale).astype(np.float32)
    Q[7] *= 1e-6
    Q[9] = 0
    t = pano.panorama_transform_import(np.eye(d), np.zeros(d), np.ones(d))
    idx = pano.panorama_build_ivfpq(t, X, 8, 32, 8, centroids=X[:8].copy())
    q = torch.from_numpy(Q).to(DEV)
    for nprobe, k in ((8, 10), (3, 100)):
        a, b = idx.search_pq(q, nprobe, k), idx.search_pq(q, nprobe, k, mode=1)
        assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])
