"""Assignment by the tensor-core products at tile edges (128 rows, 256 centroids,
panels of 64 coordinates), with duplicate centroids (ties to the lower id, more
of them than a half keeps) and rows that lie on a centroid."""
import numpy as np
import pytest
import torch

import paper_2510_00566_gb300 as pano

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("n,d,nlist", [(129, 8, 3), (1_000, 64, 256), (1_001, 72, 257),
                                       (700, 200, 33), (900, 136, 520)])
@pytest.mark.parametrize("copies", [1, 7])
def test_assignment_is_the_nearest_centroid(n, d, nlist, copies):
    rng = np.random.default_rng(n + d)
    C = rng.standard_normal((nlist, d)).astype(np.float32)
    C[rng.permutation(nlist)[:copies]] = C[0]  # equal centroids
    X = rng.standard_normal((n, d)).astype(np.float32)
    X[:nlist // 2] = C[:nlist // 2][:n]
    t = pano.panorama_fit_transform(X, identity=True)
    idx = pano.panorama_build_ivf(t, torch.from_numpy(X).to(DEV), nlist, level_widths=[d],
                                  centroids=C)
    e = ((X[:, None].astype(np.float64) - C[None]) ** 2).sum(2)
    best = e.argmin(1)  # (the lowest id of equals)
    got = idx.assignment()
    rows = np.arange(n)
    near = np.abs(e[rows, got] - e[rows, best]) <= 1e-6 * np.maximum(e[rows, best], 1e-30)
    assert np.all((got == best) | near)
    same = np.all(C[got] == C[best], axis=1)  # among equal centroids the lowest
    assert np.all(got[same] == best[same])
