"""Rows whose squares leave FP32's range (elements above 1.8e19), infinities and NaN
among ordinary ones: such a row goes to the first list, as the expansion form says the
same of every centroid, and the others to their nearest one."""
import numpy as np
import pytest
import torch

import paper_2510_00566_gb300 as pano

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("value", [1e20, 3e38, np.inf, -np.inf, np.nan])
def test_assignment_of_rows_beyond_the_range(value):
    rng = np.random.default_rng(3)
    n, d, nlist = 1_500, 64, 37
    C = rng.standard_normal((nlist, d)).astype(np.float32)
    X = (C[rng.integers(0, nlist, n)] + 0.3 * rng.standard_normal((n, d))).astype(np.float32)
    odd = rng.permutation(n)[:40]
    X[odd] = 0.5
    X[odd[:20]] = value  # whole rows
    X[odd[20:], 5] = value  # one element
    t = pano.panorama_transform_import(np.eye(d), np.zeros(d), np.ones(d))
    got = pano.panorama_build_ivf(t, torch.from_numpy(X).to(DEV), nlist, level_widths=[32, 32],
                                  centroids=C).assignment()
    assert np.all(got[odd] == 0)
    rest = np.setdiff1d(np.arange(n), odd)
    e = ((X[rest, None].astype(np.float64) - C[None]) ** 2).sum(2)
    assert np.array_equal(got[rest], e.argmin(1))
