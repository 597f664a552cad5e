"""The search workspace that is kept between calls: at most 1 GiB for all indexes of the
device together, and none once the last index is gone."""
import numpy as np
import pytest
import torch

import paper_2510_00566_gb300 as pano

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def test_several_indexes_keep_one_workspace():
    rng = np.random.default_rng(4)
    n, d, nlist, nq = 20_000, 8, 16_384, 8_192  # 537 MB of probe distances a search
    X = rng.standard_normal((n, d)).astype(np.float32)
    t = pano.panorama_transform_import(np.eye(d), np.zeros(d), np.ones(d))
    Q = torch.from_numpy(rng.standard_normal((nq, d)).astype(np.float32)).to(DEV)
    out = (torch.empty((nq, 1), dtype=torch.int64, device=DEV),
           torch.empty((nq, 1), dtype=torch.float32, device=DEV))

    def build():
        return pano.panorama_build_ivf(t, torch.from_numpy(X).to(DEV), nlist, level_widths=[8],
                                       centroids=X[:nlist].copy())

    def free():
        torch.cuda.synchronize()
        return torch.cuda.mem_get_info()[0]

    indexes = [build() for _ in range(4)]
    indexes[0].search(Q[:8].contiguous(), 1, 1)  # (code and tables are loaded at first use)
    before = free()
    for idx in indexes:
        idx.search(Q, 1, 1, out=out)
        assert before - free() <= (1 << 30) + (64 << 20)
    held = [idx.info().device_bytes for idx in indexes]
    for idx in indexes:
        idx.free()
    assert free() >= before + sum(held) // 2  # the indexes' own memory, and no workspace
