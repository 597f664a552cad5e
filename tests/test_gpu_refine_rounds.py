"""Refinement by rounds of 256 candidates (many results, or a relaxed bound) at the
rounds' edges, with repeated and absent ids, for few and for many queries; and a relaxed
refinement that gives the same answer every time."""
import numpy as np
import pytest
import torch

import paper_2510_00566_gb300 as pano
import synth
from parity import check_topk

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _index(d, n=6_000, nq=160):
    s = synth.scaled(1, n=n, n_queries=nq, nlist=1, n_clusters=0, d=d, n_levels=1, decay=4.0 / d)
    w = synth.generate(s)
    t = pano.panorama_fit_transform(w.X.numpy())
    idx = pano.panorama_build_flat(t, w.X.to(DEV), level_widths=[d // 4] * 4)
    return idx, w.X.numpy(), w.Q.numpy()


@pytest.mark.parametrize("kprime,k", [(255, 100), (256, 40), (257, 41), (513, 200), (3_000, 1000)])
@pytest.mark.parametrize("nq", [1, 160])
def test_many_results(kprime, k, nq):
    idx, X, Q = _index(96, nq=nq)
    rng = np.random.default_rng(k)
    cand = np.stack([rng.permutation(len(X))[:kprime] for _ in range(nq)]).astype(np.int64)
    cand[:, 5::9] = cand[:, 4:-1:9][:, :cand[:, 5::9].shape[1]]  # repeats
    cand[:, 7::31] = -1  # absent
    ids, dist = idx.refine(torch.from_numpy(Q).to(DEV), torch.from_numpy(cand).to(DEV), k)
    want_i, want_d = np.full((nq, k), -1, np.int64), np.full((nq, k), np.inf)
    for i in range(nq):
        c = np.unique(cand[i][cand[i] >= 0])
        e = ((X[c].astype(np.float64) - Q[i]) ** 2).sum(1)
        o = np.lexsort((c, e))[:k]
        want_i[i, :len(o)], want_d[i, :len(o)] = c[o], e[o]
    check_topk(X, Q, ids.cpu().numpy(), dist.cpu().numpy(), want_i, want_d, k)


@pytest.mark.parametrize("d,nq", [(96, 9), (960, 9), (960, 480)])
@pytest.mark.parametrize("kprime", [100, 700])
def test_lists_of_repeats(d, nq, kprime):
    # every id three to six times: repeats are no others that rule a candidate out
    idx, X, Q = _index(d, n=2_000, nq=nq)
    rng = np.random.default_rng(kprime)
    cand = np.stack([rng.permutation(np.repeat(rng.permutation(len(X))[:kprime // 3], 6)[:kprime])
                     for _ in range(nq)]).astype(np.int64)
    for k in (1, 3, 10):
        ids, dist = idx.refine(torch.from_numpy(Q).to(DEV), torch.from_numpy(cand).to(DEV), k)
        want_i, want_d = np.full((nq, k), -1, np.int64), np.full((nq, k), np.inf)
        for i in range(nq):
            c = np.unique(cand[i])
            e = ((X[c].astype(np.float64) - Q[i]) ** 2).sum(1)
            o = np.lexsort((c, e))[:k]
            want_i[i, :len(o)], want_d[i, :len(o)] = c[o], e[o]
        check_topk(X, Q, ids.cpu().numpy(), dist.cpu().numpy(), want_i, want_d, k)


@pytest.mark.parametrize("widths", [[64] * 12, [4, 764], [100, 68, 632], [32] * 25, [256] * 4])
@pytest.mark.parametrize("kprime,k", [(1, 1), (5, 10), (37, 3), (300, 32), (2_500, 10)])
def test_groups_answer_as_rounds(widths, kprime, k):
    # many queries of long rows take groups of eight lanes, a few of them rounds
    d, nq = sum(widths), 480
    s = synth.scaled(1, n=3_000, n_queries=nq, nlist=1, n_clusters=0, d=d, n_levels=1, decay=4.0 / d)
    w = synth.generate(s)
    t = pano.panorama_transform_import(np.eye(d), np.zeros(d), np.ones(d))
    idx = pano.panorama_build_flat(t, w.X.to(DEV), level_widths=widths)
    rng = np.random.default_rng(kprime)
    cand = np.stack([rng.permutation(3_000)[:kprime] for _ in range(nq)]).astype(np.int64)
    cand[:, 11::17] = -1
    q, c = w.Q.to(DEV), torch.from_numpy(cand).to(DEV)
    ids, dist = idx.refine(q, c, k)
    for rows in (slice(0, 40), slice(440, 480)):
        a, b = idx.refine(q[rows].contiguous(), c[rows].contiguous(), k)
        assert torch.equal(a, ids[rows]) and torch.equal(b, dist[rows])
    X, Q = w.X.numpy(), w.Q.numpy()
    for i in (0, 77, 479):
        ci = np.unique(cand[i][cand[i] >= 0])
        e = ((X[ci].astype(np.float64) - Q[i]) ** 2).sum(1)
        o = np.lexsort((ci, e))[:k]
        assert np.array_equal(ids[i].cpu().numpy()[:len(o)], ci[o])
        assert np.allclose(dist[i].cpu().numpy()[:len(o)], e[o], rtol=1e-5, atol=0)
        assert np.all(ids[i].cpu().numpy()[len(o):] == -1)


@pytest.mark.parametrize("epsilon", [0.9, 0.6, 0.3])
@pytest.mark.parametrize("nq", [9, 160])
def test_relaxed_refinement_is_repeatable(epsilon, nq):
    idx, X, Q = _index(128, nq=nq)
    rng = np.random.default_rng(9)
    cand = torch.from_numpy(np.stack([rng.permutation(len(X))[:4_000] for _ in range(nq)])).to(DEV)
    q = torch.from_numpy(Q).to(DEV)
    first = idx.refine(q, cand, 10, epsilon=epsilon)
    for _ in range(20):
        again = idx.refine(q, cand, 10, epsilon=epsilon)
        assert torch.equal(first[0], again[0]) and torch.equal(first[1], again[1])
