"""Queries that are database rows: a row is its own nearest neighbour at distance 0, the
first row included, whose key (distance 0, id 0) is the smallest there is.  Every k
around the insertion's edges (sorted slots up to 40, 128 slots in registers), by a
search, a plan and the server, alone or among exact copies of the first row."""
import numpy as np
import pytest
import torch

import oracle
import paper_2510_00566_gb300 as pano
import synth
from parity import check_topk

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
KS = [40, 41, 64, 100, 127, 128, 129]
PREC = {"fp32": pano.PANO_FP32, "bf16": pano.PANO_BF16, "fp8": pano.PANO_FP8}


def _index(prec, copies, n=9_001):
    """The index, its rows, queries (rows 0 .. 31 and eight more of row 0) and coarse
    lists; `copies` rows from the middle on are the first row again."""
    w = synth.generate(synth.scaled(1, n=n, n_queries=1, nlist=2, n_clusters=0))
    X = w.X.numpy().copy()
    X[n // 2:n // 2 + copies] = X[0]
    C = synth.initial_centroids(torch.from_numpy(X), 2, seed=31).numpy()
    t = pano.panorama_fit_transform(X, n_levels=2)
    idx = pano.panorama_build_ivf(t, torch.from_numpy(X).to(DEV), nlist=2, level_widths=[64, 64],
                                  precision=PREC[prec], centroids=C)
    return idx, X, np.concatenate([X[:32], np.repeat(X[:1], 8, 0)]), C


def _check(X, Q, ref, k, ids, d):
    """Against the oracle; where its distance is 0 the ids have to be the same, too."""
    ids, d = np.asarray(ids), np.asarray(d)
    check_topk(X, Q, ids, d, ref["ids"][:, :ids.shape[1]], ref["dists"][:, :ids.shape[1]], k)
    for i, ki in enumerate(np.broadcast_to(k, (len(Q),))):
        zeros = np.count_nonzero(ref["dists"][i, :ki] == 0)
        assert zeros >= 1
        assert np.array_equal(ids[i, :zeros], ref["ids"][i, :zeros]), (i, ki)
        assert np.all(d[i, :zeros] == 0)


@pytest.mark.parametrize("prec", ["fp32", "bf16", "fp8"])
@pytest.mark.parametrize("copies", [0, 150])
def test_a_row_finds_itself(prec, copies):
    idx, X, Q, C = _index(prec, copies)
    ref = oracle.ivf_search(X, Q, C, 2, max(KS), lists_of_vector=idx.assignment())
    Qd = torch.from_numpy(Q).to(DEV)
    for k in KS:
        for m in (len(Q), 1):
            ids, d = idx.search(Qd[:m], 2, k)
            _check(X, Q[:m], {v: ref[v][:m] for v in ("ids", "dists")}, k, ids.cpu(), d.cpu())
        ids, d = pano.Plan(idx, Qd, 2, k).launch()
        torch.cuda.synchronize()
        _check(X, Q, ref, k, ids.cpu(), d.cpu())
    k = np.resize(KS, len(Q)).astype(np.int32)
    server = pano.Server(idx, max_batch=16, k_max=max(KS))
    ids, d, _ = server.run_trace(Q, np.zeros(len(Q)), np.full(len(Q), 2, np.int32), k)
    server.close()
    _check(X, Q, ref, k, ids, d)


@pytest.mark.parametrize("prec", ["fp32", "bf16", "fp8"])
@pytest.mark.parametrize("k", [64, 100, 300])
def test_relaxed_bounds_above_the_sorted_slots(prec, k):
    # epsilon 0.98 relaxes a row's bound against itself to 0.04 of its tail energy at
    # most, far below the distance of its k-th neighbour: it is always found.  The seeds
    # are in the slots before verification enters them again: no id may come twice.
    idx, X, Q, C = _index(prec, 0)
    ref = oracle.ivf_search(X, Q, C, 2, k, lists_of_vector=idx.assignment())
    tail = ((X[:32].astype(np.float64) - X.mean(0)) ** 2).sum(1)
    assert np.all(0.04 * tail < 0.5 * ref["dists"][:32, -1])
    ids, d = idx.search(torch.from_numpy(Q).to(DEV), 2, k, epsilon=0.98)
    ids, d = ids.cpu().numpy(), d.cpu().numpy()
    assert np.array_equal(ids[:, 0], ref["ids"][:, 0]) and np.all(d[:, 0] == 0)
    for i in range(len(Q)):
        got = ids[i][ids[i] >= 0]
        assert len(set(got.tolist())) == len(got)
        e = ((X[got].astype(np.float64) - Q[i]) ** 2).sum(1)
        assert np.allclose(d[i, :len(got)], e, rtol=1e-5, atol=0)
        assert np.all(np.diff(d[i, :len(got)]) >= 0)
        assert len(np.intersect1d(got, ref["ids"][i])) >= 0.9 * k
