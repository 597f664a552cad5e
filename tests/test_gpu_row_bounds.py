"""Tail norms, energies and transform-error bounds of packed rows: those of FP64 sums,
rounded once, bit for bit, though the sums are compensated FP32; also for rows whose
squares leave FP32's range at either end, rows with zero levels and zero rows.  And the
searches beside such rows."""
import struct

import numpy as np
import pytest
import torch

import paper_2510_00566_gb300 as pano

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
PREC = {"fp32": pano.PANO_FP32, "bf16": pano.PANO_BF16, "fp8": pano.PANO_FP8}


def _arrays(path, prec):
    """Slots' ids, tails, |x^|^2, e_x and scales, and c_trans, of a saved index."""
    b, o = open(path, "rb").read(), 12

    def pod(f):
        nonlocal o
        v = struct.unpack_from("<" + f, b, o)
        o += struct.calcsize("<" + f)
        return v

    n, d, nlist, L, _, chunk, _, n_chunks, _, c_trans, _ = pod("q6iq2df")

    def skip(*sizes):
        nonlocal o
        for size in sizes:
            count = pod("Q")[0]
            o += size * count

    skip(4, 4)  # level widths and offsets
    pod("2id")
    skip(8, 8, 8, 4, 4, 4, 4, 8, 4)  # the transform, centroids and lists
    dev = []
    for _ in range(7 if prec == "fp8" else 6):
        m = pod("Q")[0]
        dev.append(b[o:o + m])
        o += m
    f32 = [np.frombuffer(x, np.float32) for x in dev]
    ids = np.frombuffer(dev[4], np.int32)
    tails = f32[1].reshape(n_chunks, L + 1, chunk).transpose(0, 2, 1).reshape(-1, L + 1)
    return ids, tails, f32[2], f32[3], f32[6] if prec == "fp8" else None, c_trans


def _up(v):
    with np.errstate(over="ignore"):
        t = v.astype(np.float32)
    return np.where(t.astype(np.float64) < v, np.nextafter(t, np.float32(np.inf)), t)


def _rows(n, d):
    rng = np.random.default_rng(11)
    X = (rng.standard_normal((n, d)) * np.exp(-0.02 * np.arange(d))).astype(np.float32)
    X[::7] *= 37.0
    X[1::50, d // 2:] = 0  # zero levels
    X[2::50] = 0
    X[3::50] *= 1e-21  # squares below FP32's normal range
    X[4::50, ::3] *= 1e-20
    X[5::50] *= 1e-9
    X[6::50, 5] = 3e19  # squares beyond FP32's range
    X[7::50] *= 1e18
    return X


@pytest.mark.parametrize("prec,widths", [("fp32", [3, 29, 100, 1, 64]), ("fp32", [16] * 40),
                                         ("bf16", [64] * 6), ("bf16", [16] * 20 + [128]),
                                         ("fp8", [128, 32, 64]), ("fp8", [32] * 16)])
def test_bounds_are_those_of_fp64_sums(prec, widths, tmp_path):
    d, n = sum(widths), 4_000
    X = _rows(n, d)
    t = pano.panorama_transform_import(np.eye(d), np.zeros(d), np.ones(d))
    idx = pano.panorama_build_ivf(t, torch.from_numpy(X).to(DEV), 1, level_widths=widths,
                                  precision=PREC[prec], centroids=np.zeros((1, d), np.float32))
    path = str(tmp_path / "index")
    pano.panorama_save(idx, path)
    ids, tails, xn2, ex, scale, c_trans = _arrays(path, prec)
    used = ids >= 0
    assert used.sum() == n and not tails[~used].any() and not xn2[~used].any()
    x = X[ids[used]]
    if prec == "fp32":
        stored = x.astype(np.float64)
    elif prec == "bf16":
        stored = torch.from_numpy(x).to(torch.bfloat16).double().numpy()
    else:
        s = scale[used][:, None].astype(np.float64)
        stored = torch.from_numpy((x / s).astype(np.float32)).to(torch.float8_e4m3fn).double().numpy() * s
    ends = np.cumsum(widths)
    energy = np.stack([(stored[:, e - w:e] ** 2).sum(1) for e, w in zip(ends, widths)], 1)
    suffix = np.cumsum(energy[:, ::-1], 1)[:, ::-1]
    with np.errstate(over="ignore"):
        assert np.array_equal(xn2[used], suffix[:, 0].astype(np.float32))
    assert np.array_equal(tails[used][:, :-1], _up(np.sqrt(suffix * (1 + 1e-12))))
    x = x.astype(np.float64)
    err = np.sqrt(((stored - x) ** 2).sum(1)) + c_trans * np.sqrt((x ** 2).sum(1))
    assert np.array_equal(ex[used], _up(err * (1 + 1e-9)))


@pytest.mark.parametrize("prec", ["fp32", "bf16", "fp8"])
@pytest.mark.parametrize("value", [1e19, 1e20])
def test_search_beside_rows_beyond_the_range(prec, value):
    rng = np.random.default_rng(12)
    n, d, odd = 3_000, 128, 6
    X = rng.standard_normal((n, d)).astype(np.float32)
    X[100:100 + odd] = value
    Q = torch.from_numpy(rng.standard_normal((40, d)).astype(np.float32)).to(DEV)
    t = pano.panorama_transform_import(np.eye(d), np.zeros(d), np.ones(d))
    idx = pano.panorama_build_ivf(t, torch.from_numpy(X).to(DEV), 4, level_widths=[64, 64],
                                  precision=PREC[prec], centroids=X[:4].copy())
    k = 40
    ids = [idx.search(Q, 4, k, mode=mode)[0].cpu().numpy() for mode in (0, 1)]
    rest = np.setdiff1d(np.arange(n), np.arange(100, 100 + odd))
    e = ((X[rest].astype(np.float64)[None] - Q.cpu().numpy()[:, None]) ** 2).sum(2)
    for i in range(len(Q)):
        want = rest[e[i].argsort()[:k - odd]]
        for got in ids:
            g = got[i][~np.isin(got[i], np.arange(100, 100 + odd))][:k - odd]
            assert np.array_equal(g, want)
