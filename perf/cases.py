"""The work a user of the library has it do, as cases that can be timed: searches of
IVF indexes in each storage format, from one query to the largest batches, plans
replayed as CUDA graphs, IVFPQ searches, the refinement of candidate lists, index
builds and the request server.

A case is a dict of plain values; ``kind`` names the entry point.  The data follow the
recipe of ``synth`` (x = c + O diag(sqrt(lambda)) z, lambda_i = exp(-decay i)), drawn on
the GPU from the seed alone; the transform is the one a fit of that distribution gives
(the rows of O^T), imported, and the coarse centroids come from a few Lloyd iterations
of plain torch or, for mixtures, are the cluster centres.  All outputs are exact results,
so two correct implementations return the same ids and the same distances up to FP32.
"""
import math

import numpy as np
import torch

import paper_2510_00566_gb300 as pano

DEV = "cuda:0"
PREC = {"fp32": pano.PANO_FP32, "bf16": pano.PANO_BF16, "fp8": pano.PANO_FP8}


def _case(name, kind, prec, n, d, widths, nlist, nprobe, nq, k, clusters, decay,
          zipf=0.0, kprime=0, m=0):
    """nprobe < 0: per-query values uniform in [1, -nprobe]; k < 0: per-query values
    from {1, 10, 100}; widths: "64x12" is twelve levels of 64, joined by "+";
    clusters 0: one Gaussian; zipf > 0: cluster sizes proportional to rank^-zipf."""
    c = dict(kind=kind, prec=prec, n=n, d=d, widths=widths, nlist=nlist, nprobe=nprobe,
             nq=nq, k=k, clusters=clusters, decay=decay, zipf=zipf, kprime=kprime, m=m)
    return dict(c, name=name) if name else c


def listed():
    return [
        # The paper's plain method at SIFT's dimension: a small flat collection (one
        # list, every vector a candidate) searched for a hundred queries, all in L2.
        _case("flat-fp32-20k-d128", "search", "fp32", 20_000, 128, "16x8", 1, 1, 100, 10, 0, 0.05),
        # An interactive lookup: one query against a large BF16 index.
        _case("one-query-bf16-d128", "search", "bf16", 2_000_000, 128, "64x2", 2048, 32, 1, 10, 0, 0.05),
        # One batch of a serving process: about a thousand queries, each with its own
        # nprobe, a few queries per list.
        _case("serving-bf16-4m-d128", "search", "bf16", 4_000_003, 128, "64x2", 4096, -64, 1024, 10, 0, 0.05),
        # Bulk search of clustered GIST-like vectors stored in FP32 (no quantisation).
        _case("bulk-fp32-1m-d960", "search", "fp32", 1_000_000, 960, "60x16", 1024, 32, 10_000, 10, 1024, 0.01),
        # The same collection kept in BF16 level slices.
        _case("bulk-bf16-1m-d960", "search", "bf16", 1_000_000, 960, "64x15", 1024, 32, 10_000, 10, 1024, 0.01),
        # Bulk search of text-embedding-like vectors (one Gaussian, slow decay: the
        # bound prunes little), BF16: the framework's headline shape at fewer vectors.
        _case("bulk-bf16-4m-d768", "search", "bf16", 4_000_000, 768, "64x12", 2048, 64, 10_000, 10, 0, 0.008),
        # The capacity option: the same kind of vectors in FP8, ragged counts, k = 100.
        _case("bulk-fp8-1m-d768", "search", "fp8", 999_983, 768, "128x6", 1000, 48, 3_001, 100, 0, 0.008),
        # Offline batching: Zipf-sized lists, per-query nprobe and k, the whole search
        # replayed as one CUDA graph.
        _case("plan-zipf-bf16-d384", "plan", "bf16", 1_500_000, 384, "64x6", 1024, -128, 16_384, -1, 1024, 0.02, zipf=1.1),
        # Compressed storage: IVFPQ with pruning over shaped levels.
        _case("pq-d960", "pq", "pq", 250_007, 960, "60x16", 256, 24, 4_096, 10, 256, 0.01, m=480),
        # The second stage of a two-stage search: each query's candidate ids from a
        # coarse first stage, refined exactly on a flat index.
        _case("refine-d960", "refine", "fp32", 200_000, 960, "60x16", 1, 1, 4_096, 10, 128, 0.01, kprime=1000),
        # Building an index over new vectors with a trained coarse quantiser, and the
        # first queries on it.
        _case("build-bf16-d384", "build", "bf16", 500_009, 384, "64x6", 1024, 16, 64, 10, 0, 0.02),
        # The request server under a burst: host queries in, host results out.
        _case("server-bf16-d128", "server", "bf16", 1_000_000, 128, "64x2", 1024, -64, 4_096, 10, 0, 0.05),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["search"] * 6 + ["plan", "pq", "refine", "build"])
    if kind == "pq":
        d, levels = rng.choice([(128, 8), (384, 12), (960, 16)])
        return _case(None, "pq", "pq", _log(rng, 20_000, 250_000), d, "%dx%d" % (d // levels, levels),
                     _log(rng, 32, 256), rng.randint(1, 24), _log(rng, 1, 4_096), rng.choice([1, 10, 100]),
                     rng.choice([0, 64]), rng.choice([0.01, 0.05]), m=rng.choice([d // 2, d // 4]))
    if kind == "refine":
        d, widths = rng.choice([(128, "16x8"), (100, "20x5"), (384, "32x12"), (960, "60x16"), (129, "3x43")])
        return _case(None, "refine", "fp32", _log(rng, 10_000, 200_000), d, widths, 1, 1, _log(rng, 1, 4_096),
                     rng.choice([1, 10, 100]), rng.choice([0, 64]), rng.choice([0.01, 0.05]),
                     kprime=_log(rng, 100, 1_500))
    prec = rng.choice(["fp32", "bf16", "bf16", "fp8"]) if kind != "build" else rng.choice(["fp32", "bf16", "fp8"])
    if prec == "fp32":
        d, widths = rng.choice([(128, "16x8"), (100, "25x4"), (200, "8x1+24x8"), (384, "32x12"), (960, "60x16"),
                                (127, "31x3+34x1")])
    elif prec == "bf16":
        d, widths = rng.choice([(128, "64x2"), (128, "16x8"), (192, "32x2+64x2"), (384, "64x6"), (768, "64x12"),
                                (768, "128x6"), (960, "64x15")])
    else:
        d, widths = rng.choice([(128, "64x2"), (384, "128x3"), (768, "64x12"), (768, "128x6")])
    n = _log(rng, 20_000, 600_000 if kind == "build" or d > 384 else 1_500_000)
    nlist = min(_log(rng, 16, 2048), n // 128)
    nprobe = min(_log(rng, 1, 64), nlist)
    nq = _log(rng, 1, 128 if kind == "build" else 10_000)
    # a drawn call compares at most as many pairs as the listed bulk calls of its format
    most = 2.5e8 if prec == "fp32" else 1e9
    while nq * nprobe * (n / nlist) > most:
        nq = max(1, nq // 2)
    per_query = kind == "plan" or rng.random() < 0.25
    return _case(None, kind, prec, n, d, widths, nlist, -nprobe if per_query else nprobe, nq,
                 -1 if kind == "plan" else rng.choice([1, 10, 10, 37, 100]), rng.choice([0, 0, nlist]),
                 rng.choice([0.008, 0.02, 0.05]), zipf=rng.choice([0.0, 1.1]))


# ------------------------------------------------------------------ inputs
def _widths(c):
    out = []
    for part in c["widths"].split("+"):
        w, r = part.split("x")
        out += [int(w)] * int(r)
    return out


def _lloyd(X, nlist, gen):
    """A few Lloyd iterations on a sample (means by one-hot products: the same bits on
    every run)."""
    s = X[torch.randint(0, X.shape[0], (min(X.shape[0], 64 * nlist),), generator=gen, device=DEV)]
    C = s[torch.randperm(s.shape[0], generator=gen, device=DEV)[:nlist]].clone()
    lists = torch.arange(nlist, device=DEV)
    for _ in range(10):
        a = torch.cat([(C.square().sum(1) - 2 * p @ C.T).argmin(1) for p in s.split(65_536)])
        sums, cnt = torch.zeros_like(C), torch.zeros(nlist, device=DEV)
        for p, l in zip(s.split(65_536), a.split(65_536)):
            hot = (lists[:, None] == l).float()
            sums += hot @ p
            cnt += hot.sum(1)
        C = torch.where(cnt[:, None] > 0, sums / cnt.clamp(min=1)[:, None], C)
    return C


def _inputs(c, seed):
    """X, Q, O (FP64), coarse centroids and the per-query parameters, on the GPU."""
    gen = torch.Generator(device=DEV).manual_seed(int(seed) * 7919 + 17)
    n, d, nq, m = c["n"], c["d"], c["nq"], c["clusters"]

    def randn(*shape):
        return torch.randn(*shape, generator=gen, device=DEV)

    O, R = torch.linalg.qr(randn(d, d).double())
    O = O * torch.sign(torch.diagonal(R))
    A = (torch.exp(-0.5 * c["decay"] * torch.arange(d, device=DEV, dtype=torch.float64)) * O).float().T.contiguous()
    centres = randn(m, d) if m else None
    if m and c["zipf"]:
        centres *= 0.5
        cum = torch.arange(1, m + 1, device=DEV, dtype=torch.float64).pow(-c["zipf"]).cumsum(0).cpu()
    X = torch.empty(n + nq, d, device=DEV)
    for s in range(0, n + nq, 500_000):
        e = min(n + nq, s + 500_000)
        torch.matmul(randn(e - s, d), A, out=X[s:e])
        if m and c["zipf"]:
            u = torch.rand(e - s, generator=gen, device=DEV, dtype=torch.float64) * float(cum[-1])
            X[s:e] += centres[torch.searchsorted(cum.to(DEV), u).clamp(max=m - 1)]
        elif m:
            X[s:e] += centres[torch.randint(0, m, (e - s,), generator=gen, device=DEV)]
    X, Q = X[:n], X[n:].clone()
    if c["nlist"] == 1:
        C = torch.zeros(1, d, device=DEV)
    elif m == c["nlist"]:
        C = centres
    else:
        C = _lloyd(X, c["nlist"], gen)
    nprobe, k = c["nprobe"], c["k"]
    if nprobe < 0:
        nprobe = torch.randint(1, -nprobe + 1, (nq,), generator=gen, device=DEV, dtype=torch.int32)
    if k < 0:
        k = torch.tensor([1, 10, 100], device=DEV, dtype=torch.int32)[
            torch.randint(0, 3, (nq,), generator=gen, device=DEV)]
    return dict(X=X, Q=Q, O=O, A=A, C=C, nprobe=nprobe, k=k, gen=gen)


def _transform(c, i, T=None):
    lam = torch.exp(-c["decay"] * torch.arange(c["d"], dtype=torch.float64))
    T = i["O"].T.contiguous() if T is None else T
    return pano.panorama_transform_import(T.cpu().numpy(), np.zeros(c["d"]), lam.numpy())


def _shaped(c, i):
    """O^T with a random rotation inside every level (what spectrum shaping applies)."""
    T, a = i["O"].T.clone(), 0
    for w in _widths(c):
        H, R = torch.linalg.qr(torch.randn(w, w, generator=i["gen"], device=DEV).double())
        T[a:a + w] = (H * torch.sign(torch.diagonal(R))) @ T[a:a + w]
        a += w
    return T


def _assign(X, C):
    """Nearest centroid of every row: FP32 expansion, the best two re-scored in FP64."""
    if C.shape[0] == 1:
        return torch.zeros(X.shape[0], dtype=torch.int64, device=X.device)
    out = []
    for p in X.split(100_000):
        top = (C.square().sum(1) - 2 * p @ C.T).topk(2, largest=False).indices
        two = torch.stack([(p.double() - C[top[:, j]].double()).square().sum(1) for j in (0, 1)], 1)
        out.append(torch.where(two[:, 0] <= two[:, 1], top[:, 0], top[:, 1]))
    return torch.cat(out)


def _quantiser(c, i, T):
    """The coded database of a PQ case: lists, codebooks (sampled residual subvectors)
    and the nearest codeword of every residual subvector."""
    n, d, m = c["n"], c["d"], c["m"]
    a = _assign(i["X"], i["C"])
    T32 = T.float()
    R = i["X"] @ T32.T - (i["C"] @ T32.T)[a]
    ds = d // m
    pick = torch.randperm(n, generator=i["gen"], device=DEV)[:256]
    cb = R[pick].view(256, m, ds).transpose(0, 1).contiguous()
    codes = torch.empty(n, m, dtype=torch.uint8, device=DEV)
    for j in range(m):
        r = R[:, j * ds:(j + 1) * ds]
        codes[:, j] = (cb[j].square().sum(1) - 2 * r @ cb[j].T).argmin(1)
    return a, cb, codes


def _candidates(c, i):
    """Each query's candidate ids from a coarse first stage: the nearest by the leading
    eighth of the rotated coordinates."""
    h = max(1, c["d"] // 8)
    V = i["O"][:, :h].float()
    Xh, Qh = i["X"] @ V, i["Q"] @ V
    n2 = Xh.square().sum(1)
    return torch.cat([(n2 - 2 * q @ Xh.T).topk(c["kprime"], largest=False).indices for q in Qh.split(512)])


def prepare(case, seed):
    c = case
    i = _inputs(c, seed)
    s = {"kind": c["kind"], "Q": i["Q"], "nprobe": i["nprobe"], "k": i["k"]}
    if c["kind"] == "pq":
        T = _shaped(c, i)
        a, cb, codes = _quantiser(c, i, T)
        s["idx"] = pano.panorama_build_ivfpq(_transform(c, i, T), i["X"], c["nlist"], c["m"], len(_widths(c)),
                                             centroids=i["C"], assign=a.to(torch.int32), codebooks=cb,
                                             codes=codes)
        return s
    t = _transform(c, i)
    if c["kind"] == "refine":
        s["cand"] = _candidates(c, i)
        s["idx"] = pano.panorama_build_flat(t, i["X"], level_widths=_widths(c))
        return s
    if c["kind"] == "build":
        s.update(X=i["X"], t=t, C=i["C"].cpu().numpy(), nlist=c["nlist"], widths=_widths(c), prec=PREC[c["prec"]])
        return s
    s["idx"] = pano.panorama_build_ivf(t, i["X"], c["nlist"], level_widths=_widths(c),
                                       precision=PREC[c["prec"]], centroids=i["C"])
    if c["kind"] == "plan":
        s["plan"] = pano.Plan(s["idx"], s["Q"], s["nprobe"], s["k"], k_max=100 if c["k"] < 0 else c["k"])
    if c["kind"] == "server":
        s["server"] = pano.Server(s["idx"], max_batch=1024, max_inflight=4, k_max=c["k"])
        s["Q"], s["nprobe"] = s["Q"].cpu().numpy(), s["nprobe"].cpu().numpy()
        s["at"] = np.zeros(c["nq"])
    return s


def run(state):
    s = state
    if s["kind"] == "search":
        return s["idx"].search(s["Q"], s["nprobe"], s["k"])
    if s["kind"] == "plan":
        return s["plan"].launch()
    if s["kind"] == "pq":
        return s["idx"].search_pq(s["Q"], s["nprobe"], s["k"])
    if s["kind"] == "refine":
        return s["idx"].refine(s["Q"], s["cand"], s["k"])
    if s["kind"] == "build":
        idx = pano.panorama_build_ivf(s["t"], s["X"], s["nlist"], level_widths=s["widths"],
                                      precision=s["prec"], centroids=s["C"])
        return idx.search(s["Q"], s["nprobe"], s["k"]) + (idx.assignment(),)
    ids, dists, _ = s["server"].run_trace(s["Q"], s["at"], s["nprobe"], s["k"])
    return ids, dists


def _mean(v):
    return (1 - v) / 2 if v < 0 else v


def work(case):
    """What a pass cannot do without: every candidate's first level (pruning may spare
    the rest, more or less of it by the data), the queries' transform and the coarse
    distances; the queries, the first slices of the probed lists, the centroids and the
    transform read once and the results written once."""
    c = case
    n, d, nq = c["n"], c["d"], c["nq"]
    w0, k = _widths(c)[0], (100 if c["k"] < 0 else c["k"])
    out = nq * k * 12
    if c["kind"] == "refine":
        distinct = n * (1 - (1 - c["kprime"] / n) ** nq)
        return {"bytes": 4 * nq * d + 8 * nq * c["kprime"] + 4 * distinct * w0 + 4 * d * d + out,
                "flops": 2 * nq * (c["kprime"] * w0 + d * d)}
    p = min(1.0, _mean(c["nprobe"]) / c["nlist"])
    esize = {"fp32": 4, "bf16": 2, "fp8": 1, "pq": 0}[c["prec"]]
    row = w0 * esize if c["prec"] != "pq" else c["m"] // len(_widths(c))
    read = n * (1 - (1 - p) ** nq)
    pairs = nq * p * n
    by = 4 * nq * d + 4 * c["nlist"] * d + 4 * d * d + read * row + out
    fl = 2 * nq * d * (d + c["nlist"]) + (2 * w0 if c["prec"] != "pq" else c["m"] // len(_widths(c))) * pairs
    if c["kind"] == "build":  # rows in, rows and slices out; transform and assignment
        by += n * d * (4 + 4 + esize) + 4 * n
        fl += 2 * n * d * (d + c["nlist"])
    return {"bytes": by, "flops": fl}


# ------------------------------------------------------------ 64-bit results
def _merge(best, q, d):
    """Lowers rows q of the ascending distances best by the candidate distances d."""
    best[q] = torch.cat([best[q], d], 1).topk(best.shape[1], largest=False).values


def _exact_ivf(c, i):
    """Distances of every query's nearest vectors in its probed lists.  Vectors are
    preselected per list by FP32 expansion distances, with room to spare, and scored in
    FP64."""
    X, Q, C, nlist = i["X"], i["Q"], i["C"], c["nlist"]
    nq, kmax = c["nq"], (100 if c["k"] < 0 else c["k"])
    a = _assign(X, C)
    order = a.argsort(stable=True)
    off = [0] + torch.bincount(a, minlength=nlist).cumsum(0).tolist()
    npq = i["nprobe"] if torch.is_tensor(i["nprobe"]) else torch.full((nq,), i["nprobe"], device=DEV)
    top = min(nlist, int(npq.max()))
    near = torch.cat([torch.cdist(q.double(), C.double(), compute_mode="use_mm_for_euclid_dist")
                      .topk(top, largest=False).indices for q in Q.split(2048)])
    probed = torch.zeros(nq, nlist, dtype=torch.bool, device=DEV)
    probed.scatter_(1, near, torch.arange(top, device=DEV) < npq[:, None])
    per = probed.T.nonzero()
    cnt = [0] + torch.bincount(per[:, 0], minlength=nlist).cumsum(0).tolist()
    keep = kmax + 16
    cand_d = torch.full((nq, keep), math.inf, device=DEV)
    cand_i = torch.zeros(nq, keep, dtype=torch.int64, device=DEV)
    q2 = Q.square().sum(1)
    for l in range(nlist):
        rows, qs = order[off[l]:off[l + 1]], per[cnt[l]:cnt[l + 1], 1]
        for b in qs.split(max(1, 200_000_000 // max(1, rows.numel()))):
            if not rows.numel() or not b.numel():
                continue
            x = X[rows]
            dist = torch.addmm(q2[b][:, None] + x.square().sum(1), Q[b], x.T, alpha=-2)
            v, j = dist.topk(min(keep, rows.numel()), largest=False, sorted=False)
            v, s = torch.cat([cand_d[b], v], 1).topk(keep, largest=False)
            cand_i[b] = torch.cat([cand_i[b], rows[j]], 1).gather(1, s)
            cand_d[b] = v
    out = torch.empty(nq, kmax, dtype=torch.float64, device=DEV)
    for s in range(0, nq, 512):
        e = (X[cand_i[s:s + 512]].double() - Q[s:s + 512, None].double()).square().sum(2)
        e[cand_d[s:s + 512].isinf()] = math.inf
        out[s:s + 512] = e.topk(kmax, largest=False).values
    return out


def _exact_pq(c, i):
    T = _shaped(c, i)
    a, cb, codes = _quantiser(c, i, T)
    n, d, m, nq, nlist = c["n"], c["d"], c["m"], c["nq"], c["nlist"]
    # the list-residual frame: (q~ - c~) against the decoded residual
    qt, ct = i["Q"].double() @ T.T, i["C"].double() @ T.T
    npq = i["nprobe"] if torch.is_tensor(i["nprobe"]) else torch.full((nq,), i["nprobe"], device=DEV)
    near = torch.cdist(i["Q"].double(), i["C"].double(), compute_mode="use_mm_for_euclid_dist").argsort(1)
    best = torch.full((nq, c["k"]), math.inf, dtype=torch.float64, device=DEV)
    which = torch.arange(m, device=DEV)
    for l in range(nlist):
        rows = (a == l).nonzero()[:, 0]
        qs = ((near == l) & (torch.arange(nlist, device=DEV) < npq[:, None])).any(1).nonzero()[:, 0]
        if not rows.numel() or not qs.numel():
            continue
        x = cb[which, codes[rows].long()].reshape(rows.numel(), d).double()
        r = qt[qs] - ct[l]
        _merge(best, qs, (r.square().sum(1)[:, None] + x.square().sum(1) - 2 * r @ x.T).clamp(min=0))
    return best


def exact(case, seed):
    c = case
    i = _inputs(c, seed)
    if c["kind"] == "pq":
        return None, _exact_pq(c, i)
    if c["kind"] == "refine":
        cand, out = _candidates(c, i), []
        for q, j in zip(i["Q"].split(256), cand.split(256)):
            e = torch.cat([(i["X"][p].double() - r[:, None].double()).square().sum(2)
                           for r, p in zip(q.split(16), j.split(16))])
            out.append(torch.nn.functional.pad(e, (0, max(0, c["k"] - e.shape[1])), value=math.inf)
                       .topk(c["k"], largest=False).values)
        return None, torch.cat(out)
    d = _exact_ivf(c, i)
    if torch.is_tensor(i["k"]):  # past each query's own k there is nothing
        d[torch.arange(d.shape[1], device=DEV) >= i["k"][:, None]] = math.inf
    return (None, d, None) if c["kind"] == "build" else (None, d)
