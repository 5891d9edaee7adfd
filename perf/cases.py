"""The work a program has this library do, as cases of declared ranges.

A case is a dict of plain values; its ``kind`` names the entry point:

* ``search``: Index.search / Index.search_host, a query batch against an IVF
  (or flat) index -- the library's main path;
* ``two_stage``: Index.search_two_stage, the MSB-first search for few queries;
* ``train``: EstimatedScores, forward and backward, a query tower's step
  against a fixed compressed corpus;
* ``encode``: Algorithm 1 on rotated residuals;
* ``build``: build_index of new rows (and what an application stores of it).

Rows are Gaussian mixtures as in ``synthetic`` (drawn here on the GPU, so that
preparing a case takes about a second): "ivf" rows come from nlist/16
components with per-dimension scales U(0.5, 2), each row assigned to the
nearest of nlist sampled rows (so several lists share a component, as k-means
gives); "zipf" rows from nlist unit-scale components with Zipf(1.1) sizes, a
list being a component.
"""
import math

import numpy as np
import torch

from paper_2409_09913_gb300 import erq
from paper_2409_09913_gb300.autograd import EstimatedScores


def listed():
    return [
        # one request at a time: an interactive query against a 200k-row collection (latency and launches)
        dict(name="one_query_d960", kind="search", data="ivf", n=200_000, d=960, B=5, nlist=1024, nq=1, nprobe=16,
             k=10, rerank=20, precision="fp16", metric="l2"),
        # a small serving batch whose queries come from pinned host memory: inner product, odd sizes, 3-bit codes
        dict(name="serve_host_37q_d384_ip", kind="search", data="ivf", n=50_001, d=384, B=3, nlist=250, nq=37,
             nprobe=10, k=10, rerank=20, precision="fp16", metric="ip", host=True),
        # the plain method without an IVF: 10,000 x 128, 4 bits, 100 queries, top-10 of the re-ranked top-100
        dict(name="flat_n10k_d128_fp32", kind="search", data="ivf", n=10_000, d=128, B=4, nlist=1, nq=100, nprobe=1,
             k=10, rerank=100, precision="fp32", metric="l2"),
        # an ordinary batch on a medium collection, many lists per query
        dict(name="batch_512q_d512_nprobe64", kind="search", data="ivf", n=100_000, d=512, B=4, nlist=512, nq=512,
             nprobe=64, k=10, rerank=20, precision="fp16", metric="l2"),
        # offline batch over GIST-like rows: 10,000 queries, nprobe 16, about 78 queries per list
        dict(name="ivf_10kq_d960", kind="search", data="ivf", n=400_000, d=960, B=5, nlist=2048, nq=10_000, nprobe=16,
             k=10, rerank=20, precision="fp16", metric="l2", nosync=True),
        # the largest: Zipf-sized lists, a different nprobe (8..256) for each of 16,384 queries
        dict(name="zipf_16kq_d768", kind="search", data="zipf", n=500_000, d=768, B=5, nlist=4096, nq=16_384,
             nprobe=256, nprobe_lo=8, k=10, rerank=20, precision="fp16", metric="l2", nosync=True),
        # embedding-like unit vectors, 7 bits, FP8 queries
        dict(name="embed_4kq_d1536_fp8", kind="search", data="ivf", n=50_000, d=1536, B=7, nlist=512, nq=4000,
             nprobe=32, k=10, rerank=20, precision="fp8", metric="cos"),
        # the default precision of Index.search
        dict(name="ivf_1kq_d960_fp32", kind="search", data="ivf", n=100_000, d=960, B=5, nlist=512, nq=1000,
             nprobe=32, k=10, rerank=20, precision="fp32", metric="l2"),
        # the two-stage search in its regime of few queries per list
        dict(name="two_stage_16q_d960", kind="two_stage", data="ivf", n=200_000, d=960, B=5, nlist=1024, nq=16,
             nprobe=16, k=10, rerank=20, eps0=1.9),
        # a training step of a query tower: 100 scores per query and their gradient
        dict(name="train_4kq_d1024", kind="train", data="ivf", n=100_000, d=1024, B=4, nlist=512, nq=4096, nc=100,
             metric="l2"),
        # the encoder alone at the widest embeddings' dimension
        dict(name="encode_d3072_b8", kind="encode", n=2048, d=3072, B=8),
        # index build of a new collection: k-means, rotation, codes, layout; centroids, lists and codes read back
        dict(name="build_100k_d768", kind="build", data="ivf", n=100_000, d=768, B=5, nlist=256, kmeans=True),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["search"] * 6 + ["two_stage", "train", "encode", "build"])
    d = 64 * _log_int(rng, 2, 24)                       # 128 .. 1536
    B = rng.choice([1, 2, 3, 4, 5, 5, 6, 7, 8, 9])
    if kind == "encode":
        d = 64 * _log_int(rng, 1, 48)                   # 64 .. 3072
        B = rng.randint(1, 10)
        n = _log_int(rng, 100, 100_000)
        n = max(16, min(n, int(8e8 / (d * 2 ** B))))     # up to about the listed case's critical values
        return dict(kind=kind, n=n, d=d, B=B)
    n_max = 400_000
    n_max = min(n_max, int(3.6e11 / (d * d)), int(4e8 * 32 / (d * 2 ** B)))
    n = _log_int(rng, 5_000, max(6_000, n_max))
    nlist = max(8, min(4096, _log_int(rng, 16, max(17, n // 48))))
    if kind == "build":
        n = min(n, int(6e10 / (d * d)), 100_000)
        nlist = max(8, min(nlist, n // 48))
        return dict(kind=kind, data="ivf", n=n, d=d, B=B, nlist=nlist, kmeans=rng.random() < 0.5)
    if kind == "train":
        return dict(kind=kind, data="ivf", n=min(n, 100_000), d=min(d, 1024), B=B, nlist=nlist,
                    nq=_log_int(rng, 16, 4096), nc=_log_int(rng, 10, 100), metric=rng.choice(["l2", "l2", "ip"]))
    k = rng.choice([1, 5, 10, 10, 10])
    rerank = rng.choice([16, 20, 20, 32])
    if kind == "two_stage":
        nq = _log_int(rng, 1, 256)
        return dict(kind=kind, data="ivf", n=n, d=d, B=5 if B == 4 else B, nlist=nlist, nq=nq,
                    nprobe=min(nlist, _log_int(rng, 4, 64)), k=k, rerank=rerank, eps0=1.9)
    data = rng.choice(["ivf", "ivf", "ivf", "zipf"])
    precision = rng.choice(["fp16", "fp16", "fp16", "fp32", "fp32", "fp8"])
    if precision == "fp8":
        B = min(B, 8)
    nq = _log_int(rng, 1, 16_384)
    nprobe = min(nlist, _log_int(rng, 4, 256 if data == "zipf" else 96))
    pairs = nq * nprobe * n / nlist * (4 if data == "zipf" else 1)
    most = 4e8 if precision != "fp32" else 1.2e8
    if pairs * d / 768 > most:
        nq = max(1, int(nq * most / (pairs * d / 768)))
    case = dict(kind=kind, data=data, n=n, d=d, B=B, nlist=nlist, nq=nq, nprobe=nprobe, k=k, rerank=rerank,
                precision=precision, metric=rng.choice(["l2", "l2", "l2", "ip", "cos"]))
    if rng.random() < 0.25:
        case["host"] = True
    elif rng.random() < 0.4:
        case["nosync"] = True
    if data == "zipf" and nprobe > 8:
        case["nprobe_lo"] = 8
    return case


# ------------------------------------------------------------------------------------------------ inputs
def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(1_000_003 * (int(seed) + 1))
    return g


def _orthogonal(d, g):
    a = torch.randn(d, d, generator=g, device="cuda", dtype=torch.float64)
    q, r = torch.linalg.qr(a)
    return (q * torch.sign(torch.diagonal(r))[None, :]).to(torch.float32).contiguous()


def _nearest(X, S, chunk=1 << 16):
    """Row of S nearest to each row of X (FP32)."""
    sn = (S * S).sum(1)
    out = torch.empty(len(X), dtype=torch.int32, device=X.device)
    for s0 in range(0, len(X), chunk):
        b = X[s0:s0 + chunk]
        out[s0:s0 + len(b)] = (sn[None, :] - 2.0 * (b @ S.T)).argmin(1).to(torch.int32)
    return out


def _collection(case, seed):
    """Rows X, their lists, queries Q and P, from the seed alone."""
    g = _generator(seed)
    n, d, nlist, nq = case["n"], case["d"], case["nlist"], case.get("nq", 1)
    zipf = case["data"] == "zipf"
    ncomp = nlist if zipf else max(1, nlist // 16)
    if nlist == 1:
        ncomp = 16
    centres = 2.0 * torch.randn(ncomp, d, generator=g, device="cuda")
    if zipf:
        w = 1.0 / torch.arange(1, ncomp + 1, device="cuda", dtype=torch.float64) ** 1.1
        lab = torch.multinomial(w / w.sum(), n, replacement=True, generator=g)
        qlab = torch.multinomial(w / w.sum(), nq, replacement=True, generator=g)
    else:
        lab = torch.randint(0, ncomp, (n,), generator=g, device="cuda")
        qlab = torch.randint(0, ncomp, (nq,), generator=g, device="cuda")
    scales = None if zipf else 0.5 + 1.5 * torch.rand(ncomp, d, generator=g, device="cuda")

    def rows(labels):
        x = torch.randn(len(labels), d, generator=g, device="cuda")
        for s0 in range(0, len(labels), 1 << 16):
            b = labels[s0:s0 + (1 << 16)]
            v = x[s0:s0 + len(b)]
            if scales is not None:
                v *= scales[b]
            v += centres[b]
        if case.get("metric") == "cos":
            x /= x.norm(dim=1, keepdim=True)
        return x

    X, Q = rows(lab), rows(qlab)
    P = _orthogonal(d, g)
    if zipf:
        assign = lab.to(torch.int32)
    elif nlist == 1:
        assign = torch.zeros(n, dtype=torch.int32, device="cuda")
    else:
        assign = _nearest(X, X[torch.randperm(n, generator=g, device="cuda")[:nlist]])
    return X, assign, Q, P, g


def _nprobe_per_query(case, g):
    if "nprobe_lo" not in case:
        return None
    return torch.randint(case["nprobe_lo"], case["nprobe"] + 1, (case["nq"],), generator=g, device="cuda",
                         dtype=torch.int32)


def _residuals(case, seed):
    return torch.randn(case["n"], case["d"], generator=_generator(seed), device="cuda")


def _train_inputs(case, g):
    ids = torch.randint(0, case["n"], (case["nq"], case["nc"]), generator=g, device="cuda")
    grad = torch.randn(case["nq"], case["nc"], generator=g, device="cuda")
    return ids, grad


def prepare(case, seed):
    kind = case["kind"]
    if kind == "encode":
        return dict(kind=kind, B=case["B"], R=_residuals(case, seed))
    X, assign, Q, P, g = _collection(case, seed)
    if kind == "build":
        return dict(kind=kind, X=X, P=P, B=case["B"], nlist=case["nlist"], assign=None if case["kmeans"] else assign)
    ix = erq.build_index(X, P, case["B"], case["nlist"], assign=assign, normalize=case.get("metric") == "cos")
    if kind == "train":
        ids, grad = _train_inputs(case, g)
        return dict(kind=kind, ix=ix, Q=Q, ids=ids, grad=grad, metric=case["metric"])
    kw = dict(rerank_k=case["rerank"], nprobe=case["nprobe"], nprobe_per_query=_nprobe_per_query(case, g))
    if kind == "two_stage":
        return dict(kind=kind, ix=ix, Q=Q, k=case["k"], kw=dict(kw, eps0=case["eps0"]))
    kw.update(precision=case["precision"], metric=case["metric"], async_mode=bool(case.get("nosync")))
    if case.get("host"):
        return dict(kind="search_host", ix=ix, Q=Q.cpu().pin_memory(), k=case["k"], kw=kw)
    return dict(kind=kind, ix=ix, Q=Q, k=case["k"], kw=kw)


def run(state):
    kind = state["kind"]
    if kind == "search":
        return state["ix"].search(state["Q"], state["k"], **state["kw"])
    if kind == "search_host":
        return state["ix"].search_host(state["Q"], state["k"], **state["kw"])
    if kind == "two_stage":
        return state["ix"].search_two_stage(state["Q"], state["k"], **state["kw"])
    if kind == "train":
        Q = state["Q"].detach().requires_grad_()
        est = EstimatedScores.apply(Q, state["ix"], state["ids"], state["metric"])
        (gq,) = torch.autograd.grad(est, Q, state["grad"])
        return est.detach(), gq
    if kind == "encode":
        return erq.encode(state["R"], state["B"])
    ix = erq.build_index(state["X"], state["P"], state["B"], state["nlist"], assign=state["assign"])
    return {f: ix.export(f) for f in ("centroids", "list_offsets", "list_ids", "codes", "f_add", "f_res")}


def work(case):
    """Bytes and operations of one pass: every input that the path needs read
    once, every output written once; multiply-adds of the method in its stated
    form (2 per coordinate of an estimated pair)."""
    kind, d, B = case["kind"], case["d"], case["B"]
    cb = 2 if B > 8 else 1
    if kind == "encode":
        n = case["n"]
        # the sums over the coordinates at the optimum (norm, inner product); the walk's length is not a given
        return {"bytes": n * d * (4 + cb) + 8 * n, "flops": 4.0 * n * d}
    n, nlist = case["n"], case["nlist"]
    if kind == "build":
        return {"bytes": 4.0 * n * d + n * d * cb + 16.0 * n + 4.0 * nlist * d, "flops": 2.0 * n * d * d}
    nq = case["nq"]
    row = B * d / 8 + 8
    if kind == "train":
        pairs = nq * case["nc"]
        rows = n * (1 - math.exp(-pairs / n))
        return {"bytes": rows * row + 4.0 * nlist * d + 4.0 * d * d + 8.0 * nq * d + 16.0 * pairs,
                "flops": 2.0 * 2 * nq * d * d + 2.0 * 2 * pairs * d}
    nprobe = (case["nprobe"] + case["nprobe_lo"]) / 2 if "nprobe_lo" in case else case["nprobe"]
    pairs = nq * nprobe * n / nlist
    rows = n * (1 - math.exp(-nq * nprobe / nlist)) if nlist > 1 else n
    kp = max(case["k"], case["rerank"])
    raw = n * (1 - math.exp(-nq * kp / n))
    if kind == "two_stage":
        row = d / 8 + 8                                 # every probed row's first bit plane
    return {"bytes": rows * row + raw * 4 * d + 4.0 * nq * d + 4.0 * d * d + 4.0 * nlist * d + 12.0 * nq * case["k"],
            "flops": 2.0 * pairs * d + 2.0 * nq * d * d + (2.0 * nq * nlist * d if nlist > 1 else 0.0)}


# ------------------------------------------------------------------------------------------------ 64-bit answers
def _codes64(r, B):
    """Algorithm 1 in 64 bits on rows r: the signed grid point of largest cosine
    (y in odd multiples of 1/2) and <y, r>."""
    n, d = r.shape
    M = 2 ** (B - 1) - 1
    y = torch.empty_like(r)
    ip = torch.empty(n, dtype=torch.float64, device=r.device)
    step = max(1, (1 << 25) // (d * max(M, 1)))
    lev = torch.arange(1, M + 1, dtype=torch.float64, device=r.device)
    for s0 in range(0, n, step):
        a = r[s0:s0 + step].abs()
        m = torch.zeros(a.shape, dtype=torch.float64, device=r.device)
        if M > 0:
            t, idx = (lev[None, None, :] / a[:, :, None]).reshape(len(a), -1).sort(dim=1, stable=True)
            co, le = idx // M, idx % M
            S = 0.5 * a.sum(1, keepdim=True) + torch.where(torch.isinf(t), 0.0, a.gather(1, co)).cumsum(1)
            N = 0.25 * d + (2.0 * (le + 1)).to(torch.float64).cumsum(1)
            v = torch.where(torch.isinf(t), -1.0, S / N.sqrt())
            best, at = v.max(1)
            some = best > 0.5 * a.sum(1) / math.sqrt(0.25 * d)
            taken = (torch.arange(t.shape[1], device=r.device)[None, :] <= at[:, None]) & some[:, None]
            m.scatter_add_(1, co, taken.to(torch.float64))
        yy = m + 0.5
        ip[s0:s0 + step] = (yy * a).sum(1)
        y[s0:s0 + step] = torch.where(r[s0:s0 + step] >= 0, yy, -yy)
    return y, ip


def _f_res(nr2, ip):
    """-2 ||o'||^2 / <y, o'>, 0 for a row that is its list's centroid."""
    return torch.where(nr2 > 0, -2.0 * nr2 / ip, 0.0)


def _means64(X, assign, nlist):
    C = torch.zeros(nlist, X.shape[1], dtype=torch.float64, device=X.device)
    for s0 in range(0, len(X), 1 << 16):
        C.index_add_(0, assign[s0:s0 + (1 << 16)].long(), X[s0:s0 + (1 << 16)].double())
    return C / torch.bincount(assign.long(), minlength=nlist).clamp(min=1)[:, None]


def _exact_search(case, seed):
    """Exact top-k over the rows of the probed lists."""
    X, assign, Q, P, g = _collection(case, seed)
    del P
    nlist, k = case["nlist"], case["k"]
    npq = _nprobe_per_query(case, g)
    ip = case.get("metric", "l2") != "l2"
    if case.get("metric") == "cos":
        X = (X.double() / X.double().norm(dim=1, keepdim=True)).float()
        Q = (Q.double() / Q.double().norm(dim=1, keepdim=True)).float()
    C = _means64(X, assign, nlist)
    xn = (X * X).sum(1)
    out = torch.empty(len(Q), k, dtype=torch.float64, device="cuda")
    step = max(1, min(len(Q), (1 << 29) // len(X)))
    for s0 in range(0, len(Q), step):
        q = Q[s0:s0 + step]
        cd = -(q.double() @ C.T)
        if not ip:
            cd = (C * C).sum(1)[None, :] + 2.0 * cd
        order = cd.topk(case["nprobe"], dim=1, largest=False).indices
        keep = torch.arange(case["nprobe"], device="cuda")[None, :] < (
            npq[s0:s0 + step, None] if npq is not None else case["nprobe"])
        probed = torch.zeros(len(q), nlist + 1, dtype=torch.bool, device="cuda")
        probed.scatter_(1, torch.where(keep, order, nlist), True)
        v = -(q @ X.T)
        if not ip:
            v = xn[None, :] + 2.0 * v
        v.masked_fill_(~probed[:, assign.long()], math.inf)
        near = v.topk(min(k + 22, len(X)), dim=1, largest=False).indices
        for i0 in range(0, len(q), 1024):
            qq = q[i0:i0 + 1024].double()[:, None, :]
            xx = X[near[i0:i0 + 1024]].double()
            e = -(qq * xx).sum(2) if ip else ((qq - xx) ** 2).sum(2)
            e = torch.where(torch.isinf(v[i0:i0 + 1024].gather(1, near[i0:i0 + 1024])), math.inf, e)
            out[s0 + i0:s0 + i0 + len(e)] = e.sort(1).values[:, :k]
    return -out if ip else out


def exact(case, seed):
    kind, B = case["kind"], case["B"]
    if kind in ("search", "two_stage"):
        return None, _exact_search(case, seed)
    if kind == "encode":
        r = _residuals(case, seed).double()
        _, ip = _codes64(r, B)
        nr2 = (r * r).sum(1)
        return None, nr2, _f_res(nr2, ip)
    if kind == "build":
        if case["kmeans"]:
            return None
        X, assign, _, P, _ = _collection(case, seed)
        order = assign.long().argsort(stable=True)
        C = _means64(X, assign, case["nlist"])
        c32 = C.float()
        fa, fr = [], []
        for s0 in range(0, len(X), 1 << 14):
            rows = order[s0:s0 + (1 << 14)]
            o = ((X[rows] - c32[assign[rows].long()]).double() @ P.double()).float().double()
            _, ip = _codes64(o, B)
            nr2 = (o * o).sum(1)
            fa.append(nr2)
            fr.append(_f_res(nr2, ip))
        return dict(centroids=C, list_offsets=None, list_ids=None, codes=None, f_add=torch.cat(fa), f_res=torch.cat(fr))
    # train: est = ||q - c||^2 + ||o'||^2 + f_res <y, P^T (q - c)> (or <c, q> - f_res / 2 <y, P^T q>), gradient in q
    X, assign, Q, P, g = _collection(case, seed)
    ids, grad = _train_inputs(case, g)
    c32 = _means64(X, assign, case["nlist"]).float()
    P = P.double()
    used, inv = ids.unique(return_inverse=True)
    inv = inv.reshape(ids.shape)
    y = torch.empty(len(used), case["d"], dtype=torch.float64, device="cuda")
    fres = torch.empty(len(used), dtype=torch.float64, device="cuda")
    nr2 = torch.empty_like(fres)
    for s0 in range(0, len(used), 1 << 14):
        rows = used[s0:s0 + (1 << 14)]
        o = ((X[rows] - c32[assign[rows].long()]).double() @ P).float().double()
        y[s0:s0 + len(rows)], ip = _codes64(o, B)
        nr2[s0:s0 + len(rows)] = (o * o).sum(1)
        fres[s0:s0 + len(rows)] = _f_res(nr2[s0:s0 + len(rows)], ip)
    cl = assign[used].long()
    est = torch.empty(ids.shape, dtype=torch.float64, device="cuda")
    gq = torch.empty(len(Q), case["d"], dtype=torch.float64, device="cuda")
    for s0 in range(0, len(Q), 64):
        q, j, w = Q[s0:s0 + 64].double(), inv[s0:s0 + 64], grad[s0:s0 + 64].double()
        cc, yy, f = c32[cl[j]].double(), y[j], fres[j]
        qc = q[:, None, :] - cc
        if case["metric"] == "ip":
            est[s0:s0 + 64] = (cc * q[:, None, :]).sum(2) - 0.5 * f * (yy * (q @ P)[:, None, :]).sum(2)
            gq[s0:s0 + 64] = (w[..., None] * cc).sum(1) - 0.5 * ((w * f)[..., None] * yy).sum(1) @ P.T
        else:
            est[s0:s0 + 64] = (qc * qc).sum(2) + nr2[j] + f * (yy * (qc @ P)).sum(2)
            gq[s0:s0 + 64] = 2.0 * (w[..., None] * qc).sum(1) + ((w * f)[..., None] * yy).sum(1) @ P.T
    return est, gq
