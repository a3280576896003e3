"""Timed cases of the EMD lower-bound library: what a program that holds a database of
histograms asks of it, through the package's public entry points.

A case is a database (text histograms over an embedded vocabulary, or 28x28 images with a
ground-cost matrix), the options it was created with, and one call on a set of queries.
The sizes are the repository's own workloads (tiny text V = 2000; text V = 1e5, n = 2e4,
m = 300; images n = 6e4; the serving database V = 2e5, n = 1e6 with queries of 5..2000
bins) and cuts of them.  Inputs follow the same laws as the synthetic workloads -- Zipf(1.1)
vocabularies, log-normal document sizes, unit-norm embeddings, stroke images -- and are
drawn on the GPU from the seed.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1812_02091_gb300 as emd

GRID = 28


def listed():
    cases = [
        # the smallest call: a handful of short queries on a tiny database with every option at
        # its default (plain FP32), host buffers; launches and host work dominate
        dict(name="tiny_topk", kind="topk", data="text", V=2000, m=64, n=1000, doc_h=25, nq=10, qlo=10, qhi=40,
             precision="fp32", meas="act", k=3, K=10, host=True, defaults=True),
        # one interactive search against the text database, host buffers: latency
        dict(name="single_topk", kind="topk", data="text", V=100000, m=300, n=20000, doc_h=100, nq=1, qlo=113, qhi=113,
             precision="fp32_tc", meas="act", k=4, K=16, host=True),
        # a full batch of document-sized queries against the text database: bulk search
        dict(name="text_topk", kind="topk", data="text", V=100000, m=300, n=20000, doc_h=100, nq=64, qlo=40, qhi=260,
             precision="fp32_tc", meas="act", k=4, K=16, host=False),
        # the serving-size database, a full batch of mixed query sizes: the headline workload
        dict(name="serving_topk", kind="topk", data="text", V=200000, m=300, n=1000000, doc_h=100, nq=64, qlo=5, qhi=2000,
             precision="fp32_tc", meas="act", k=4, K=16, host=False),
        # the same search with the default arithmetic (plain FP32)
        dict(name="fp32_topk", kind="topk", data="text", V=100000, m=300, n=20000, doc_h=100, nq=64, qlo=40, qhi=260,
             precision="fp32", meas="act", k=4, K=16, host=False),
        # the approximate Phase 1 with exact re-rank, a partly filled batch
        dict(name="bf16_topk", kind="topk", data="text", V=100000, m=300, n=20000, doc_h=100, nq=41, qlo=20, qhi=400,
             precision="bf16", meas="act", k=2, K=10, host=False),
        # ICT, the tightest bound, as a re-ranking search
        dict(name="ict_topk", kind="topk", data="text", V=100000, m=300, n=20000, doc_h=100, nq=32, qlo=40, qhi=260,
             precision="fp32_tc", meas="ict", k=1, K=16, host=False),
        # image retrieval with a pixel ground-cost matrix, the evaluation's k = 8
        dict(name="image_topk", kind="topk", data="image", V=784, m=0, n=60000, doc_h=0, nq=64, qlo=0, qhi=0,
             precision="fp32", meas="act", k=8, K=16, host=False),
        # every distance in both directions (a kernel matrix for a classifier, a re-ranking stage)
        dict(name="distances_max", kind="dist", data="text", V=100000, m=300, n=20000, doc_h=100, nq=29, qlo=20, qhi=400,
             precision="fp32_tc", meas="act", k=4, dir="max"),
        # every forward distance with the cheapest bound, odd sizes
        dict(name="distances_fwd", kind="dist", data="text", V=99991, m=300, n=99991, doc_h=100, nq=61, qlo=5, qhi=700,
             precision="fp32_tc", meas="rwmd", k=1, dir="fwd"),
        # all pairs of a text collection (nearest-neighbour graph), host buffers
        dict(name="all_pairs", kind="pairs", data="text", V=50000, m=300, n=3000, doc_h=100, nq=3000, qlo=0, qhi=0,
             precision="fp32_tc", meas="act", k=2, K=16),
        # requests through the server: a burst of mixed-size queries submitted one by one
        dict(name="serve_burst", kind="serve", data="text", V=100000, m=300, n=100000, doc_h=100, nq=128, qlo=5, qhi=1000,
             precision="fp32_tc", meas="act", k=4, K=16),
    ]
    return [dict(c, defaults=c.get("defaults", False)) for c in cases]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: a kind of call, then sizes over its range (logarithmic), odd ones as they fall."""
    case = _draw(rng)
    return dict(case, defaults=case["precision"] == "fp32" and case["n"] <= 2000)


def _draw(rng):
    what = rng.choice(["topk", "topk", "topk", "topk", "image", "dist", "dist", "pairs", "serve"])
    prec = rng.choice(["fp32_tc", "fp32_tc", "fp32", "bf16"])
    meas = rng.choice(["act", "act", "act", "rwmd", "omr", "ict"])
    k = rng.randint(2, 8) if meas == "act" else 1
    if what == "image":
        return dict(kind="topk", data="image", V=784, m=0, n=_log_int(rng, 500, 60000), doc_h=0, nq=rng.randint(1, 64),
                    qlo=0, qhi=0, precision="fp32", meas="act", k=rng.randint(1, 16), K=rng.randint(1, 16),
                    host=rng.random() < 0.5)
    n = _log_int(rng, 1000, 200000)
    base = dict(data="text", V=_log_int(rng, 2000, 200000), m=rng.choice([64, 300, rng.randint(32, 300)]), n=n,
                doc_h=rng.randint(25, 100))
    qlo = _log_int(rng, 5, 100)
    qhi = min(_log_int(rng, qlo, 1500), base["V"] // 4)
    qlo = min(qlo, qhi)
    if what == "topk":
        if meas == "ict":
            prec = rng.choice(["fp32_tc", "fp32"])
            n = min(n, 20000)
            qhi = min(qhi, 400)
            qlo = min(qlo, qhi)
        return dict(base, kind="topk", n=n, nq=rng.randint(1, 64), qlo=qlo, qhi=qhi, precision=prec, meas=meas, k=k,
                    K=rng.randint(1, 16), host=rng.random() < 0.5)
    if meas == "ict":
        meas, k = "act", 4
    if what == "dist":
        way = rng.choice(["fwd", "rev", "max"])
        if way != "fwd":
            n, qhi = min(n, 20000), min(qhi, 400)
        return dict(base, kind="dist", n=n, nq=rng.randint(1, 64), qlo=min(qlo, qhi), qhi=qhi,
                    precision=rng.choice(["fp32_tc", "fp32"]), meas=meas, k=k, dir=way)
    if what == "pairs":
        n = _log_int(rng, 300, 3000)
        return dict(base, kind="pairs", V=min(base["V"], 50000), n=n, nq=n, qlo=0, qhi=0, precision="fp32_tc", meas=meas,
                    k=k, K=rng.randint(1, 16))
    return dict(base, kind="serve", n=min(n, 100000), nq=rng.randint(16, 128), qlo=qlo, qhi=min(qhi, 1000),
                precision="fp32_tc", meas=meas, k=k, K=rng.randint(1, 16))


# ------------------------------------------------------------------ inputs

def _zipf(V):
    p = np.arange(1, V + 1, dtype=np.float64) ** -1.1
    return p / p.sum()


def _tokens_for(p, h):
    """Draws with replacement whose expected number of distinct ids is h."""
    lo, hi = 1.0, 64.0 * h + 64
    for _ in range(50):
        mid = 0.5 * (lo + hi)
        lo, hi = (mid, hi) if np.sum(-np.expm1(-mid * p)) < h else (lo, mid)
    return lo


def _weights(row_ptr, nnz, g):
    """Term counts 1..5, normalised per histogram in FP64."""
    c = torch.randint(1, 6, (nnz,), generator=g, device="cuda").double()
    lens = row_ptr[1:] - row_ptr[:-1]
    own = torch.repeat_interleave(torch.arange(lens.numel(), device="cuda"), lens)
    s = torch.zeros(lens.numel(), dtype=torch.float64, device="cuda").index_add_(0, own, c)
    return (c / s[own]).float()


def _text_docs(case, g):
    """Documents: distinct ids of log-normally many Zipf draws; CSR on the GPU (int64, int32, float32)."""
    V, n = case["V"], case["n"]
    p = _zipf(V)
    cdf = torch.from_numpy(np.cumsum(p) / p.sum()).cuda()
    typical = _tokens_for(p, min(case["doc_h"], V / 3))
    t = torch.exp(0.5 * torch.randn(n, generator=g, device="cuda", dtype=torch.float64)) * typical
    t = t.round().clamp(8, 10 * typical).long()
    cols, lens = [], []
    step = 100000
    for a in range(0, n, step):
        tt = t[a:a + step]
        own = torch.repeat_interleave(torch.arange(tt.numel(), device="cuda"), tt)
        u = torch.rand(own.numel(), generator=g, device="cuda", dtype=torch.float64)
        key = torch.unique_consecutive((own * V + torch.searchsorted(cdf, u).clamp(max=V - 1)).sort().values)
        lens.append(torch.bincount(key // V, minlength=tt.numel()))
        cols.append((key % V).int())
    row_ptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    row_ptr[1:] = torch.cat(lens).cumsum(0)
    col = torch.cat(cols)
    return row_ptr, col, _weights(row_ptr, col.numel(), g)


def _text_queries(case, g):
    """Queries of log-uniform sizes qlo..qhi: successive sampling by Gumbel keys, ids ascending."""
    V, nq = case["V"], case["nq"]
    logp = torch.from_numpy(np.log(_zipf(V))).float().cuda()
    r = torch.rand(nq, generator=g, device="cuda", dtype=torch.float64)
    h = torch.exp(math.log(case["qlo"]) + r * (math.log(case["qhi"]) - math.log(case["qlo"]))).round().long()
    rows = []
    for i in range(nq):
        e = torch.empty(V, device="cuda").exponential_(generator=g)
        rows.append((logp - torch.log(e)).topk(int(h[i])).indices.sort().values.int())
    row_ptr = torch.zeros(nq + 1, dtype=torch.int64, device="cuda")
    row_ptr[1:] = h.cumsum(0)
    col = torch.cat(rows)
    return row_ptr, col, _weights(row_ptr, col.numel(), g)


def _images(n, g):
    """Clipped sums of 3..6 Gaussian strokes on a 28x28 grid, small pixels zeroed: CSR on the GPU."""
    xy = torch.cartesian_prod(torch.arange(GRID, device="cuda"), torch.arange(GRID, device="cuda")).float()
    lens, cols, vals = [], [], []
    for a in range(0, n, 10000):
        c = min(10000, n - a)
        strokes = torch.randint(3, 7, (c,), generator=g, device="cuda")
        img = torch.zeros(c, GRID * GRID, device="cuda")
        for s in range(6):
            p0, p1 = (9 + 9 * torch.rand(c, 2, generator=g, device="cuda") for _ in range(2))
            sig = 1 + torch.rand(c, 1, generator=g, device="cuda")
            d = p1 - p0
            rel = xy[None] - p0[:, None]
            at = ((rel * d[:, None]).sum(-1) / d.square().sum(1, keepdim=True).clamp(min=1e-12)).clamp(0, 1)
            dist2 = (rel - at[..., None] * d[:, None]).square().sum(-1)
            img += (strokes > s)[:, None] * torch.exp(-dist2 / (2 * sig * sig))
        img = img.clamp(0, 1).double()
        img[img < 0.1] = 0
        img /= img.sum(1, keepdim=True)
        at = img.nonzero()
        lens.append(torch.bincount(at[:, 0], minlength=c))
        cols.append(at[:, 1].int())
        vals.append(img[at[:, 0], at[:, 1]].float())
    row_ptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    row_ptr[1:] = torch.cat(lens).cumsum(0)
    return row_ptr, torch.cat(cols), torch.cat(vals)


def _pixel_costs():
    xy = torch.cartesian_prod(torch.arange(GRID), torch.arange(GRID)).double().cuda()
    return (xy[:, None] - xy[None]).square().sum(-1).sqrt().float()


def _inputs(case, seed):
    """Ground costs (embeddings or matrix), documents and queries of a case, on the GPU."""
    g = torch.Generator(device="cuda").manual_seed(seed * 7919 + 17)
    if case["data"] == "image":
        return None, _pixel_costs(), _images(case["n"], g), _images(case["nq"], g)
    x = torch.randn(case["V"], case["m"], generator=g, device="cuda", dtype=torch.float64)
    e = (x / x.norm(dim=1, keepdim=True)).float()
    docs = _text_docs(case, g)
    return e, None, docs, docs if case["kind"] == "pairs" else _text_queries(case, g)


# ------------------------------------------------------------------ the calls

class _Database:
    """A database handle (and its server) that is released with the state that holds it."""

    def __init__(self, emb, cost, docs, options, serve):
        rp, col, val = (t.cpu().numpy() for t in docs)
        self.server = None
        self.db = emd.emd_db_create(None if emb is None else emb.cpu().numpy(), None if cost is None else cost.cpu().numpy(),
                                    rp, col, val, options)
        if serve:
            self.server = emd.emd_server_create(self.db, emd.emd_server_options_default())

    def __del__(self):
        if self.server is not None:
            emd.emd_server_destroy(self.server)
        if getattr(self, "db", None) is not None:
            emd.emd_db_destroy(self.db)


def _options(case, docs, queries):
    """The defaults, or options as the benchmark and the tests set them: the precision, room for the
    largest query, and for long queries a workspace that holds a full batch of them."""
    if case["defaults"]:
        return emd.emd_db_options_default()
    longest = int((queries[0][1:] - queries[0][:-1]).max())
    o = dict(precision=case["precision"], max_query_h=1024 if longest <= 1024 else 2048)
    if case["qhi"] > 700 and case["kind"] != "serve":
        o["batch_columns"] = 32768
    return emd.emd_db_options_default(**o)


def prepare(case, seed):
    emb, cost, docs, queries = _inputs(case, seed)
    handle = _Database(emb, cost, docs, _options(case, docs, queries), case["kind"] == "serve")
    rp, idx, w = queries
    state = dict(case=case, handle=handle, rp=rp.cpu().numpy())
    if case["kind"] in ("topk", "serve") and (case.get("host") or case["kind"] == "serve"):
        state.update(idx=idx.cpu().numpy(), w=w.cpu().numpy())
    elif case["kind"] != "pairs":
        state.update(idx=idx.contiguous(), w=w.contiguous())
    return state


def run(state):
    c, db = state["case"], state["handle"].db
    if c["kind"] == "pairs":
        return emd.emd_all_pairs_topk(db, c["meas"], c["k"], c["K"])
    if c["kind"] == "serve":
        server, rp = state["handle"].server, state["rp"]
        tickets = [emd.emd_server_submit(server, state["idx"][rp[i]:rp[i + 1]], state["w"][rp[i]:rp[i + 1]], c["meas"],
                                         c["k"], c["K"]) for i in range(c["nq"])]
        ids, dist = np.empty((c["nq"], c["K"]), np.int64), np.empty((c["nq"], c["K"]), np.float32)
        for i, t in enumerate(tickets):
            emd.emd_server_poll(server, t, -1, ids[i], dist[i])
        return ids, dist
    stream = torch.cuda.current_stream().cuda_stream
    if c["kind"] == "dist":
        out = torch.empty(c["nq"], c["n"], device="cuda")
        emd.emd_query_batch_device(db, state["rp"], state["idx"], state["w"], out, c["meas"], c["k"], c["dir"], stream)
        return out
    if c["host"]:
        return emd.emd_topk(db, state["rp"], state["idx"], state["w"], c["meas"], c["k"], "max", c["K"])
    ids = torch.empty(c["nq"], c["K"], device="cuda", dtype=torch.int64)
    dist = torch.empty(c["nq"], c["K"], device="cuda")
    emd.emd_topk_device(db, state["rp"], state["idx"], state["w"], ids, dist, c["meas"], c["k"], "max", c["K"], stream)
    return ids, dist


# ------------------------------------------------------------------ what a pass cannot do without

def _mean_query_h(c):
    if c["data"] == "image":
        return 146.0
    if c["kind"] == "pairs":
        return 1.13 * c["doc_h"]
    return (c["qhi"] - c["qlo"]) / math.log(c["qhi"] / c["qlo"]) if c["qhi"] > c["qlo"] else float(c["qhi"])


def work(case):
    """Bytes: the CSR, the used vocabulary's embeddings (or the cost matrix) and the queries read
    once, the results written once.  FLOPs: the distances of the used vocabulary to every query bin
    (2 m each), the transfers of the forward pass (3 per table entry and nonzero) and, for all reverse
    distances, one comparison per document bin and query bin."""
    c = case
    H = c["nq"] * _mean_query_h(c)
    if c["data"] == "image":
        used, nnz, base, dims = GRID * GRID, 146.0 * c["n"], 4.0 * (GRID * GRID) ** 2, 0
    else:
        p = _zipf(c["V"])
        nnz = 1.1 * c["n"] * min(c["doc_h"], c["V"] / 3)
        used = float(np.sum(-np.expm1(-1.13 * c["n"] * _tokens_for(p, min(c["doc_h"], c["V"] / 3)) * p)))
        base, dims = 4.0 * used * c["m"], c["m"]
    k = {"rwmd": 1, "omr": 2, "act": c["k"], "ict": 8}[c["meas"]]
    results = 4.0 * c["nq"] * c["n"] if c["kind"] == "dist" else 12.0 * c["nq"] * c["K"]
    way = c.get("dir", "max" if c["kind"] in ("topk", "serve") else "fwd")
    flops = 2.0 * used * H * dims
    if way != "rev":
        flops += 3.0 * k * nnz * c["nq"]
    if c["kind"] == "dist" and way != "fwd":
        flops += nnz * H
    return {"bytes": 8.0 * nnz + 4.0 * c["n"] + base + 8.0 * H + results, "flops": flops}


# ------------------------------------------------------------------ the same in 64 bits

def _spend(mass, z, cap, meas, k):
    """Cost of moving `mass` along ascending distances z with capacities cap (last dimension)."""
    if meas == "rwmd":
        return mass * z[..., 0]
    if meas == "omr":
        if z.shape[-1] < 2:
            return mass * z[..., 0]
        free = (mass - torch.minimum(mass, cap[..., 0])) * z[..., 1]
        return torch.where(z[..., 0] == 0, free, mass * z[..., 0])
    left, cost = mass.clone(), torch.zeros_like(mass)
    last = z.shape[-1] if meas == "ict" else min(k, z.shape[-1])
    for l in range(last - 1):
        t = torch.minimum(left, cap[..., l])
        cost += t * z[..., l]
        left -= t
        if l % 16 == 15 and not bool((left > 0).any()):
            return cost
    return cost + left * z[..., last - 1]


class _Exact:
    """Distances of one case's histograms in 64 bits, on the GPU."""

    def __init__(self, case, seed):
        self.c = case
        emb, cost, (self.rp, col, val), self.q = _inputs(case, seed)
        ids, inv = torch.unique(col.long(), return_inverse=True)
        self.ids, self.u, self.x = ids, inv, val.double()
        self.own = torch.repeat_interleave(torch.arange(case["n"], device="cuda"), self.rp[1:] - self.rp[:-1])
        self.emb = None if emb is None else emb.double()
        self.cost = None if cost is None else cost.double()
        self.lens = self.rp[1:] - self.rp[:-1]
        if self.emb is not None:
            self.E = self.emb[ids]
            self.E2 = self.E.square().sum(1)

    def query(self, i):
        a, b = int(self.q[0][i]), int(self.q[0][i + 1])
        return self.q[1][a:b].long(), self.q[2][a:b].double()

    def distances(self, idx):
        if self.cost is not None:
            return self.cost[self.ids][:, idx]
        Q = self.emb[idx]
        D = (self.E2[:, None] + Q.square().sum(1)[None] - 2 * self.E @ Q.T).clamp_(min=0).sqrt_()
        return D.masked_fill_(self.ids[:, None] == idx[None], 0.0)

    def forward(self, D, w):
        meas, k = self.c["meas"], self.c["k"]
        width = {"rwmd": 1, "omr": 2, "act": k, "ict": D.shape[1]}[meas]
        z, s = D.topk(min(width, D.shape[1]), dim=1, largest=False, sorted=True)
        cap = w[s]
        if meas != "ict":
            out = torch.empty_like(self.x)
            step = 1 << 25
            for a in range(0, self.x.numel(), step):
                u = self.u[a:a + step]
                out[a:a + step] = _spend(self.x[a:a + step], z[u], cap[u], meas, k)
        else:  # only what still has mass moves on
            out, left, at = torch.zeros_like(self.x), self.x.clone(), torch.arange(self.x.numel(), device="cuda")
            for l in range(z.shape[1]):
                u = self.u[at]
                t = left if l == z.shape[1] - 1 else torch.minimum(left, cap[u, l])
                out[at] += t * z[u, l]
                left = left - t
                keep = left > 0
                at, left = at[keep], left[keep]
                if not at.numel():
                    break
        return torch.zeros(self.c["n"], dtype=torch.float64, device="cuda").index_add_(0, self.own, out)

    def reverse(self, D, w, docs):
        meas, k = self.c["meas"], self.c["k"]
        out = torch.empty(docs.numel(), dtype=torch.float64, device="cuda")
        order = self.lens[docs].argsort()
        a = 0
        while a < docs.numel():
            step = max(1, int(1.5e8 // (int(self.lens[docs[order[min(docs.numel(), a + 4096) - 1]]]) * D.shape[1])))
            sel = order[a:a + min(step, 4096)]
            ln = self.lens[docs[sel]]
            at = torch.arange(int(ln.max()), device="cuda")
            ok = at[None] < ln[:, None]
            e = (self.rp[docs[sel]][:, None] + at[None]).clamp(max=self.x.numel() - 1)
            C = D[self.u[e]].masked_fill_(~ok[:, :, None], math.inf).transpose(1, 2)  # doc, query bin, doc bin
            X = torch.where(ok, self.x[e], 0.0)
            width = {"rwmd": 1, "omr": 2, "act": k, "ict": C.shape[2]}[meas]
            z, s = C.topk(min(width, C.shape[2]), dim=2, largest=False, sorted=True)
            cap = torch.gather(X[:, None].expand(-1, D.shape[1], -1), 2, s)
            mass = w[None].expand(sel.numel(), -1)
            if meas in ("ict", "act"):  # documents shorter than the width end at their own last bin
                last = torch.minimum(ln, torch.tensor(z.shape[2], device="cuda"))
                place = torch.arange(z.shape[2], device="cuda")[None, None]
                cap = torch.where(place == last[:, None, None] - 1, math.inf, cap)
                cap = torch.where(place >= last[:, None, None], 0.0, cap)
                z = torch.where(torch.isinf(z), 0.0, z)
                out[sel] = _spend(mass, torch.cat([z, z[:, :, -1:]], 2), cap, "ict", 0).sum(1)
            elif meas == "omr":  # a document of one bin has no second place to go to
                one = (ln == 1)[:, None]
                first = mass * z[..., 0]
                two = z if z.shape[2] > 1 else torch.cat([z, z], 2)
                two = torch.where(torch.isinf(two), 0.0, two)
                out[sel] = torch.where(one, first, _spend(mass, two, cap, "omr", 0)).sum(1)
            else:
                out[sel] = (mass * z[..., 0]).sum(1)
            a += sel.numel()
        return out

    def nearest(self, D, w, K):
        """The K smallest of max(forward, reverse), reverse values where they can matter."""
        f = self.forward(D, w)
        m = min(self.c["n"], 256)
        while True:
            fs, docs = f.topk(m, largest=False, sorted=True)
            best = torch.maximum(fs, self.reverse(D, w, docs)).topk(K, largest=False, sorted=True).values
            if m == self.c["n"] or float(best[-1]) <= float(fs[-1]):
                return best
            m = min(self.c["n"], 4 * m)


def exact(case, seed):
    c, x = case, _Exact(case, seed)
    if c["kind"] == "pairs":
        F = torch.empty(c["n"], c["n"], dtype=torch.float64, device="cuda")
        A = x.E @ x.E.T
        A = (x.E2[:, None] + x.E2[None] - 2 * A).clamp_(min=0).sqrt_().fill_diagonal_(0.0)
        for i in range(c["n"]):
            a, b = int(x.rp[i]), int(x.rp[i + 1])
            F[i] = x.forward(A[:, x.u[a:b]], x.x[a:b])
        F = torch.maximum(F, F.T).fill_diagonal_(math.inf)
        return None, F.topk(c["K"], dim=1, largest=False, sorted=True).values
    rows = []
    for i in range(c["nq"]):
        idx, w = x.query(i)
        D = x.distances(idx)
        if c["kind"] != "dist":
            rows.append(x.nearest(D, w, c["K"]))
            continue
        f = x.forward(D, w) if c["dir"] != "rev" else None
        r = x.reverse(D, w, torch.arange(c["n"], device="cuda")) if c["dir"] != "fwd" else None
        rows.append(r if f is None else f if r is None else torch.maximum(f, r))
    return torch.stack(rows) if c["kind"] == "dist" else (None, torch.stack(rows))
