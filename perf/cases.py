"""Performance cases of the GB300 re-ranking library.

Each case is one call (or one burst of serving requests) that a user of the
library makes, through ``paper_2012_07620_gb300.rerank.Reranker``:

  run    Algorithm 1 end to end on one query set and one gallery
  knn    the exact top-k neighbour lists alone
  batch  many independent instances in one call
  serve  a burst of requests against a resident gallery

Shapes are those of this repository's workloads (synthetic.py, bench.py) and
of its tests; features are clustered Gaussian embeddings drawn with the same
recipe as synthetic.py (unit centres, noise of norm sigma, optional
distractors uniform on the sphere), generated on the GPU so that drawing them
costs milliseconds.
"""
import math
import random

import torch

from paper_2012_07620_gb300 import rerank

_DEV = "cuda:0"


def _run_case(name, **kw):
    case = dict(kind="run", precision="bf16", dtype="f32", nq=3368, ng=19732, d=2048, clusters=1501, sigma=0.35,
                distractors=2000, k1=26, k2=7, layers=2, aggregator="sum", feature="astar", topk=0, host=False)
    case.update(kw)
    return dict(name=name, **case) if name else case


def listed():
    return [
        # The smallest everyday call: 100 queries against 900 items at the library's default precision;
        # launch latency and the closing synchronisation count.
        _run_case("tiny_fp32", precision="fp32", nq=100, ng=900, d=128, clusters=50, sigma=0.3, distractors=0),
        # A landmark collection: a few dozen queries, 5,000 images, BF16 backbone features as they come from the
        # network, and only the top 100 of each list wanted.
        _run_case("few_queries_top100", dtype="bf16", nq=55, ng=5063, clusters=360, distractors=0, topk=100),
        # Neighbour lists alone on a ragged instance (odd row count, odd width): graph building, deduplication.
        dict(name="knn_ragged", kind="knn", precision="bf16", dtype="f32", n=9973, d=511, clusters=700, sigma=0.35,
             k=30),
        # The headline workload: a person re-identification test set, 3,368 queries and 19,732 gallery images.
        _run_case("market_bf16"),
        # The same set from page-locked host memory, lists back into page-locked host memory.
        _run_case("market_host_bf16", host=True),
        # The same set at the library's default precision.
        _run_case("market_fp32", precision="fp32"),
        # The same set at the lowest similarity precision a caller can choose.
        _run_case("market_fp8", precision="fp8"),
        # Noisy 128-wide features: neighbourhoods of different identities mix, so layers and lists are dense.
        _run_case("market_hard_bf16", d=128, sigma=1.6),
        # Dense initial features (the first column of the paper's ablation): dense layers and final cosines.
        _run_case("market_xfeat_bf16", feature="x"),
        # 50,000 vertices of 512-wide features with complete lists: the largest single call.
        _run_case("large_50k_bf16", nq=5000, ng=45000, d=512, clusters=3000, distractors=0),
        # 64 independent small and middling instances in one call: offline evaluation over many splits or cameras.
        dict(name="batch64_bf16", kind="batch", precision="bf16", dtype="bf16", count=64, n_lo=500, n_hi=8000,
             d_lo=256, d_hi=2048, sigma=0.35, mix=3),
        # Sixteen requests of 1 to 512 queries arriving together at a 40,000-image resident gallery, top 100 each.
        dict(name="serve_burst16", kind="serve", precision="bf16", dtype="bf16", ng=40000, d=2048, clusters=2500,
             sigma=0.35, k1=26, k2=7, layers=2, count=16, q_lo=1, q_hi=512, topk=100, mix=4),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(lo * math.exp(rng.random() * math.log(hi / lo))))))


def _fit(n, d):
    """n, or the largest row count whose similarity costs no more than the largest listed case's."""
    return min(n, int(math.sqrt(1.1e12 / d)))


def _width(rng):
    """Feature widths: the usual backbone sizes, or an odd one between them."""
    return rng.choice([128, 256, 512, 1536, 2048, _log_int(rng, 96, 2048)])


def draw(rng):
    """One more case: kinds, precisions and options as the listed cases have them, sizes over the whole range."""
    kind = rng.choice(["run"] * 7 + ["knn", "batch", "serve"])
    sigma = 0.35
    if kind == "knn":
        d = _width(rng)
        n = _fit(_log_int(rng, 600, 30000), d)
        return dict(kind="knn", precision=rng.choice(["bf16", "bf16", "fp8"]), dtype=rng.choice(["f32", "bf16"]), n=n,
                    d=d, clusters=max(1, round(n / 14.06)), sigma=sigma, k=rng.randint(8, 48))
    if kind == "batch":
        lo = _log_int(rng, 300, 1500)
        hi = _log_int(rng, 2 * lo, 6000)
        return dict(kind="batch", precision="bf16", dtype=rng.choice(["f32", "bf16"]), count=rng.randint(4, 48),
                    n_lo=lo, n_hi=hi, d_lo=rng.choice([128, 256]), d_hi=rng.choice([512, 2048]), sigma=sigma,
                    mix=rng.randrange(1 << 20))
    if kind == "serve":
        ng = _log_int(rng, 4000, 40000)
        return dict(kind="serve", precision="bf16", dtype=rng.choice(["f32", "bf16"]), ng=ng,
                    d=rng.choice([512, 2048]), clusters=ng // 16, sigma=sigma, k1=rng.randint(20, 30),
                    k2=rng.randint(5, 7), layers=rng.randint(1, 2), count=rng.randint(1, 16), q_lo=1, q_hi=512,
                    topk=100, mix=rng.randrange(1 << 20))
    precision = rng.choice(["bf16", "bf16", "bf16", "fp32", "fp8"])
    d = _width(rng)
    n = _fit(_log_int(rng, 400, 45000), d)
    if precision == "fp32":
        n = min(n, 20001)
    nq = max(1, round(n * math.exp(rng.uniform(math.log(0.01), math.log(0.2)))))
    hard = d <= 512 and n <= 20000 and rng.random() < 0.25
    xfeat = n <= 20000 and rng.random() < 0.15
    return _run_case(None, precision=precision, dtype=rng.choice(["f32", "f32", "bf16"]), nq=nq, ng=n - nq, d=d,
                     clusters=max(1, round(n / 14.06)), sigma=round(rng.uniform(1.0, 1.6), 2) if hard else sigma,
                     distractors=rng.choice([0, 0, n // 12]), k1=rng.randint(20, 30), k2=rng.randint(5, 7),
                     layers=rng.randint(1, 3), aggregator=rng.choice(["sum", "sum", "sum", "mean"]),
                     feature="x" if xfeat else "astar", topk=rng.choice([0, 0, min(100, n - nq)]),
                     host=rng.random() < 0.15)


# ---- inputs ----

def _dtype(case):
    return torch.bfloat16 if case["dtype"] == "bf16" else torch.float32


def _unit(x):
    return x / x.norm(dim=1, keepdim=True)


def _centres(clusters, d, gen):
    return _unit(torch.randn(clusters, d, device=_DEV, generator=gen))


def _around(centres, n, sigma, gen):
    """n unit rows, each a random centre plus noise of expected norm sigma."""
    c, d = centres.shape
    label = torch.randint(c, (n,), device=_DEV, generator=gen)
    return _unit(centres[label] + torch.randn(n, d, device=_DEV, generator=gen) * (sigma / math.sqrt(d)))


def _embeddings(case, nq, ng, d, clusters, distractors, gen):
    """(queries, gallery): clustered rows, the gallery's last `distractors` replaced by uniform directions, shuffled."""
    x = _around(_centres(clusters, d, gen), nq + ng, case["sigma"], gen)
    if distractors:
        x[nq + ng - distractors:] = _unit(torch.randn(distractors, d, device=_DEV, generator=gen))
    xg = x[nq:][torch.randperm(ng, device=_DEV, generator=gen)]
    return x[:nq].to(_dtype(case)).contiguous(), xg.to(_dtype(case)).contiguous()


def _generator(seed):
    g = torch.Generator(device=_DEV)
    g.manual_seed(int(seed))
    return g


def _batch_shapes(case):
    """Sizes and parameters of a batch's instances; they belong to the case, not to the inputs."""
    rng = random.Random(case["mix"])
    dims = [d for d in (128, 256, 512, 2048) if case["d_lo"] <= d <= case["d_hi"]]
    out = []
    for _ in range(case["count"]):
        n = _log_int(rng, case["n_lo"], case["n_hi"])
        nq = round(0.146 * n)
        out.append(dict(nq=nq, ng=n - nq, d=rng.choice(dims), clusters=max(1, round(n / 14.06)),
                        k1=rng.randint(20, 30), k2=rng.randint(5, 7), layers=rng.randint(1, 3)))
    return out


def _request_sizes(case):
    rng = random.Random(case["mix"])
    return [_log_int(rng, case["q_lo"], case["q_hi"]) for _ in range(case["count"])]


def _inputs(case, seed):
    """The features of a case: what both prepare() and exact() start from."""
    gen = _generator(seed)
    kind = case["kind"]
    if kind == "run":
        return _embeddings(case, case["nq"], case["ng"], case["d"], case["clusters"], case["distractors"], gen)
    if kind == "knn":
        return _around(_centres(case["clusters"], case["d"], gen), case["n"], case["sigma"], gen).to(_dtype(case))
    if kind == "batch":
        return [(s, *_embeddings(case, s["nq"], s["ng"], s["d"], s["clusters"], 0, gen)) for s in _batch_shapes(case)]
    centres = _centres(case["clusters"], case["d"], gen)
    xg = _around(centres, case["ng"], case["sigma"], gen).to(_dtype(case))
    return xg, [_around(centres, q, case["sigma"], gen).to(_dtype(case)) for q in _request_sizes(case)]


def prepare(case, seed):
    kind = case["kind"]
    data = _inputs(case, seed)
    if kind == "run":
        R = rerank.Reranker(device=0, precision=case["precision"], aggregator=case["aggregator"],
                            feature=case["feature"])
        xq, xg = data
        out = (None, None)
        if case["host"]:  # page-locked buffers that the caller's program reuses
            shape = (case["nq"], case["topk"] or case["ng"])
            xq, xg = xq.cpu().pin_memory(), xg.cpu().pin_memory()
            out = (torch.zeros(shape, dtype=torch.int32, pin_memory=True),
                   torch.zeros(shape, dtype=torch.float32, pin_memory=True))
        return dict(case=case, R=R, xq=xq, xg=xg, out=out)
    R = rerank.Reranker(device=0, precision=case["precision"])
    if kind == "knn":
        return dict(case=case, R=R, x=data)
    if kind == "batch":
        # One buffer holds every instance's lists, each on a 512-byte boundary.
        place, total = [], 0
        for s, _, _ in data:
            place.append(total)
            total += (s["nq"] * s["ng"] + 127) // 128 * 128
        idx = torch.zeros(total, dtype=torch.int32, device=_DEV)
        dist = torch.zeros(total, dtype=torch.float32, device=_DEV)
        jobs = []
        for (s, xq, xg), at in zip(data, place):
            span = slice(at, at + s["nq"] * s["ng"])
            jobs.append(dict(xq=xq, xg=xg, k1=s["k1"], k2=s["k2"], layers=s["layers"],
                             out_idx=idx[span].view(s["nq"], s["ng"]), out_dist=dist[span].view(s["nq"], s["ng"])))
        return dict(case=case, R=R, jobs=jobs, idx=idx, dist=dist)
    xg, requests = data
    R.load_gallery(xg, max_query=512, k1=case["k1"], k2=case["k2"], layers=case["layers"])
    return dict(case=case, R=R, requests=requests)


def run(state):
    case, R = state["case"], state["R"]
    kind = case["kind"]
    if kind == "run":
        return R.run(state["xq"], state["xg"], case["k1"], case["k2"], case["layers"], case["topk"],
                     out_idx=state["out"][0], out_dist=state["out"][1])
    if kind == "knn":
        return R.knn(state["x"], case["k"])
    if kind == "batch":
        R.run_batch(state["jobs"])
        return state["idx"], state["dist"]
    pending = [R.submit(q, case["topk"]) for q in state["requests"]]
    for ticket, _, _ in pending:
        R.wait(ticket)
    return [(idx, dist) for _, idx, dist in pending]


# ---- work ----

def _rank_work(nq, ng, d, esize, layers, k2, k1, topk, new_rows=None):
    """One instance: features read once, lists written once; every unordered pair's dot product once (a request
    needs only the pairs that its own queries are in)."""
    n = nq + ng
    pairs = n * n / 2 if new_rows is None else new_rows * n
    return ((n if new_rows is None else new_rows) * d * esize + nq * (topk or ng) * 8,
            2.0 * pairs * d + 2.0 * layers * n * (k2 + 1) * k1)


def work(case):
    es = 2 if case["dtype"] == "bf16" else 4
    kind = case["kind"]
    if kind == "run":
        b, f = _rank_work(case["nq"], case["ng"], case["d"], es, case["layers"], case["k2"], case["k1"], case["topk"])
        if case["feature"] == "x":
            f += 2.0 * case["nq"] * case["ng"] * case["d"]
    elif kind == "knn":
        b, f = case["n"] * case["d"] * es + case["n"] * case["k"] * 8, float(case["n"]) ** 2 * case["d"]
    elif kind == "batch":
        parts = [_rank_work(s["nq"], s["ng"], s["d"], es, s["layers"], s["k2"], s["k1"], 0)
                 for s in _batch_shapes(case)]
        b, f = sum(p[0] for p in parts), sum(p[1] for p in parts)
    else:
        # The gallery is scored against every request's queries: read once for the burst.
        parts = [_rank_work(q, case["ng"], case["d"], es, case["layers"], case["k2"], case["k1"], case["topk"],
                            new_rows=q) for q in _request_sizes(case)]
        b, f = case["ng"] * case["d"] * es + sum(p[0] for p in parts), sum(p[1] for p in parts)
    return {"bytes": float(b), "flops": float(f)}


# ---- the same results in 64 bits ----

def _exact_knn(x, k, rows=None, chunk=2048):
    """Top-k of each row of the cosine matrix in float64, self counted as exactly 1 and first."""
    x = x.double()
    x = x / x.norm(dim=1, keepdim=True)
    n = x.shape[0]
    rows = torch.arange(n, device=x.device) if rows is None else rows
    idx, val = [], []
    for a in range(0, rows.numel(), chunk):
        r = rows[a:a + chunk]
        s = x[r] @ x.T
        at = torch.arange(r.numel(), device=x.device)
        s[at, r] = 2.0
        v, i = s.topk(k, dim=1)
        idx.append(i)
        val.append(torch.where(i == r[:, None], torch.ones_like(v), v))
    return torch.cat(idx), torch.cat(val)


def _exact_ranking(x, nq, knn, score, k2, layers, aggregator, feature, topk):
    """Distances of every query's list, ascending, from the neighbour lists (float64)."""
    n, k1 = knn.shape
    if feature == "x":
        h = x.double()
        h = h / h.norm(dim=1, keepdim=True)
    else:
        h = torch.zeros(n, n, dtype=torch.float64, device=x.device)
        h.scatter_(1, knn, 0.5)
        for a in range(0, n, 4096):  # + A^T / 2, by the targets of each slice of rows
            r = torch.arange(a, min(n, a + 4096), device=x.device).repeat_interleave(k1)
            h.index_put_((knn[a:a + 4096].reshape(-1), r), torch.tensor(0.5, dtype=torch.float64, device=x.device),
                         accumulate=True)
    w = score[:, :k2] ** 2
    if aggregator == "mean":
        w = w / k2
    for _ in range(layers):
        new = torch.empty_like(h)
        for a in range(0, n, 4096):
            t = h[a:a + 4096].clone()
            for m in range(k2):
                t.addcmul_(h[knn[a:a + 4096, m]], w[a:a + 4096, m:m + 1])
            new[a:a + 4096] = t / t.norm(dim=1, keepdim=True)
        h = new
    h /= h.norm(dim=1, keepdim=True)
    out = []
    hg = h[nq:]
    for a in range(0, nq, 1024):
        q = h[a:min(nq, a + 1024)]
        if feature == "x":
            s = q @ hg.T
        else:  # only the columns that the queries use
            s = torch.zeros(q.shape[0], hg.shape[0], dtype=torch.float64, device=x.device)
            for b in range(0, q.shape[0], 128):
                p = q[b:b + 128]
                cols = (p != 0).any(dim=0).nonzero().reshape(-1)
                s[b:b + 128] = p[:, cols] @ hg[:, cols].T
        out.append((1.0 - s).sort(dim=1).values[:, :topk] if topk else (1.0 - s).sort(dim=1).values)
    return torch.cat(out)


def _exact_run(xq, xg, c, topk, lists=None):
    x = torch.cat([xq, xg])
    knn, score = _exact_knn(x, c["k1"]) if lists is None else lists
    return _exact_ranking(x, xq.shape[0], knn, score, c["k2"], c["layers"], c.get("aggregator", "sum"),
                          c.get("feature", "astar"), topk)


def exact(case, seed):
    kind = case["kind"]
    data = _inputs(case, seed)
    if kind == "run":
        return None, _exact_run(*data, case, case["topk"])
    if kind == "knn":
        return None, _exact_knn(data, case["k"])[1]
    if kind == "batch":
        flat = []
        for s, xq, xg in data:
            d = _exact_run(xq, xg, s, 0).reshape(-1)
            flat.append(torch.cat([d, d.new_zeros(-d.numel() % 128)]))
        return None, torch.cat(flat)
    if case["ng"] * case["count"] > 200000:  # one full-size 64-bit graph per request: too long for a large burst
        return None
    xg, requests = data
    return [(None, _exact_run(q, xg, case, case["topk"])) for q in requests]
