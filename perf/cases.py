"""Performance cases of the AdANNS library: what a user has it do, through its
public entry points, on seeded synthetic Matryoshka-like embeddings.

A case is a dict of plain values; `prepare` makes its inputs on the GPU from
the seed alone, `run` is one pass through the library, `exact` the same result
in 64 bits from plain torch.  The embeddings follow the generative model of
`synthdata` (Gaussian mixture, per-dimension scale (j + 1) ** -0.5, spread 0.5
within a component), drawn on the GPU.  Kinds of case:

  ivf      search_ivf: cluster mapping at d_c, list scan at d_s, top-k, in the
           FP32 tier or in BF16 / FP8 storage with the exact rerank
  budgets  search_ivf_budgets: every query with its own d_s, nprobe and k
  opq      search_ivfopq: ADC scan of OPQ codes (one list: exhaustive OPQ),
           optionally with the exact rerank
  graph    graph_search: low-d graph shortlist, high-d rerank
  kmeans   one Lloyd step of the index build: kmeans_assign + kmeans_update
  encode   opq_encode: rotation and nearest codewords of a block of rows
"""
from __future__ import annotations

import math

import torch

import paper_2305_19435_gb300 as P

TIERS = {"f32": P.STORE_F32, "bf16": P.STORE_BF16, "fp8": P.STORE_FP8}
BYTES = {"f32": 4, "bf16": 2, "fp8": 1}
METRICS = {"prefixnorm": P.METRIC_L2_PREFIXNORM, "l2": P.METRIC_L2}
IMAGENET_N = 1_281_167
SPREAD = 0.5
BLOCK = 1 << 18  # rows drawn at a time


# ------------------------------------------------------------------ the cases
def _ivf(N, d, K, nlist, B, d_c, d_s, nprobe, k, tier="f32", rerank=0, metric="prefixnorm"):
    return {"kind": "ivf", "N": N, "d": d, "K": K, "nlist": nlist, "B": B,
            "d_c": d_c, "d_s": d_s, "nprobe": nprobe, "k": k, "tier": tier, "rerank": rerank,
            "metric": metric}


def listed():
    return [
        # the smallest workload of the tests (10,000 x 64, 200 queries): a call
        # whose launches weigh as much as its work
        {"name": "tiny_f32"} | _ivf(10_000, 64, 64, 64, 200, 16, 64, 4, 10),
        # one user's query against the ImageNet-shaped index, exact FP32
        {"name": "online_f32"} | _ivf(IMAGENET_N, 2048, 1000, 1024, 1, 32, 512, 16, 100),
        # a packed serving batch: requests that each bring their own d_s,
        # nprobe and k to one resident index
        {"name": "serving_budgets_f32", "kind": "budgets", "N": IMAGENET_N, "d": 2048, "K": 1000,
         "nlist": 1024, "B": 1021, "d_c": 32, "d_s_max": 512, "nprobe_max": 16, "k": 100},
        # the ImageNet-shaped evaluation (50,000 queries) in the exact FP32 tier
        {"name": "bulk_f32"} | _ivf(IMAGENET_N, 2048, 1000, 1024, 50_000, 32, 512, 16, 100),
        # the same evaluation in the BF16 tier with the exact rerank of 4k: the
        # benchmark's own step
        {"name": "bulk_bf16"} | _ivf(IMAGENET_N, 2048, 1000, 1024, 50_000, 32, 512, 16, 100, "bf16", 400),
        # a serving-sized batch at the full 2048 coordinates, few queries per
        # probed list: the list scan streams the database
        {"name": "stream_bf16"} | _ivf(IMAGENET_N, 2048, 1000, 1024, 2048, 32, 2048, 1, 10, "bf16", 40),
        # the FP8 tier at a longer prefix, a ragged mid-sized batch
        {"name": "mid_fp8"} | _ivf(IMAGENET_N, 2048, 1000, 1024, 10_007, 64, 1024, 8, 10, "fp8", 40),
        # IVF-OPQ of NQ-shaped passages (a quarter of its rows and lists, so
        # lists keep their length): 32-byte codes of the 384 prefix, rerank of 4k
        {"name": "nq_ivfopq", "kind": "opq", "N": 5_253_831, "d": 768, "K": 1024, "nlist": 1024,
         "B": 8000, "d_c": 64, "d_s": 384, "M": 32, "nprobe": 32, "k": 100, "rerank": 400},
        # exhaustive OPQ: 16-byte codes of the 128 prefix, every row of the
        # ImageNet-shaped database scored for each query
        {"name": "flat_opq", "kind": "opq", "N": IMAGENET_N, "d": 2048, "K": 1000, "nlist": 1,
         "B": 1000, "d_c": 8, "d_s": 128, "M": 16, "nprobe": 1, "k": 10, "rerank": 0},
        # graph shortlist at 16 coordinates, rerank at 512
        {"name": "graph_rerank", "kind": "graph", "N": 262_144, "d": 2048, "K": 1000, "B": 10_000,
         "d_g": 16, "cand": 64, "R": 32, "L": 64, "d_s": 512, "k": 10, "rerank": 40},
        # the build's inner step: one Lloyd iteration on the training sample
        # (256 rows per list) at the clustering prefix
        {"name": "kmeans_step", "kind": "kmeans", "n": 262_144, "d": 2048, "K": 1000, "nc": 1024,
         "dim": 32, "metric": "prefixnorm"},
        # the build's encode step: OPQ codes of a block of database rows
        {"name": "opq_encode", "kind": "encode", "n": 262_144, "d": 768, "K": 1024, "d_s": 384,
         "M": 32, "metric": "prefixnorm"},
    ]


_MOST = 50_000 * 16 * (IMAGENET_N / 1024) * 512.0  # (query, member) coordinates of the largest


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges: sizes log-uniform, mostly odd."""
    kind = rng.choice(["ivf", "ivf", "ivf", "ivf", "budgets", "opq", "opq", "graph", "kmeans",
                       "encode"])
    if kind in ("ivf", "budgets"):
        d = rng.choice([64, 256, 768, 2048])
        N = _log_int(rng, 10_000, IMAGENET_N)
        nlist = min(1024, max(16, _log_int(rng, N // 2500 + 1, N // 150)))
        d_c = rng.choice([16, 32, 64])
        K = min(1000, max(16, nlist))
        if kind == "budgets":
            return {"kind": kind, "N": N, "d": d, "K": K, "nlist": nlist,
                    "B": _log_int(rng, 1, 2048), "d_c": d_c, "d_s_max": min(d, 512),
                    "nprobe_max": min(16, nlist), "k": _log_int(rng, 1, 100)}
        d_s = rng.choice([x for x in (64, 96, 128, 256, 512, 768, 1024, 2048) if x <= d])
        nprobe = min(nlist, _log_int(rng, 1, 32))
        B = _log_int(rng, 1, 50_000)
        B = max(1, min(B, int(_MOST / (nprobe * (N / nlist) * d_s))))
        k = _log_int(rng, 1, 100)
        tier = rng.choice(["f32", "f32", "bf16", "fp8"])
        if tier == "f32":
            metric = "l2" if rng.random() < 0.2 else "prefixnorm"
            return _ivf(N, d, K, nlist, B, d_c, d_s, nprobe, k, metric=metric)
        return _ivf(N, d, K, nlist, B, d_c, d_s, nprobe, k, tier, 4 * k)
    if kind == "opq":
        d_s, M = rng.choice([(64, 8), (128, 16), (192, 16), (128, 32), (384, 32), (768, 64)])
        if rng.random() < 0.3:  # exhaustive
            N = _log_int(rng, 50_000, IMAGENET_N)
            return {"kind": kind, "N": N, "d": 768, "K": 1000, "nlist": 1,
                    "B": _log_int(rng, 1, 1000), "d_c": 8, "d_s": d_s, "M": M, "nprobe": 1,
                    "k": _log_int(rng, 1, 100), "rerank": 0}
        N = _log_int(rng, 50_000, 3_000_000)
        k = _log_int(rng, 1, 100)
        nlist = min(1024, max(64, N // 2000))
        return {"kind": kind, "N": N, "d": 768, "K": 1024, "nlist": nlist,
                "B": _log_int(rng, 1, 8000), "d_c": rng.choice([32, 64]), "d_s": d_s, "M": M,
                "nprobe": _log_int(rng, 1, 64), "k": k, "rerank": rng.choice([0, 4 * k])}
    if kind == "graph":
        L = rng.choice([32, 64, 128])
        return {"kind": kind, "N": _log_int(rng, 20_000, 262_144), "d": rng.choice([768, 2048]),
                "K": 1000, "B": _log_int(rng, 1, 10_000), "d_g": rng.choice([16, 32]), "cand": 64,
                "R": 32, "L": L, "d_s": rng.choice([256, 512, 768]), "k": 10,
                "rerank": rng.choice([10, L // 2, L])}
    n = _log_int(rng, 20_000, 262_144)
    metric = "l2" if rng.random() < 0.2 else "prefixnorm"
    if kind == "kmeans":
        return {"kind": kind, "n": n, "d": rng.choice([64, 768, 2048]), "K": 1000,
                "nc": _log_int(rng, 64, 4096), "dim": rng.choice([16, 32, 64]), "metric": metric}
    d_s, M = rng.choice([(64, 8), (128, 16), (192, 16), (384, 32), (768, 64)])
    return {"kind": kind, "n": n, "d": rng.choice([768, 2048]), "K": 1024, "d_s": d_s, "M": M,
            "metric": metric}


# ------------------------------------------------------------------ the inputs
def _gen(seed, stream):
    return torch.Generator(device="cuda").manual_seed(1_000_003 * int(seed) + stream)


def _scale(d):
    return (torch.arange(d, device="cuda", dtype=torch.float32) + 1.0) ** -0.5


def _means(case, seed):
    return torch.randn(case["K"], case["d"], device="cuda",
                       generator=_gen(seed, 1)) * _scale(case["d"])


def _points(n, means, seed, stream):
    """n rows of the mixture, FP32 [n, d]."""
    g, d = _gen(seed, stream), means.shape[1]
    lab = torch.randint(means.shape[0], (n,), device="cuda", generator=g)
    x, spread = torch.empty(n, d, device="cuda"), SPREAD * _scale(d)
    for lo in range(0, n, BLOCK):
        part = x[lo:lo + BLOCK]
        part.normal_(generator=g)
        part.mul_(spread).add_(means[lab[lo:lo + BLOCK]])
    return x


def _rep(x, m, metric):
    """The m-prefix as a representation (normalised at its own length unless raw L2)."""
    x = x[:, :m]
    if metric == "l2":
        return x
    n = x.norm(dim=1, keepdim=True)
    return torch.where(n > 0, x / n, torch.zeros_like(x))


def _nearest(x, cent):
    """Nearest row of cent for every row of x, in row blocks."""
    half = 0.5 * (cent * cent).sum(1)
    out = torch.empty(x.shape[0], dtype=torch.int64, device="cuda")
    rows = max(1024, (1 << 27) // cent.shape[0])
    for lo in range(0, x.shape[0], rows):
        out[lo:lo + rows] = (half - x[lo:lo + rows] @ cent.T).argmin(1)
    return out


def _lloyd(x, cent, steps):
    """A few Lloyd steps in torch, the means as one-hot products (the same bits every time)."""
    for _ in range(steps):
        hot = torch.nn.functional.one_hot(_nearest(x, cent), cent.shape[0]).to(torch.float32)
        cnt = hot.sum(0).unsqueeze(1)
        cent = torch.where(cnt > 0, (hot.T @ x) / cnt.clamp(min=1), cent)
    return cent.contiguous()


def _database(case, seed):
    """Rows, centroids and list assignment of an IVF case: lists of a k-means
    clustering at d_c, as a program has them once its index is formed."""
    db = _points(case["N"], _means(case, seed), seed, 2)
    if case["nlist"] == 1:
        return (db, torch.zeros(1, case["d_c"], device="cuda"),
                torch.zeros(case["N"], dtype=torch.int32, device="cuda"))
    metric = case.get("metric", "prefixnorm")
    pick = torch.randperm(case["N"], device="cuda", generator=_gen(seed, 3))
    sample = _rep(db[pick[:16 * case["nlist"]]], case["d_c"], metric)
    cent = _lloyd(sample, sample[:case["nlist"]].clone(), 3)
    assign = torch.empty(case["N"], dtype=torch.int32, device="cuda")
    for lo in range(0, case["N"], BLOCK):
        assign[lo:lo + BLOCK] = _nearest(_rep(db[lo:lo + BLOCK], case["d_c"], metric), cent).int()
    return db, cent, assign


def _queries(case, seed):
    return _points(case["B"], _means(case, seed), seed, 4)


def _budgets(case, seed):
    """(d_s, nprobe, k) per query: a program's host-side lists."""
    g = torch.Generator().manual_seed(int(seed) + 5)
    grid = [x for x in (64, 128, 256, 512) if x <= case["d_s_max"]]
    B = case["B"]
    ds = torch.tensor(grid)[torch.randint(len(grid), (B,), generator=g)]
    npr = torch.randint(1, case["nprobe_max"] + 1, (B,), generator=g)
    k = torch.randint(1, case["k"] + 1, (B,), generator=g)
    k[0] = case["k"]
    return ds.tolist(), npr.tolist(), k.tolist()


def _opq(x, case, seed, metric="prefixnorm"):
    """A rotation and codebooks for rows like x (an orthonormal matrix and a
    few Lloyd steps per sub-vector on a sample)."""
    d_s, M = case["d_s"], case["M"]
    R = torch.linalg.qr(torch.randn(d_s, d_s, device="cuda", generator=_gen(seed, 6),
                                    dtype=torch.float64))[0].float().contiguous()
    z = _rep(x[:8192], d_s, metric) @ R
    w = d_s // M
    books = [_lloyd(z[:, m * w:(m + 1) * w].contiguous(), z[:256, m * w:(m + 1) * w].clone(), 2)
             for m in range(M)]
    return R, torch.stack(books).contiguous()


def _codes(x, case, R, books):
    """Codes by row, in torch."""
    d_s, M, n = case["d_s"], case["M"], x.shape[0]
    w = d_s // M
    out = torch.empty(n, M, dtype=torch.uint8, device="cuda")
    half = 0.5 * (books * books).sum(2).unsqueeze(1)  # [M, 1, 256]
    for lo in range(0, n, 1 << 17):
        z = _rep(x[lo:lo + (1 << 17)], d_s, "prefixnorm") @ R
        z = z.reshape(-1, M, w).transpose(0, 1)
        out[lo:lo + z.shape[1]] = torch.baddbmm(half, z, books.transpose(1, 2),
                                                alpha=-1).argmin(2).T.to(torch.uint8)
    return out


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("ivf", "budgets"):
        db, cent, assign = _database(case, seed)
        store = P.STORE_F32 | TIERS[case.get("tier", "f32")]
        metric = METRICS[case.get("metric", "prefixnorm")]
        state = {"case": case, "q": _queries(case, seed),
                 "index": P.index_create(db, cent, assign, metric=metric, storage=store)}
        if kind == "budgets":
            state["budgets"] = _budgets(case, seed)
        return state
    if kind == "opq":
        db, cent, assign = _database(case, seed)
        R, books = _opq(db, case, seed)
        index = P.index_create(db, cent, assign)
        P.set_opq(index, case["d_s"], case["M"], R, books, _codes(db, case, R, books))
        return {"case": case, "q": _queries(case, seed), "index": index}
    if kind == "graph":
        db = _points(case["N"], _means(case, seed), seed, 2)
        return {"case": case, "q": _queries(case, seed),
                "graph": P.graph_build(db, case["d_g"], case["cand"], case["R"], 1.2)}
    x = _points(case["n"], _means(case, seed), seed, 2)
    if kind == "kmeans":
        return {"case": case, "x": x,
                "cent": _rep(x[:case["nc"]], case["dim"], case["metric"]).contiguous()}
    R, books = _opq(x, case, seed, case["metric"])
    return {"case": case, "x": x, "R": R, "books": books}


# -------------------------------------------------------------------- one pass
def run(state):
    c = state["case"]
    kind = c["kind"]
    if kind == "ivf":
        return P.search_ivf(state["index"], state["q"], c["d_c"], c["d_s"], c["nprobe"], c["k"],
                            storage=TIERS[c["tier"]], rerank_k=c["rerank"])
    if kind == "budgets":
        ds, npr, k = state["budgets"]
        return P.search_ivf_budgets(state["index"], state["q"], c["d_c"], ds, npr, k)
    if kind == "opq":
        return P.search_ivfopq(state["index"], state["q"], c["d_c"], c["nprobe"], c["k"],
                               rerank_k=c["rerank"])
    if kind == "graph":
        return P.graph_search(state["graph"], state["q"], c["L"], c["d_s"], c["k"], c["rerank"])
    if kind == "kmeans":
        assign, dist = P.kmeans_assign(state["x"], state["cent"], c["dim"],
                                       metric=METRICS[c["metric"]])
        cent = P.kmeans_update(state["x"], assign, state["cent"].clone(), c["dim"],
                               metric=METRICS[c["metric"]])
        return assign, dist, cent
    return P.opq_encode(state["x"], c["d_s"], c["M"], state["R"], state["books"],
                        metric=METRICS[c["metric"]])


# ------------------------------------------------------------ its least work
def work(case):
    """Unique bytes and arithmetic of one pass (lists taken as equally long and
    equally popular; a rerank re-scores at least the k returned rows)."""
    kind = case["kind"]
    if kind in ("kmeans", "encode"):
        n = case["n"]
        if kind == "kmeans":
            dim, nc = case["dim"], case["nc"]
            return {"bytes": 4.0 * (2 * n * dim + 2 * nc * dim + 3 * n),
                    "flops": 2.0 * n * nc * dim + n * dim}
        d_s, M = case["d_s"], case["M"]
        return {"bytes": 4.0 * (n * d_s + d_s * d_s + 256 * d_s) + n * M,
                "flops": 2.0 * n * d_s * d_s + 2.0 * n * 256 * d_s}
    B, k = case["B"], case["k"]
    if kind == "graph":
        # every query expands at least rerank entries, each with R neighbours
        seen = case["rerank"] * case["R"]
        rows = min(float(case["N"]), float(B) * seen)
        return {"bytes": rows * 4 * (case["d_g"] + case["R"]) + 4.0 * B * case["d_s"]
                + min(case["N"], B * case["rerank"]) * 4.0 * case["d_s"] + 12.0 * B * k,
                "flops": 2.0 * B * (seen * case["d_g"] + case["rerank"] * case["d_s"])}
    nlist, per = case["nlist"], case["N"] / case["nlist"]
    nprobe, d_s = case.get("nprobe"), case.get("d_s")
    if kind == "budgets":
        grid = [x for x in (64, 128, 256, 512) if x <= case["d_s_max"]]
        nprobe, d_s = (1 + case["nprobe_max"]) / 2, sum(grid) / len(grid)
    lists = nlist * (1 - (1 - 1 / nlist) ** (B * nprobe))
    coarse = 2.0 * B * nlist * case["d_c"] if nlist > 1 else 0.0
    out = 12.0 * B * k + 4.0 * B * max(d_s, case["d_c"]) + 4.0 * nlist * case["d_c"]
    if kind == "opq":
        r = max(case["rerank"] and k, 0)
        return {"bytes": out + lists * per * case["M"] + min(case["N"], B * r) * 4.0 * d_s,
                "flops": coarse + B * nprobe * per * case["M"] + 2.0 * B * (d_s * d_s + 256 * d_s)
                + 2.0 * B * r * d_s}
    tier = case.get("tier", "f32")
    r = 0 if tier == "f32" else k
    return {"bytes": out + lists * per * d_s * BYTES[tier] + min(case["N"], B * r) * 4.0 * d_s,
            "flops": coarse + 2.0 * B * nprobe * per * d_s + 2.0 * B * r * d_s}


# ------------------------------------------------------------- in 64 bits
def _pair_dist(q, x):
    return ((q * q).sum(1, keepdim=True) + (x * x).sum(1) - 2.0 * (q @ x.T)).clamp(min=0)


def _probes(case, q, cent, nprobe):
    metric = case.get("metric", "prefixnorm")
    d = _pair_dist(_rep(q[:, :case["d_c"]].double(), case["d_c"], metric), cent.double())
    return d.topk(nprobe, dim=1, largest=False, sorted=True)[1]


def _scan(assign, probes, score, B, k, nlist):
    """The k smallest scores of every query over the members of its probed
    lists (probes -1: none), with their rows; score(queries, rows) -> fp64."""
    nprobe = probes.shape[1]
    best = torch.full((B, nprobe, k), math.inf, device="cuda", dtype=torch.float64)
    row = torch.full((B, nprobe, k), -1, device="cuda", dtype=torch.int64)
    members = torch.sort(assign.long(), stable=True)[1]
    ends = torch.bincount(assign.long(), minlength=nlist).cumsum(0).tolist()
    flat = probes.reshape(-1)
    order = torch.sort(flat, stable=True)[1]
    skip = int((flat < 0).sum())
    stops = (skip + torch.bincount(flat[flat >= 0], minlength=nlist).cumsum(0)).tolist()
    for c in range(nlist):
        lo, a = (ends[c - 1] if c else 0), (stops[c - 1] if c else skip)
        rows, slots = members[lo:ends[c]], order[a:stops[c]]
        if not len(rows) or not len(slots):
            continue
        step = max(1, (1 << 28) // len(rows))
        for s in range(0, len(slots), step):
            part = slots[s:s + step]
            v, at = score(part // nprobe, rows).topk(min(k, len(rows)), dim=1, largest=False)
            best.view(-1, k)[part, :v.shape[1]] = v
            row.view(-1, k)[part, :v.shape[1]] = rows[at]
    v, at = best.view(B, -1).topk(k, dim=1, largest=False, sorted=True)
    return v, row.view(B, -1).gather(1, at)


def _exact_ivf(case, q, db, cent, assign):
    metric, d_s = case.get("metric", "prefixnorm"), case["d_s"]
    qr = _rep(q[:, :d_s].double(), d_s, metric)

    def score(qs, rows):
        return _pair_dist(qr[qs], _rep(db[rows, :d_s].double(), d_s, metric))

    return _scan(assign, _probes(case, q, cent, case["nprobe"]), score, case["B"], case["k"],
                 case["nlist"])[0]


def _exact_budgets(case, q, db, cent, assign, seed):
    ds, npr, k = (torch.tensor(v, device="cuda") for v in _budgets(case, seed))
    probes = _probes(case, q, cent, case["nprobe_max"])
    probes[torch.arange(probes.shape[1], device="cuda") >= npr.unsqueeze(1)] = -1
    out = torch.full((case["B"], case["k"]), math.inf, device="cuda", dtype=torch.float64)
    for d_s in sorted(set(ds.tolist())):
        at = (ds == d_s).nonzero().flatten()
        qr = _rep(q[at, :d_s].double(), d_s, "prefixnorm")

        def score(qs, rows, qr=qr, d_s=d_s):
            return _pair_dist(qr[qs], _rep(db[rows, :d_s].double(), d_s, "prefixnorm"))

        out[at] = _scan(assign, probes[at], score, len(at), case["k"], case["nlist"])[0]
    out[torch.arange(case["k"], device="cuda") >= k.unsqueeze(1)] = math.inf
    return out


def _exact_opq(case, q, db, cent, assign, seed):
    d_s, M, k = case["d_s"], case["M"], case["k"]
    R, books = _opq(db, case, seed)
    codes = _codes(db, case, R, books).long()
    cb, w = books.double(), d_s // M
    z = _rep(q[:, :d_s].double(), d_s, "prefixnorm") @ R.double()

    def score(qs, rows):  # |z - decode(code)|^2 through the decoded rows
        parts = []
        for lo in range(0, len(rows), 1 << 16):
            y = torch.cat([cb[m][codes[rows[lo:lo + (1 << 16)], m]] for m in range(M)], 1)
            parts.append(_pair_dist(z[qs], y))
        return torch.cat(parts, 1)

    keep = max(case["rerank"], k)
    v, rows = _scan(assign, _probes(case, q, cent, case["nprobe"]), score, case["B"], keep,
                    case["nlist"])
    if not case["rerank"]:
        return v
    qr = _rep(q[:, :d_s].double(), d_s, "prefixnorm")
    for lo in range(0, case["B"], 64):
        x = db[rows[lo:lo + 64].clamp(min=0).reshape(-1), :d_s].double()
        x = _rep(x, d_s, "prefixnorm").view(-1, keep, d_s)
        dist = (x - qr[lo:lo + 64].unsqueeze(1)).square().sum(2)
        v[lo:lo + 64] = dist.masked_fill(rows[lo:lo + 64] < 0, math.inf)
    return v.topk(k, dim=1, largest=False, sorted=True)[0]


def exact(case, seed):
    kind = case["kind"]
    if kind in ("graph", "encode"):  # a traversal's order and code bytes
        return None
    if kind == "kmeans":
        x = _points(case["n"], _means(case, seed), seed, 2)
        dim, metric = case["dim"], case["metric"]
        cent = _rep(x[:case["nc"]], dim, metric).contiguous().double()
        x = _rep(x[:, :dim].double(), dim, metric)
        dist = torch.empty(case["n"], device="cuda", dtype=torch.float64)
        assign = torch.empty(case["n"], device="cuda", dtype=torch.int64)
        for lo in range(0, case["n"], 1 << 15):
            dist[lo:lo + (1 << 15)], assign[lo:lo + (1 << 15)] = \
                _pair_dist(x[lo:lo + (1 << 15)], cent).min(1)
        cnt = torch.bincount(assign, minlength=case["nc"]).unsqueeze(1)
        mean = torch.zeros_like(cent).index_add_(0, assign, x) / cnt.clamp(min=1)
        return None, dist, torch.where(cnt > 0, mean, cent)
    db, cent, assign = _database(case, seed)
    q = _queries(case, seed)
    if kind == "budgets":
        return None, _exact_budgets(case, q, db, cent, assign, seed)
    if kind == "opq":
        return None, _exact_opq(case, q, db, cent, assign, seed)
    return None, _exact_ivf(case, q, db, cent, assign)
