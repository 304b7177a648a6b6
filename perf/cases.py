"""Timed cases of the streaming IVF-Flat index: what a program has it do.

Every case is one pass through the package's public calls (``Index.search``,
``add``, ``remove``, ``train`` and the recorded queue of ``executor``) on an
index of seeded synthetic vectors.  Sizes are those of the package's own
workloads (``workloads.CONFIGS``) or odd ones between them.

Inputs are drawn on the GPU from the seed alone:

* ``sift``: mixture of ``comps`` centers U[0, 255]^d, sigma 20, rounded and
  clipped to [0, 255] (SIFT-like descriptors);
* ``box``: centers U[-1, 1]^d, sigma 0.1 (generic embeddings);
* ``sphere``: unit centers, sigma 0.02, rows normalised (Deep-like).

The quantizer is the first ``lists`` mixture centers; with more lists than
centers it is a sample of the vectors' own distribution, as an untrained
quantizer would be.  ``zipf`` draws the component of rank r with probability
proportional to 1 / r.
"""
import math

import numpy as np
import torch

from paper_2601_11808_gb300.sivf import Index

SIGMA = {"sift": 20.0, "box": 0.1, "sphere": 0.02}
WIDTH = {"fp32": 4, "bf16": 2, "fp8": 1}
CHUNK = 1_000_000   # vectors drawn and added at a time
RING_STEPS = 8      # batches a sliding window's id space holds beyond the window


# ------------------------------------------------------------------ cases
def _search(name, data, d, n, lists, comps, slab, queries, k, nprobe, dtype, zipf=False):
    return {"name": name, "op": "search", "data": data, "d": d, "n": n, "lists": lists,
            "comps": comps, "slab": slab, "zipf": zipf, "queries": queries, "k": k,
            "nprobe": nprobe, "dtype": dtype}


def listed():
    return [
        # one query against a small index: the latency of a call (tiny window)
        _search("q1_fp32_tiny", "box", 32, 20_000, 64, 64, 32, 1, 10, 8, "fp32"),
        # a server's small query batch over many lists: few queries per list,
        # so the scan streams its lists for one or two queries each
        _search("serving_bf16", "box", 128, 10_000_000, 16384, 16384, 128, 61, 10, 32, "bf16"),
        # the exact FP32 form at throughput: 10,000 queries over a SIFT-like million
        _search("search_fp32_sift", "sift", 128, 1_000_000, 1024, 1024, 64, 10_000, 10, 8, "fp32"),
        # nothing a power of two: odd counts, d not a multiple of 16, deeper k
        _search("search_fp32_ragged", "box", 100, 300_007, 1000, 300, 64, 777, 50, 20, "fp32"),
        # a medium query batch with wide probing, quantizer cells close together
        _search("search_bf16_mixed", "box", 128, 5_000_000, 2048, 64, 64, 1000, 10, 64, "bf16"),
        # skewed lists: the heaviest holds a large share of the vectors
        _search("search_fp8_zipf", "sift", 128, 1_000_000, 1024, 1024, 64, 10_000, 10, 8, "fp8",
                zipf=True),
        # high recall, many results: k = 100 over a Deep-like ten million
        _search("search_fp8_deep", "sphere", 96, 10_000_000, 4096, 4096, 32, 10_000, 100, 64,
                "fp8"),
        # the sliding-window step as one recorded queue: insert 10,000, delete
        # the oldest 10,000, search 10,000 fresh queries
        {"name": "step_fp8_sift", "op": "step", "data": "sift", "d": 128, "n": 1_000_000,
         "lists": 1024, "comps": 1024, "slab": 64, "zipf": False, "batch": 10_000,
         "queries": 10_000, "k": 10, "nprobe": 1, "dtype": "fp8"},
        # a small mixed update (insert, query, delete) on a large live index
        {"name": "update_small", "op": "update", "data": "box", "d": 128, "n": 5_000_000,
         "lists": 2048, "comps": 64, "slab": 64, "zipf": False, "batch": 301,
         "queries": 64, "k": 10, "nprobe": 8, "dtype": "bf16"},
        # the largest mixed update of the same queue
        {"name": "update_large", "op": "update", "data": "box", "d": 128, "n": 5_000_000,
         "lists": 2048, "comps": 64, "slab": 64, "zipf": False, "batch": 49_999,
         "queries": 1000, "k": 10, "nprobe": 8, "dtype": "bf16"},
        # bulk load of an empty index with both reduced copies, a check by
        # queries, bulk delete
        {"name": "ingest_zipf", "op": "update", "data": "sift", "d": 128, "n": 0,
         "lists": 1024, "comps": 1024, "slab": 64, "zipf": True, "batch": 1_000_000,
         "queries": 256, "k": 10, "nprobe": 8, "dtype": "fp8"},
        # the quantizer itself: Lloyd's k-means on a sample
        {"name": "train_sift", "op": "train", "data": "sift", "d": 128, "n": 200_000,
         "lists": 1024, "comps": 1024, "slab": 64, "zipf": False, "iters": 10},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["search"] * 5 + ["update"] * 2 + ["step", "train"])
    data = rng.choice(["sift", "box", "sphere"])
    dtype = rng.choice(["fp32", "bf16", "fp8"])
    d = rng.choice([32, 64, 96, 128] if dtype != "fp32" else [20, 32, 64, 96, 100, 128, 132, 192])
    slab = rng.choice([c for c in (32, 64, 128) if c * d <= 20480])
    n = _log(rng, 20_000, 5_000_000)
    lists = min(_log(rng, 64, 4096), n // 64)
    comps = lists if rng.random() < 0.6 else max(16, lists // rng.randint(2, 32))
    c = {"op": op, "data": data, "d": d, "n": n, "lists": lists, "comps": comps, "slab": slab,
         "zipf": rng.random() < 0.2}
    if op == "train":
        c.update(n=max(lists, min(n, 200_000)), iters=rng.randint(2, 10))
        return c
    nprobe = min(lists, _log(rng, 1, 64))
    queries = _log(rng, 1, 10_000) if op != "step" else _log(rng, 100, 10_000)
    # no more scanned pairs than the largest listed search
    per = nprobe * (n / lists) * d * (4 if c["zipf"] else 1) * (4 if dtype == "fp32" else 1)
    queries = max(1, min(queries, int(1e11 / per)))
    c.update(queries=queries, k=rng.choice([1, 5, 10, 10, 10, 20, 50, 100]), nprobe=nprobe,
             dtype=dtype)
    if op == "step":
        c["batch"] = min(_log(rng, 100, 10_000), n // 4)
    elif op == "update":
        c["batch"] = _log(rng, 1, 100_000)
    return c


# ----------------------------------------------------------------- inputs
class _Source:
    """Vectors of one case's distribution, drawn on the GPU from the seed."""

    def __init__(self, case, seed):
        self.c = case
        self.g = torch.Generator(device="cuda")
        self.g.manual_seed(int(seed))
        m, d = case["comps"], case["d"]
        u = torch.rand((m, d), generator=self.g, device="cuda")
        if case["data"] == "sift":
            self.centers = u * 255.0
        elif case["data"] == "box":
            self.centers = u * 2.0 - 1.0
        else:
            z = torch.randn((m, d), generator=self.g, device="cuda")
            self.centers = z / z.norm(dim=1, keepdim=True)
        self.law = None
        if case["zipf"]:
            p = 1.0 / torch.arange(1, m + 1, device="cuda", dtype=torch.float64)
            rank = torch.randperm(m, generator=self.g, device="cuda")
            self.law = torch.cumsum((p / p.sum())[rank], 0)

    def rows(self, n):
        m, d, kind = self.c["comps"], self.c["d"], self.c["data"]
        if self.law is None:
            comp = torch.randint(0, m, (n,), generator=self.g, device="cuda")
        else:
            u = torch.rand(n, generator=self.g, device="cuda", dtype=torch.float64)
            comp = torch.searchsorted(self.law, u).clamp_(max=m - 1)
        x = torch.randn((n, d), generator=self.g, device="cuda")
        x = x.mul_(SIGMA[kind]).add_(self.centers[comp])
        if kind == "sift":
            x = x.round_().clamp_(0.0, 255.0)
        elif kind == "sphere":
            x = x / x.norm(dim=1, keepdim=True)
        return x.contiguous()

    def quantizer(self):
        L = self.c["lists"]
        return self.centers[:L].contiguous() if L <= self.c["comps"] else self.rows(L)


def _inputs(case, seed):
    """(quantizer, base vector chunks, new vectors or None, queries) in order."""
    s = _Source(case, seed)
    cent = s.quantizer()
    n, q = case["n"], case["queries"]
    if case["op"] == "step":
        n = _ring(case)[0] * case["batch"]
    queries = s.rows(q)
    new = s.rows(case["batch"]) if case["op"] == "update" else None
    chunks = (s.rows(min(CHUNK, n - i)) for i in range(0, n, CHUNK))
    return cent, chunks, new, queries


def _ring(case):
    """(batches of the id space, batches of the window) of a sliding window."""
    window = max(1, case["n"] // case["batch"])
    return window + RING_STEPS, window


def _index(case, n_max):
    L, C = case["lists"], case["slab"]
    n_slabs = -(-n_max // C) + 4 * L
    dir_cap = 0 if L * n_slabs <= 1 << 29 else 64 + 16 * (-(-n_max // (L * C)))
    dtype = case.get("dtype", "fp32")
    # a bulk load keeps both reduced copies, the other cases the one they scan
    kinds = ("bf16", "fp8") if case["op"] == "update" and case["n"] == 0 and dtype != "fp32" else \
        () if dtype == "fp32" else (dtype,)
    return Index(case["d"], L, C, n_max, n_slabs, dir_cap, kinds)


def prepare(case, seed):
    if case["op"] == "train":
        s = _Source(case, seed)
        return {"case": case, "index": _index(case, case["n"]), "x": s.rows(case["n"]),
                "seed": int(seed)}
    cent, chunks, new, queries = _inputs(case, seed)
    st = {"case": case, "q": queries, "new": new}
    if case["op"] == "step":
        ring, window = _ring(case)
        B, k = case["batch"], case["k"]
        index = _index(case, ring * B)
        index.set_centroids(cent)
        st["x"] = torch.cat(list(chunks)).view(ring, B, -1)
        st["ids"] = torch.arange(ring * B, device="cuda").view(ring, B)
        index.add(st["ids"][:window].reshape(-1), st["x"][:window].reshape(window * B, -1))
        buf = {"ids_in": torch.empty(B, dtype=torch.int64, device="cuda"),
               "x_in": torch.empty((B, case["d"]), device="cuda"),
               "ids_out": torch.empty(B, dtype=torch.int64, device="cuda"),
               "q": torch.empty_like(queries),
               "dist": torch.empty((case["queries"], k), device="cuda"),
               "labels": torch.empty((case["queries"], k), dtype=torch.int64, device="cuda")}
        index.sync()
        st["queue"] = index.executor([
            {"kind": "add", "ids": buf["ids_in"], "x": buf["x_in"]},
            {"kind": "remove", "ids": buf["ids_out"]},
            {"kind": "search", "q": buf["q"], "k": k, "nprobe": case["nprobe"],
             "dtype": case["dtype"], "dist": buf["dist"], "labels": buf["labels"]}])
        st.update(buf=buf, ring=ring, window=window, at=0)
    else:
        n, extra = case["n"], case.get("batch", 0)
        index = _index(case, n + extra)
        index.set_centroids(cent)
        at = 0
        for x in chunks:
            index.add(torch.arange(at, at + len(x), device="cuda"), x)
            at += len(x)
        if new is not None:
            st["ids"] = torch.arange(n, n + extra, device="cuda")
        index.sync()
    st["index"] = index
    return st


# ------------------------------------------------------------------- pass
def run(state):
    case, index = state["case"], state["index"]
    if case["op"] == "train":
        index.train(state["x"], case["iters"], state["seed"])
        return index.centroids()
    if case["op"] == "search":
        return index.search(state["q"], case["k"], case["nprobe"], case["dtype"])
    if case["op"] == "update":
        index.add(state["ids"], state["new"])
        out = index.search(state["q"], case["k"], case["nprobe"], case["dtype"])
        index.remove(state["ids"])
        return out
    b, ring = state["buf"], state["ring"]
    new, old = (state["at"] + state["window"]) % ring, state["at"] % ring
    state["at"] += 1
    b["ids_in"].copy_(state["ids"][new])
    b["x_in"].copy_(state["x"][new])
    b["ids_out"].copy_(state["ids"][old])
    b["q"].copy_(state["q"])
    state["queue"].launch()
    return b["dist"], b["labels"]


# ------------------------------------------------------------------- work
def work(case):
    """Bytes and operations one pass cannot do without."""
    d, L = case["d"], case["lists"]
    if case["op"] == "train":
        n = case["n"]
        return {"bytes": case["iters"] * (n * d * 4 + 2 * L * d * 4),
                "flops": case["iters"] * 2.0 * n * L * d}
    nq, k, P = case["queries"], case["k"], case["nprobe"]
    live = case["n"] + (case["batch"] if case["op"] == "update" else 0)
    w = WIDTH[case["dtype"]]
    share = 1.0 - (1.0 - P / L) ** nq                 # lists that some query probes
    pairs = nq * P * (live / L)
    read = share * live * d * w + nq * d * 4 + L * d * 4
    if case["dtype"] != "fp32":
        read += min(nq * 4 * k, live) * d * 4         # the rows of the exact re-rank
    b = read + nq * k * 12
    f = 2.0 * d * pairs + 2.0 * nq * L * d
    if case["op"] != "search":
        copies = 4 + (3 if case["n"] == 0 and case["dtype"] != "fp32" else
                      0 if case["dtype"] == "fp32" else w)
        B = case["batch"]
        b += B * (d * 4 + d * copies + 2 * 8 + 24) + B * 32
        f += 2.0 * B * L * d
    return {"bytes": b, "flops": f}


# ----------------------------------------------------- answers in 64 bits
def _nearest(x, cent, P):
    """The P nearest rows of `cent` to each row of x by FP64 distance: FP32
    picks 8 more than asked for, FP64 decides among them."""
    cn = (cent.double() ** 2).sum(1)
    m = min(len(cent), P + 8)
    out = []
    step = max(1, min(65536, (1 << 29) // len(cent), (1 << 28) // (m * x.shape[1])))
    for i in range(0, len(x), step):
        a = x[i:i + step]
        some = (cn.float() - 2.0 * (a @ cent.T)).topk(m, dim=1, largest=False).indices
        some = some.sort(dim=1).values
        far = ((a.double()[:, None] - cent.double()[some]) ** 2).sum(2)
        at = far.sort(dim=1, stable=True).indices[:, :P]
        out.append(some.gather(1, at))
    return torch.cat(out)


def _knn(case, cent, x, q):
    """FP64 distances of the k nearest vectors of each query's lists."""
    k, P, L = case["k"], case["nprobe"], len(cent)
    lab = _nearest(x, cent, 1)[:, 0]
    order = lab.argsort()
    cnt = torch.bincount(lab, minlength=L).tolist()
    off = np.concatenate([[0], np.cumsum(cnt)])
    probe = _nearest(q, cent, P)
    best = torch.full((len(q), P, k), math.inf, dtype=torch.float64, device="cuda")
    pl, pair = probe.reshape(-1).sort()
    pn = torch.bincount(pl, minlength=L).tolist()
    po = np.concatenate([[0], np.cumsum(pn)])
    for c in range(L):
        if not pn[c] or not cnt[c]:
            continue
        xc = x[order[off[c]:off[c + 1]]].double()
        xs = (xc ** 2).sum(1)
        kk = min(k, cnt[c])
        step = max(1, (1 << 28) // cnt[c])
        for i in range(int(po[c]), int(po[c + 1]), step):
            e = pair[i:min(i + step, int(po[c + 1]))]
            qc = q[e // P].double()
            dd = (qc ** 2).sum(1)[:, None] + xs[None] - 2.0 * (qc @ xc.T)
            best[e // P, e % P, :kk] = dd.topk(kk, dim=1, largest=False).values
    return best.reshape(len(q), -1).topk(k, dim=1, largest=False).values.clamp_(min=0.0)


def _first_rows(seed, n, L):
    """The rows that start k-means: SplitMix64 outputs mod n, repeats skipped."""
    mask, state, rows, seen = (1 << 64) - 1, int(seed) & ((1 << 64) - 1), [], set()
    while len(rows) < L:
        state = (state + 0x9E3779B97F4A7C15) & mask
        z = state
        z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & mask
        z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & mask
        r = (z ^ (z >> 31)) % n
        if r not in seen:
            seen.add(r)
            rows.append(r)
    return rows


def exact(case, seed):
    if case["op"] == "train":
        x = _Source(case, seed).rows(case["n"])
        L = case["lists"]
        cent = x[torch.tensor(_first_rows(seed, len(x), L), device="cuda")].clone()
        for _ in range(case["iters"]):
            lab = _nearest(x, cent, 1)[:, 0]
            total = torch.zeros((L, case["d"]), dtype=torch.float64, device="cuda")
            total.index_add_(0, lab, x.double())
            cnt = torch.bincount(lab, minlength=L)
            mean = total / cnt.clamp(min=1)[:, None]
            cent = torch.where(cnt[:, None] > 0, mean.float(), cent)
        return cent.double()
    cent, chunks, new, q = _inputs(case, seed)
    x = torch.cat(list(chunks) + ([] if new is None else [new]))
    if case["op"] == "step":
        B = case["batch"]
        x = x[B:B + _ring(case)[1] * B]
    return [_knn(case, cent, x, q), None]
