"""The work a user of this framework has it do, as measurable cases.

Every case goes through the public entry points (``flinng.Index``,
``flinng.Server``, ``sharded``) on seeded synthetic data shaped like the
repository's own workloads: genomic reads and URL-like strings as sets
(Jaccard), Gaussian-mixture vectors and ReLU embeddings as rows (cosine).
Inputs are made with torch on the GPU, so that preparing a case is quick.

A case's ``do`` is one of

* ``query``  - a batch of queries against a built index (device or host
  buffers): hash, gather, group tests, decode, top-k;
* ``serve``  - a trace of requests replayed by the continuous-batching server
  from host memory, with k mixed in {1, 10, 100};
* ``build``  - an index built from scratch, then asked for the counts and the
  top-k of a few queries (a build has no other output);
* ``ingest`` - an index built, then grown by insert batches of several sizes,
  then queried;
* ``hash``   - the codes of a batch of vectors, as a program that streams its
  points into ``build_buckets`` asks for them;
* ``shards`` - a table-sharded query: every shard's counts, their sum, the
  decode from the sum.

``points`` names the data: ``reads``, ``urls``, ``mixture``, ``relu``.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2106_11565_gb300 import flinng as F
from paper_2106_11565_gb300 import sharded
from paper_2106_11565_gb300 import workloads as WL

PRECISION = {"fp32": F.PREC_FP32, "bf16x2": F.PREC_BF16X2, "bf16": F.PREC_BF16, "fp8": F.PREC_FP8}

READS = {"points": "reads", "len": 1000}
# the genomic workload at its configured parameters and where its recall@10 reaches 0.9
CONFIGURED = dict(READS, n=100_000, R=2, B=1000, L=32, K=2, W=17)
TARGET = dict(READS, n=100_000, R=3, B=4096, L=512, K=1, W=17)
URLS = {"points": "urls", "len": 60, "n": 1_000_000, "R": 4, "B": 5000, "L": 64, "K": 1, "W": 17}
MIXTURE = {"points": "mixture", "dim": 128, "n": 10_000, "R": 3, "B": 100, "L": 16, "K": 12, "W": 12}
RELU = {"points": "relu", "dim": 4096, "R": 3, "B": 20_000, "L": 64, "K": 16, "W": 16}
# products of a vector with a projection in one pass: those of 10,000 embeddings
MOST_PRODUCTS = 10_000 * 4096 * 1024


def listed():
    return [
        # one set looked up from host memory: what an interactive caller waits for
        dict(CONFIGURED, name="one_read_host", do="query", nq=1, k=10, host=True),
        # a small batch of small vectors, hashed inside the query kernel
        dict(MIXTURE, name="query_mixture", do="query", nq=100, k=10, precision="fp32"),
        # the workload the headline metric is quoted on, as one batch
        dict(TARGET, name="query_reads", do="query", nq=1000, k=100),
        # many short ragged sets against a large index, whose lists are mostly bitmaps
        dict(URLS, name="query_urls", do="query", nq=10_000, k=10),
        # embeddings in the default precision: the projection dominates
        dict(RELU, name="query_relu_fp32", do="query", n=250_000, nq=2000, k=10, precision="fp32"),
        # a large batch of embeddings on the tensor cores
        dict(RELU, name="query_relu_bf16x2", do="query", n=1_000_000, nq=10_000, k=10, precision="bf16x2"),
        # the headline serving form: requests in host memory, batched as they come
        dict(TARGET, name="serve_reads", do="serve", requests=32_768, k=100, slots=8, batch=1024),
        # the genomic index from scratch at the headline parameters
        dict(TARGET, name="build_reads", do="build", nq=256, k=100),
        # the largest build: a million ragged sets
        dict(URLS, name="build_urls", do="build", nq=256, k=10),
        # an index that grows: small batches (the smallest of one read) and one large one
        dict(TARGET, name="ingest_reads", do="ingest", n=20_000, batches=6, most=6000, nq=256, k=100),
        # points hashed batch by batch for a streamed build, single-term precision
        dict(RELU, name="hash_relu_bf16", do="hash", n=8192, precision="bf16", proj=False),
        # an index whose tables are split over two shards
        dict(TARGET, name="shards_reads", do="shards", n=50_000, shards=2, nq=512, k=100),
    ]


def _log(rng, lo, hi):
    """An integer spread over the logarithm of [lo, hi]."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(("query", "query", "query", "query", "serve", "build", "build", "ingest", "hash", "shards"))
    if kind == "hash":
        prec = rng.choice(("fp32", "bf16x2", "bf16", "fp8"))
        c = {"points": rng.choice(("relu", "mixture")), "precision": prec,
             "dim": 16 * _log(rng, 2, 256) if prec != "fp32" else _log(rng, 24, 4096),
             "n": _log(rng, 100, 8192), "R": 3, "B": 1000, "L": rng.randint(8, 64), "K": rng.randint(6, 16),
             "proj": rng.random() < 0.4}
        c["n"] = min(c["n"], MOST_PRODUCTS // (c["dim"] * c["L"] * c["K"]))
        return dict(c, do=kind, W=c["K"])
    points = "reads" if kind in ("serve", "ingest", "shards") else rng.choice(("reads", "reads", "urls", "mixture", "relu"))
    k = _log(rng, 1, 200)
    if points in ("reads", "urls"):
        tables = _log(rng, 16, 512)
        K = 1 if tables > 64 else rng.choice((1, 2))
        W = rng.randint(12, 17)
        R = rng.randint(2, 4)
        n = _log(rng, 2000, 100_000) if points == "reads" else _log(rng, 20_000, 600_000)
        n = min(n, 150_000_000 // (tables * R))
        c = {"points": points, "len": _log(rng, 300, 1000) if points == "reads" else rng.randint(40, 80), "n": n,
             "R": R, "B": _log(rng, 200, 12_000), "L": tables, "K": K, "W": W}
    else:
        K = rng.randint(8, 16)
        prec = rng.choice(("fp32", "bf16x2"))
        c = {"points": points, "dim": 16 * _log(rng, 2, 16) if points == "mixture" else 16 * _log(rng, 32, 256),
             "n": _log(rng, 2000, 100_000), "R": rng.randint(2, 4), "B": _log(rng, 100, 15_000),
             "L": rng.randint(8, 64), "K": K, "W": K, "precision": prec}
    c.update(do=kind, k=k)
    if kind == "query":
        c["nq"] = _log(rng, 1, 4000)
        if "dim" in c:
            c["nq"] = min(c["nq"], MOST_PRODUCTS // (c["dim"] * c["L"] * c["K"]))
        c["host"] = c["nq"] <= 64 and rng.random() < 0.5
    elif kind == "serve":
        c.update(requests=_log(rng, 500, 30_000), slots=rng.randint(2, 8), batch=_log(rng, 64, 2048))
    elif kind == "build":
        c["nq"] = rng.randint(1, 256)
        if "dim" in c:
            c["n"] = min(c["n"], MOST_PRODUCTS // (c["dim"] * c["L"] * c["K"]))
    elif kind == "ingest":
        c.update(n=min(c["n"], 20_000), batches=rng.randint(2, 6), most=_log(rng, 50, 6000), nq=rng.randint(1, 256))
    else:
        c.update(shards=rng.randint(2, 3), nq=_log(rng, 1, 512))
    return c


# --------------------------------------------------------------------------
# inputs, made on the GPU from the seed
# --------------------------------------------------------------------------

def _gen(seed, part):
    g = torch.Generator(device="cuda")
    g.manual_seed((int(seed) * 1_000_003 + part) % (1 << 62))
    return g


def _reads(seed, n, length, first_part):
    """n reads of a random reference with 1-10 % substitutions, as sets of
    hashed 18-mers: (offsets int64, elements int32) on the GPU."""
    g0 = _gen(seed, 0)
    ref = torch.randint(0, 4, (5_000_000,), generator=g0, device="cuda", dtype=torch.int64)
    key = int(torch.randint(0, 1 << 62, (1,), generator=g0, device="cuda").item()) | 1
    g = _gen(seed, first_part)
    elems, sizes = [], []
    for c0 in range(0, n, 16_384):
        m = min(16_384, n - c0)
        start = torch.randint(0, ref.numel() - length + 1, (m, 1), generator=g, device="cuda")
        reads = ref[start + torch.arange(length, device="cuda")]
        rate = 0.01 + 0.09 * torch.rand((m, 1), generator=g, device="cuda")
        sub = torch.rand((m, length), generator=g, device="cuda") < rate
        shift = torch.randint(1, 4, (m, length), generator=g, device="cuda")
        reads = torch.where(sub, (reads + shift) & 3, reads)
        nk = length - 17
        code = torch.zeros((m, nk), dtype=torch.int64, device="cuda")
        for j in range(18):
            code = code * 4 + reads[:, j:j + nk]
        h = ((code * key) >> 32) & 0xFFFFFFFF
        h = h.sort(dim=1).values
        keep = torch.ones_like(h, dtype=torch.bool)
        keep[:, 1:] = h[:, 1:] != h[:, :-1]
        elems.append(h[keep].to(torch.int32))
        sizes.append(keep.sum(1))
    off = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    off[1:] = torch.cat(sizes).cumsum(0)
    return off, torch.cat(elems)


def _gram_sets(text, start, length):
    """Sets of character 3-grams of the slices text[start : start + length]."""
    n = start.numel()
    owner = torch.repeat_interleave(torch.arange(n, device="cuda"), length - 2)
    first = torch.cumsum(length - 2, 0) - (length - 2)
    pos = start[owner] + torch.arange(owner.numel(), device="cuda") - first[owner]
    gram = (text[pos] << 16) | (text[pos + 1] << 8) | text[pos + 2]
    key = ((owner << 24) | gram).sort().values
    keep = torch.ones_like(key, dtype=torch.bool)
    keep[1:] = key[1:] != key[:-1]
    key = key[keep]
    off = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    off[1:] = torch.bincount(key >> 24, minlength=n).cumsum(0)
    return off, (key & 0xFFFFFF).to(torch.int32)


def _urls(seed, n, nq, median):
    """n strings cut from a stream of Zipf(1.1) tokens joined by '/', and nq
    of them again with 5 % of their characters changed, as 3-gram sets."""
    g = _gen(seed, 1)
    vocab = 50_000
    tok_len = torch.randint(2, 13, (vocab,), generator=g, device="cuda")
    letters = torch.tensor(list(b"abcdefghijklmnopqrstuvwxyz0123456789"), device="cuda")
    chars = letters[torch.randint(0, 36, (vocab, 13), generator=g, device="cuda")]
    chars[torch.arange(vocab, device="cuda"), tok_len] = ord("/")
    cdf = (1.0 / torch.arange(1, vocab + 1, device="cuda", dtype=torch.float64) ** 1.1).cumsum(0)
    cdf /= cdf[-1].clone()
    length = (median * torch.exp(0.5 * torch.randn(n, generator=g, device="cuda", dtype=torch.float64)))
    length = length.round().clamp(3, 4096).to(torch.int64)
    start = length.cumsum(0) - length
    total = int(length.sum().item())
    toks = torch.searchsorted(cdf, torch.rand(total // 3 + 16, generator=g, device="cuda", dtype=torch.float64))
    toks = toks.clamp(max=vocab - 1)
    tl = tok_len[toks] + 1
    end = tl.cumsum(0)
    toks = toks[: int(torch.searchsorted(end, total).item()) + 1]
    tl = tl[: toks.numel()]
    owner = torch.repeat_interleave(torch.arange(toks.numel(), device="cuda"), tl)
    text = chars[toks[owner], torch.arange(owner.numel(), device="cuda") - (end[: toks.numel()] - tl)[owner]]
    pts = _gram_sets(text, start, length)
    src = torch.randint(0, n, (nq,), generator=g, device="cuda")
    ql = length[src]
    qs = ql.cumsum(0) - ql
    owner = torch.repeat_interleave(torch.arange(nq, device="cuda"), ql)
    qt = text[start[src][owner] + torch.arange(owner.numel(), device="cuda") - qs[owner]]
    edit = torch.rand(qt.numel(), generator=g, device="cuda") < 0.05
    other = letters[torch.randint(0, 36, (qt.numel(),), generator=g, device="cuda")]
    return pts, _gram_sets(torch.where(edit, other, qt), qs, ql)


def _vectors(seed, kind, n, dim, part, centers, first=0):
    """Rows of a Gaussian mixture (sigma 0.1), rectified for ``relu``."""
    g = _gen(seed, part + first)
    x = centers[torch.randint(0, centers.shape[0], (n,), generator=g, device="cuda")]
    x += 0.1 * torch.randn((n, dim), generator=g, device="cuda")
    return x.relu_() if kind == "relu" else x


def _centers(seed, c):
    k = 1000 if c["points"] == "relu" else 100
    return torch.randn((k, c["dim"]), generator=_gen(seed, 2), device="cuda")


def _queries_of_vectors(seed, c, centers, nq):
    # a point of the stream with a little noise
    g = _gen(seed, 4)
    x = centers[torch.randint(0, centers.shape[0], (nq,), generator=g, device="cuda")]
    x += 0.1 * torch.randn((nq, c["dim"]), generator=g, device="cuda")
    x += 0.05 * torch.randn((nq, c["dim"]), generator=g, device="cuda")
    return x.relu_() if c["points"] == "relu" else x


def _perm(seed, R, n, part):
    g = _gen(seed, 1000 + part)
    return torch.stack([torch.randperm(n, generator=g, device="cuda") for _ in range(R)]).to(torch.int32)


def _is_set(c):
    return c["points"] in ("reads", "urls")


def _hash_params(seed, c):
    seed = int(seed) % (1 << 31)
    return WL.doph_params(seed, c["L"], c["K"]) if _is_set(c) else WL.srp_projections(seed, c["L"] * c["K"], c["dim"])


def _index(c, params, capacity, tables=None):
    return F.Index("jaccard" if _is_set(c) else "cosine", c["R"], c["B"], tables or c["L"], c["K"],
                   capacity=capacity, params=params, dim=c.get("dim", 0), W=c["W"],
                   precision=PRECISION[c.get("precision", "fp32")])


def _sets(seed, c, n, nq):
    if c["points"] == "urls":
        return _urls(seed, n, nq, c["len"])
    return _reads(seed, n, c["len"], 10), _reads(seed, nq, c["len"], 11)


def _host(q):
    if isinstance(q, tuple):
        return q[0].cpu().numpy().astype(np.uint64), q[1].cpu().numpy().view(np.uint32)
    return q.cpu().numpy()


def _slice_sets(pts, a, b):
    off, el = pts
    return (off[a:b + 1] - off[a]).contiguous(), el[int(off[a]):int(off[b])].contiguous()


def _built(seed, c, n):
    """A built index, and a function that draws queries for it."""
    ix = _index(c, _hash_params(seed, c), n)
    if _is_set(c):
        pts, q = _sets(seed, c, n, c.get("nq") or c["requests"])
        ix.build(pts, _perm(seed, c["R"], n, 0))
        return ix, q
    centers = _centers(seed, c)
    # rows hashed batch by batch, as a program whose points do not fit at once does
    codes = torch.empty((n, c["L"]), dtype=torch.int32, device="cuda")
    for i, a in enumerate(range(0, n, 65_536)):
        m = min(65_536, n - a)
        codes[a:a + m] = ix.hash(_vectors(seed, c["points"], m, c["dim"], 100, centers, i))[0]
    ix.build_buckets(codes, _perm(seed, c["R"], n, 0))
    return ix, _queries_of_vectors(seed, c, centers, c["nq"])


# --------------------------------------------------------------------------
# the cases
# --------------------------------------------------------------------------

def _batch_sizes(c):
    """Insert batches from one point up to the largest, over their logarithm."""
    b = c["batches"]
    return [max(1, int(round(c["most"] ** (i / (b - 1))))) for i in range(b)]


def prepare(case, seed):
    c = dict(case)
    st = {"case": c}
    n = c["n"]
    if c["do"] == "query":
        st["ix"], q = _built(seed, c, n)
        st["q"] = _host(q) if c.get("host") else q
    elif c["do"] == "serve":
        ix, q = _built(seed, c, n)
        off, el = _host(q)
        m = c["requests"]
        srv = F.Server(hbm_budget=64 << 30, n_slots=c["slots"], max_batch=c["batch"], k_max=max(c["k"], 1))
        which = srv.add_index(ix)
        reqs = np.zeros(m, F.REQ_DTYPE)
        ks = np.minimum(np.array([1, 10, 100], np.uint32), c["k"])
        reqs["kind"], reqs["index"] = F.REQ_QUERY, which
        reqs["k"] = ks[np.random.default_rng(int(seed)).integers(0, 3, m)]
        reqs["n"] = np.diff(off)
        reqs["data"] = el.ctypes.data + off[:-1] * np.uint64(4)
        out = np.zeros((m, max(c["k"], 1)), np.uint32), np.zeros((m, max(c["k"], 1)), np.uint16)
        st.update(ix=ix, srv=srv, reqs=reqs, keep=(off, el), out=out)
    elif c["do"] == "build":
        st["ix"] = ix = _index(c, _hash_params(seed, c), n)
        if _is_set(c):
            st["pts"], st["q"] = _sets(seed, c, n, c["nq"])
        else:
            centers = _centers(seed, c)
            st["pts"] = _vectors(seed, c["points"], n, c["dim"], 100, centers)
            st["q"] = _queries_of_vectors(seed, c, centers, c["nq"])
        st["perm"] = _perm(seed, c["R"], n, 0)
        st["qb"] = ix.hash(st["q"])[0]
    elif c["do"] == "ingest":
        sizes = _batch_sizes(c)
        total = n + sum(sizes)
        st["ix"] = _index(c, _hash_params(seed, c), total)
        pts, st["q"] = _sets(seed, c, total, c["nq"])
        ends = np.cumsum([n] + sizes)
        st["parts"] = [_slice_sets(pts, a, b) for a, b in zip([0] + list(ends[:-1]), ends)]
        st["perms"] = [_perm(seed, c["R"], m, i) for i, m in enumerate([n] + sizes)]
        st["qb"] = st["ix"].hash(st["q"])[0]
    elif c["do"] == "hash":
        st["ix"] = _index(c, _hash_params(seed, c), 16)
        st["x"] = _vectors(seed, c["points"], n, c["dim"], 100, _centers(seed, c))
    else:
        # every shard holds all points and its own range of the tables
        full = _index(c, _hash_params(seed, c), 16)
        pts, q = _sets(seed, c, n, c["nq"])
        codes, qb = full.hash(pts)[0], full.hash(q)[0]
        perm = _perm(seed, c["R"], n, 0)
        st["shards"], st["qb"] = [], []
        for r in range(c["shards"]):
            a, b = sharded.table_range(c["L"], c["shards"], r)
            ix = _index(c, WL.doph_params(1, b - a, c["K"]), n, tables=b - a)
            ix.build_buckets(codes[:, a:b].contiguous(), perm)
            st["shards"].append(ix)
            st["qb"].append(qb[:, a:b].contiguous())
    return st


def run(state):
    c = state["case"]
    if c["do"] == "query":
        return state["ix"].query(state["q"], c["k"])
    if c["do"] == "serve":
        ids, scores, _ = state["srv"].replay(state["reqs"], out=state["out"])
        return ids, scores
    if c["do"] == "build":
        ix = state["ix"]
        ix.build(state["pts"], state["perm"])
        return ix.query(state["q"], c["k"]), ix.counts(state["qb"])
    if c["do"] == "ingest":
        ix = state["ix"]
        ix.build(state["parts"][0], state["perms"][0])
        for pts, perm in zip(state["parts"][1:], state["perms"][1:]):
            ix.insert(pts, perm)
        return ix.query(state["q"], c["k"]), ix.counts(state["qb"])
    if c["do"] == "hash":
        codes, _, proj = state["ix"].hash(state["x"], proj=c["proj"])
        return [codes, proj] if c["proj"] else [codes]
    parts = [ix.counts(qb) for ix, qb in zip(state["shards"], state["qb"])]
    total = parts[0]
    for p in parts[1:]:
        total = total + p
    return total, state["shards"][0].query_counts(total, c["k"], c["L"])


def _point_bytes(c):
    return 4 * c["dim"] if not _is_set(c) else 4 * (c["len"] - 18 if c["points"] == "reads" else c["len"])


def _hash_flops(c, n):
    # one multiply and one add per projection and dimension; a few operations per set element
    return 2.0 * n * c["dim"] * c["L"] * c["K"] if not _is_set(c) else n * _point_bytes(c) / 4 * 4.0


def _query_work(c, nq):
    """One query reads its input, its tables' list bounds and their lists (at
    least the bucket's average), and writes k ids and scores."""
    cells = c["R"] * max(1.0, c["n"] / 2.0 ** c["W"])
    return nq * (_point_bytes(c) + c["L"] * (8.0 + 2.0 * cells) + 6.0 * c["k"])


def work(case):
    c = dict(case)
    n, slots = c["n"], float(c["L"]) * 2 ** c["W"]
    if c["do"] == "query":
        return {"bytes": _query_work(c, c["nq"]), "flops": _hash_flops(c, c["nq"])}
    if c["do"] == "serve":
        return {"bytes": _query_work(c, c["requests"]), "flops": _hash_flops(c, c["requests"])}
    if c["do"] == "hash":
        out = 4.0 * n * c["L"] + (4.0 * n * c["L"] * c["K"] if c["proj"] else 0.0)
        return {"bytes": n * _point_bytes(c) + 4.0 * c["L"] * c["K"] * c["dim"] + out, "flops": _hash_flops(c, n)}
    if c["do"] == "shards":
        counts = 2.0 * c["nq"] * c["B"] * c["R"]
        return {"bytes": _query_work(c, c["nq"]) + counts * (2 * c["shards"] + 2), "flops": float(c["nq"] * c["L"])}
    # the points and their placement read, every list's bounds and cells and the members written
    total = n + (sum(_batch_sizes(c)) if c["do"] == "ingest" else 0)
    built = total * (_point_bytes(c) + 4.0 * c["R"]) + 4.0 * slots + 2.0 * total * c["L"] * c["R"] + 8.0 * total * c["R"]
    counts = 2.0 * c["nq"] * c["B"] * c["R"]
    return {"bytes": built + counts + _query_work(c, c["nq"]), "flops": _hash_flops(c, total)}


def exact(case, seed):
    """The projections and codes of a hashed batch in 64 bits; every other
    output is a whole number the framework promises exactly."""
    c = dict(case)
    if c["do"] != "hash":
        return None
    x = _vectors(seed, c["points"], c["n"], c["dim"], 100, _centers(seed, c)).double()
    w = torch.from_numpy(_hash_params(seed, c)).cuda().double()
    p = x @ w.T
    bits = (p > 0).view(c["n"], c["L"], c["K"]).to(torch.int64)
    codes = (bits << torch.arange(c["K"], device="cuda")).sum(2).to(torch.int32)
    return [codes, p] if c["proj"] else [codes]
