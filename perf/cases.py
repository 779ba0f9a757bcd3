"""The work that programs have this library do, as cases that can be measured.

A case is a dict of plain values; ``prepare`` makes what a program holds
before the call (an index, a snapshot, an executor, the queries), ``run`` is
one pass through the public entry points, and ``exact`` gives the same
scores in binary64 from plain torch.  Kinds:

* ``query``   one dense cursor: open, read the ranks page by page, close;
* ``serve``   many requests through the native executor, eight to a group;
* ``batch``   a query batch on the tensor cores, read in a few pulls;
* ``fuse``    an EAHR Top-20 over a dense cursor and a host sparse ranking;
* ``hybrid``  an EAHR Top-20 over a dense cursor and a PBM cursor;
* ``sparse``  one PBM cursor: open, read the ranks page by page, close;
* ``rerank``  the allocation-free ranking of a few thousand caller's vectors;
* ``build``   a corpus quantized into an index, which answers its first page.

Corpora are Gaussian mixtures of unit vectors (``components`` centres, 0.35
noise; queries are centres with 0.5 noise) or i.i.d. unit normals
(``components`` 0); postings carry BM25 impacts of a Zipf vocabulary.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2608_07152_gb300 as pvs

PASSAGES = 8_841_823      # MS MARCO passages, the benchmark's corpus size
DEVICE = "cuda"
CHUNK = 1 << 20
K = 20                    # EAHR Top-K, w / (60 + rank)
VOCAB = 200_000           # background terms of the synthetic postings
SKIP = 100                # most frequent ranks removed, like stopwords
TOKENS = 40               # mean tokens per item
TOPIC_TERMS = 64          # terms of each topic's own block (hybrid)
TOPIC_SHARE = 0.3


def listed():
    return [
        # a small collection's first page: open, one pull, close (latency and launches)
        dict(name="first_page_10k", kind="query", n=10_000, dim=128, components=0,
             deleted=0.0, ranks=20, page=20),
        # a lone user pages through the first 1,000 ranks of the passage corpus
        dict(name="pages_passage", kind="query", n=PASSAGES, dim=768, components=4096,
             deleted=0.0, ranks=1000, page=20),
        # a width that fits no tile, on a snapshot with deletions
        dict(name="pages_ragged_1M", kind="query", n=1_000_003, dim=385, components=512,
             deleted=0.02, ranks=300, page=50),
        # the serving workload: 128 requests from pinned host memory
        dict(name="serve_passage", kind="serve", n=PASSAGES, dim=768, components=4096,
             requests=128, ranks=1000, page=20, host=True),
        # a smaller service (bge-small width) with its buffers on the device
        dict(name="serve_500k", kind="serve", n=500_000, dim=384, components=256,
             requests=48, ranks=100, page=20, host=False),
        # an offline batch of 256 queries, their first 200 ranks
        dict(name="batch_1M", kind="batch", n=1_000_000, dim=768, components=1024,
             queries=256, ranks=200, pulls=4),
        # hybrid search with a sparse ranking unrelated to the dense one
        dict(name="fuse_passage", kind="fuse", n=PASSAGES, dim=768, components=4096,
             deleted=0.0, duplicates=0.0, tau=0.0),
        # the same on a growing collection: near-duplicates and deletions
        dict(name="fuse_snapshot_2M", kind="fuse", n=2_000_000, dim=1024, components=1024,
             deleted=0.02, duplicates=0.2, tau=0.2),
        # both channels from indexes of this library
        dict(name="hybrid_2M", kind="hybrid", n=2_000_000, dim=768, components=1024, terms=4),
        # the sparse channel alone
        dict(name="sparse_4M", kind="sparse", n=4_000_000, terms=5, ranks=1000, page=20),
        # a first stage's candidates ordered exactly, without allocations
        dict(name="rerank_1000", kind="rerank", n=1000, dim=768, top=100),
        # a new Segment is indexed and answers its first page
        dict(name="build_500k", kind="build", n=500_000, dim=768, components=512),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _dim(rng):
    return rng.choice([64, 96, 100, 128, 200, 256, 300, 384, 385, 512, 640, 768, 1000, 1024,
                       rng.randint(64, 1024)])


def _components(rng, n):
    return 0 if rng.random() < 0.25 else max(4, min(4096, n // rng.randint(800, 2200)))


def _rows(rng, dim, lo=10_000, hi=PASSAGES):
    return min(_log(rng, lo, hi), PASSAGES * 768 // dim)


def draw(rng):
    kind = rng.choice(["query", "query", "serve", "serve", "batch", "fuse", "hybrid", "sparse",
                       "rerank", "build"])
    dim = _dim(rng)
    if kind == "query":
        n = _rows(rng, dim)
        page = rng.choice([10, 20, 33, 50, 100])
        return dict(kind=kind, n=n, dim=dim, components=_components(rng, n),
                    deleted=rng.choice([0.0, 0.0, 0.02]), ranks=page * rng.randint(1, 10),
                    page=page)
    if kind == "serve":   # odd widths at up to 20 requests' worth of the whole passage corpus
        requests = _log(rng, 9, 128)
        hi = PASSAGES
        if dim not in (64, 128, 256, 384, 512, 768, 1024):
            hi = min(hi, 20 * PASSAGES * 768 // (requests * dim))
        n = _rows(rng, dim, 20_000, hi)
        return dict(kind=kind, n=n, dim=dim, components=_components(rng, n),
                    requests=requests, ranks=rng.choice([20, 100, 250, 500, 1000]),
                    page=20, host=rng.random() < 0.5)
    if kind == "batch":
        n = _rows(rng, dim, 50_000, 2_000_000)
        pulls = rng.randint(1, 4)
        return dict(kind=kind, n=n, dim=dim, components=_components(rng, n),
                    queries=_log(rng, 16, 256), ranks=pulls * rng.choice([10, 25, 50]),
                    pulls=pulls)
    if kind == "fuse":
        n = _rows(rng, dim, 20_000, 4_000_000)
        return dict(kind=kind, n=n, dim=dim, components=_components(rng, n),
                    deleted=rng.choice([0.0, 0.02]), duplicates=rng.choice([0.0, 0.2]),
                    tau=rng.choice([-0.5, -0.2, 0.0, 0.2, 0.5]))
    if kind == "hybrid":
        n = _rows(rng, dim, 50_000, 2_000_000)
        return dict(kind=kind, n=n, dim=dim, components=max(4, n // 2000),
                    terms=rng.randint(2, 6))
    if kind == "sparse":
        page = rng.choice([10, 20, 50, 100])
        return dict(kind=kind, n=_log(rng, 50_000, 4_000_000), terms=rng.randint(1, 8),
                    ranks=page * rng.randint(1, 10), page=page)
    if kind == "rerank":
        n = _log(rng, 50, pvs.PVS_NOALLOC_MAX_VECTORS)
        return dict(kind=kind, n=n, dim=dim, top=min(n, rng.choice([10, 20, 50, 100, 500])))
    n = _rows(rng, dim, 10_000, 1_000_000)
    return dict(kind=kind, n=n, dim=dim, components=_components(rng, n))


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _gen(seed, part, device=DEVICE):
    g = torch.Generator(device=device)
    g.manual_seed((int(seed) * 1_000_003 + 7919 * int(part) + 17) & ((1 << 62) - 1))
    return g


def _unit(x):
    return x.div_(torch.linalg.vector_norm(x, dim=1, keepdim=True).clamp_min_(1e-30))


def _centres(case, seed):
    c = case.get("components", 0)
    return torch.randn((c, case["dim"]), generator=_gen(seed, -1), device=DEVICE) if c else None


def _corpus(case, seed):
    """(float32 [n, dim] unit rows, component of each row or None)."""
    n, dim, centres = case["n"], case["dim"], _centres(case, seed)
    out = torch.empty((n, dim), device=DEVICE)
    comp = None if centres is None else torch.randint(
        0, centres.shape[0], (n,), generator=_gen(seed, -2), device=DEVICE)
    for r in range(0, n, CHUNK):
        x = out[r:r + CHUNK]
        x.normal_(generator=_gen(seed, r // CHUNK))
        if centres is not None:
            x.mul_(0.35).add_(centres[comp[r:r + CHUNK]])
        _unit(x)
    dup = int(n * case.get("duplicates", 0.0))
    if dup:   # the last rows are near-copies of random earlier ones
        src = torch.randint(0, n - dup, (dup,), generator=_gen(seed, -3), device=DEVICE)
        noise = torch.empty((dup, dim), device=DEVICE).normal_(0.0, 1e-4,
                                                               generator=_gen(seed, -4))
        out[n - dup:] = _unit(noise.add_(out[src]))
    return out, comp


def _queries(case, seed, nq):
    """(float32 [nq, dim] unit rows, their components or None)."""
    g = _gen(seed, -5)
    centres = _centres(case, seed)
    x = torch.randn((nq, case["dim"]), generator=g, device=DEVICE)
    comp = None
    if centres is not None:
        comp = torch.randint(0, centres.shape[0], (nq,), generator=g, device=DEVICE)
        x.mul_(0.5).add_(centres[comp])
    return _unit(x), comp


def _deleted(case, seed):
    """Ids of the deleted rows (host int64), or None."""
    share = case.get("deleted", 0.0)
    if not share:
        return None
    u = torch.rand(case["n"], generator=_gen(seed, -6), device=DEVICE)
    return torch.nonzero(u < share).flatten().cpu().numpy()


def _sparse_ranking(case, seed, corpus, query, dead):
    """A complete ranking of the visible ids (host int64) whose Kendall tau
    against the dense one is about case["tau"] (a Gaussian copula)."""
    score = corpus @ query
    n = score.numel()
    rank = torch.empty(n, device=DEVICE)
    rank[torch.argsort(score, descending=True)] = torch.arange(n, device=DEVICE,
                                                               dtype=torch.float32)
    z = torch.special.ndtri((n - rank.double() - 0.5) / n)
    rho = math.sin(math.pi * case["tau"] / 2.0)
    eps = torch.randn(n, generator=_gen(seed, -7), device=DEVICE, dtype=torch.float64)
    order = torch.argsort(rho * z + math.sqrt(1.0 - rho * rho) * eps, descending=True)
    if dead is not None:
        alive = torch.ones(n, dtype=torch.bool, device=DEVICE)
        alive[torch.from_numpy(dead).to(DEVICE)] = False
        order = order[alive[order]]
    return order.cpu().numpy()


def _postings(n, seed, topics=None, n_topics=0):
    """Term-major BM25 postings on the device: (term_off int64, docs int32,
    imps float32).  With topics, a share of each item's tokens comes from its
    topic's block of terms, numbered after the VOCAB background terms."""
    vocab = VOCAB + n_topics * TOPIC_TERMS
    w = 1.0 / (torch.arange(1, VOCAB + 1, dtype=torch.float64, device=DEVICE) + SKIP)
    cdf = torch.cumsum(w, 0)
    cdf = (cdf / cdf[-1]).float()
    length = torch.poisson(torch.full((n,), float(TOKENS), device=DEVICE),
                           generator=_gen(seed, -8)).long()
    docs = torch.repeat_interleave(torch.arange(n, device=DEVICE), length)
    g = _gen(seed, -9)
    total = docs.numel()
    term = torch.searchsorted(cdf, torch.rand(total, generator=g, device=DEVICE))
    term.clamp_max_(VOCAB - 1)
    if topics is not None:
        own = VOCAB + topics[docs] * TOPIC_TERMS + torch.randint(
            0, TOPIC_TERMS, (total,), generator=g, device=DEVICE)
        term = torch.where(torch.rand(total, generator=g, device=DEVICE) < TOPIC_SHARE, own, term)
    key = torch.sort(term.mul_(n).add_(docs)).values
    del docs, term
    key, tf = torch.unique_consecutive(key, return_counts=True)
    term = torch.div(key, n, rounding_mode="floor")
    docs = key - term * n
    df = torch.bincount(term, minlength=vocab)
    off = torch.zeros(vocab + 1, dtype=torch.int64, device=DEVICE)
    torch.cumsum(df, 0, out=off[1:])
    idf = torch.log1p((n - df + 0.5) / (df + 0.5)).float()
    norm = 0.9 * (0.6 + 0.4 * length.float() / length.float().mean())
    tf = tf.float()
    imps = idf[term] * tf * 1.9 / (tf + norm[docs])
    return off, docs.int(), imps


def _distinct(draws, count):
    """The first `count` distinct values of a list, in order."""
    seen = list(dict.fromkeys(draws))
    return np.array(seen[:count], np.int32)


def _background_terms(off, count, seed):
    """Distinct background terms drawn in proportion to their postings."""
    if count == 0:
        return np.zeros(0, np.int32)
    at = torch.randint(0, int(off[VOCAB]), (16 * count + 64,), generator=_gen(seed, -10),
                       device=DEVICE)
    return _distinct((torch.searchsorted(off, at, right=True) - 1).tolist(), count)


def _sparse_terms(case, seed, off, topic=None):
    if topic is None:
        return _background_terms(off, case["terms"], seed)
    own = (case["terms"] + 1) // 2
    pick = torch.randint(0, TOPIC_TERMS, (64 * own,), generator=_gen(seed, -11), device=DEVICE)
    block = _distinct((VOCAB + topic * TOPIC_TERMS + pick).tolist(), own)
    return np.concatenate([block, _background_terms(off, case["terms"] - own, seed)])


class _Held:
    """Handles of the library, freed when dropped, the last one kept first."""

    def __init__(self):
        self._frees = []

    def keep(self, handle, free):
        self._frees.insert(0, (free, handle))
        return handle

    def __del__(self):
        for free, handle in self._frees:
            free(handle)


def _indexed(case, seed, held):
    """(index, snapshot or None, corpus, components, deleted ids or None)."""
    corpus, comp = _corpus(case, seed)
    index = held.keep(pvs.pvs_build(corpus), pvs.pvs_index_free)
    dead = _deleted(case, seed)
    snap = None
    if dead is not None:
        pvs.pvs_tombstone(index, dead)
        snap = held.keep(pvs.pvs_snapshot_create(index), pvs.pvs_snapshot_free)
    return index, snap, corpus, comp, dead


def prepare(case, seed):
    kind, held = case["kind"], _Held()
    s = dict(case=case, held=held)
    if kind == "query":
        s["index"], s["snap"], corpus, _, _ = _indexed(case, seed, held)
        s["query"] = _queries(case, seed, 1)[0][0].contiguous()
    elif kind == "serve":
        index, _, corpus, _, _ = _indexed(case, seed, held)
        queries, _ = _queries(case, seed, case["requests"])
        s["executor"] = held.keep(pvs.pvs_executor_create(index, 8), pvs.pvs_executor_destroy)
        pvs.pvs_executor_set_group(s["executor"], 8)
        shape = (case["requests"], case["ranks"])
        if case["host"]:
            s["queries"] = queries.cpu().pin_memory()
            s["ids"] = torch.empty(shape, dtype=torch.int64).pin_memory()
            s["scores"] = torch.empty(shape, dtype=torch.float32).pin_memory()
        else:
            s["queries"] = queries
            s["ids"] = torch.empty(shape, dtype=torch.int64, device=DEVICE)
            s["scores"] = torch.empty(shape, dtype=torch.float32, device=DEVICE)
    elif kind == "batch":
        s["index"], _, corpus, _, _ = _indexed(case, seed, held)
        s["queries"], _ = _queries(case, seed, case["queries"])
        shape = (case["pulls"], case["queries"], case["ranks"] // case["pulls"])
        s["ids"] = torch.empty(shape, dtype=torch.int64, device=DEVICE)
        s["scores"] = torch.empty(shape, dtype=torch.float32, device=DEVICE)
    elif kind == "fuse":
        s["index"], s["snap"], corpus, _, dead = _indexed(case, seed, held)
        s["query"] = _queries(case, seed, 1)[0][0].contiguous()
        s["ranking"] = _sparse_ranking(case, seed, corpus, s["query"], dead)
    elif kind == "hybrid":
        s["index"], _, corpus, comp, _ = _indexed(case, seed, held)
        query, topic = _queries(case, seed, 1)
        s["query"] = query[0].contiguous()
        post = _postings(case["n"], seed, comp, case["components"])
        s["sparse"] = held.keep(pvs.pbm_build(*post, case["n"]), pvs.pbm_index_free)
        s["terms"] = _sparse_terms(case, seed, post[0], int(topic[0]))
        s["weights"] = np.ones(s["terms"].size, np.float32)
    elif kind == "sparse":
        corpus = None
        post = _postings(case["n"], seed)
        s["sparse"] = held.keep(pvs.pbm_build(*post, case["n"]), pvs.pbm_index_free)
        s["terms"] = _sparse_terms(case, seed, post[0])
        s["weights"] = np.ones(s["terms"].size, np.float32)
    elif kind == "rerank":
        corpus = None
        s["vecs"], _ = _corpus(case, seed)
        s["query"] = _queries(case, seed, 1)[0][0].contiguous()
        s["ids"] = torch.empty(case["top"], dtype=torch.int64, device=DEVICE)
        s["scores"] = torch.empty(case["top"], dtype=torch.float32, device=DEVICE)
    elif kind == "build":
        s["vecs"], _ = _corpus(case, seed)
        s["query"] = _queries(case, seed, 1)[0][0].contiguous()
        return s
    else:
        raise ValueError(kind)
    del corpus
    torch.cuda.empty_cache()   # the library allocates its own device memory
    return s


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

def _paged(next_page, cursor, ranks, page):
    ids, scores = [], []
    for first in range(0, ranks, page):
        i, sc, status = next_page(cursor, min(page, ranks - first))
        ids.append(i)
        scores.append(sc)
        if status == pvs.PVS_EXHAUSTED:
            break
    return dict(ids=np.concatenate(ids), scores=np.concatenate(scores))


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "query":
        cursor = pvs.pvs_cursor_open(s["index"], s["query"], s["snap"])
        try:
            return _paged(pvs.pvs_next, cursor, case["ranks"], case["page"])
        finally:
            pvs.pvs_cursor_close(cursor)
    if kind == "serve":
        if case["host"]:
            ids, scores, n_out, status, _ = pvs.pvs_executor_run(
                s["executor"], s["queries"], case["ranks"], case["page"], ids=s["ids"],
                scores=s["scores"])
            return dict(ids=ids, scores=scores, n_out=n_out, status=status)
        n_out, status, _ = pvs.pvs_executor_run_device(
            s["executor"], s["queries"], case["ranks"], case["page"], s["ids"], s["scores"])
        return dict(ids=s["ids"], scores=s["scores"], n_out=n_out, status=status)
    if kind == "batch":
        cursors = pvs.pvs_cursor_open_batch(s["index"], s["queries"], case["ranks"])
        try:
            n_out = [pvs.pvs_next_batch(cursors, case["ranks"] // case["pulls"], s["ids"][p],
                                        s["scores"][p]) for p in range(case["pulls"])]
            status = pvs.pvs_cursor_sync_batch(cursors)
        finally:
            pvs.pvs_cursor_close_batch(cursors)
        return dict(ids=s["ids"], scores=s["scores"], n_out=np.stack(n_out), status=status)
    if kind == "fuse":
        cursor = pvs.pvs_cursor_open(s["index"], s["query"], s["snap"])
        try:
            ids, fused, _ = pvs.eahr_topk(cursor, s["ranking"], K=K, k=60,
                                          form=pvs.EAHR_NUMERATOR,
                                          policy=pvs.EAHR_POLICY_ADAPTIVE)
        finally:
            pvs.pvs_cursor_close(cursor)
        return dict(ids=ids, fused=fused)
    if kind == "hybrid":
        dense = pvs.pvs_cursor_open(s["index"], s["query"])
        sparse = pvs.pbm_cursor_open(s["sparse"], s["terms"], s["weights"])
        try:
            ids, fused, _ = pvs.eahr_topk_pbm(dense, sparse, K=K, k=60, form=pvs.EAHR_NUMERATOR,
                                              policy=pvs.EAHR_POLICY_ADAPTIVE)
        finally:
            pvs.pbm_cursor_close(sparse)
            pvs.pvs_cursor_close(dense)
        return dict(ids=ids, fused=fused)
    if kind == "sparse":
        cursor = pvs.pbm_cursor_open(s["sparse"], s["terms"], s["weights"])
        try:
            return _paged(pvs.pbm_next, cursor, case["ranks"], case["page"])
        finally:
            pvs.pbm_cursor_close(cursor)
    if kind == "rerank":
        pvs.pvs_rank_exact_noalloc(s["query"], s["vecs"], case["top"], s["ids"], s["scores"])
        return dict(ids=s["ids"], scores=s["scores"])
    index = pvs.pvs_build(s["vecs"])
    try:
        cursor = pvs.pvs_cursor_open(index, s["query"])
        try:
            return _paged(pvs.pvs_next, cursor, 20, 20)
        finally:
            pvs.pvs_cursor_close(cursor)
    finally:
        pvs.pvs_index_free(index)


# ---------------------------------------------------------------------------
# what a pass cannot do without, and what it must give
# ---------------------------------------------------------------------------

def _postings_read(case):
    """Bytes of the query terms' postings (4-byte id, 4-byte impact each), as
    expected of terms drawn in proportion to their postings."""
    topical = case["kind"] == "hybrid"
    own = (case["terms"] + 1) // 2 if topical else 0
    tokens = case["n"] * TOKENS * ((1.0 - TOPIC_SHARE) if topical else 1.0)
    h = math.log((VOCAB + SKIP) / SKIP)
    mean_df = tokens * (1.0 / SKIP - 1.0 / (VOCAB + SKIP)) / (h * h)
    own_df = case["n"] / max(1, case.get("components", 1)) * TOKENS * TOPIC_SHARE / TOPIC_TERMS
    return 8.0 * ((case["terms"] - own) * mean_df + own * own_df)


def work(case):
    """The codes with their three parameters once per pass (however many
    queries share it), the fp32 rows of the ranks delivered and the outputs;
    two operations per code and query.  Building reads the fp32 rows and
    writes them back with their codes and parameters."""
    kind, n, dim = case["kind"], case["n"], case.get("dim", 0)
    codes = n * (dim + 12)
    if kind in ("query", "serve", "batch"):
        nq = case.get("requests", case.get("queries", 1))
        ranks = nq * min(case["ranks"], n)
        return dict(bytes=codes + ranks * (4 * dim + 12) + 4 * nq * dim, flops=2 * nq * n * dim)
    if kind in ("fuse", "hybrid"):
        sparse = _postings_read(case) if kind == "hybrid" else 8 * K
        return dict(bytes=codes + K * (4 * dim + 16) + sparse, flops=2 * n * dim)
    if kind == "sparse":
        return dict(bytes=_postings_read(case) + 12 * case["ranks"],
                    flops=_postings_read(case) / 4)
    if kind == "rerank":
        return dict(bytes=4 * (n + 1) * dim + 12 * case["top"], flops=2 * n * dim)
    return dict(bytes=n * (9 * dim + 12) + codes, flops=8 * n * dim)


def tolerance(case):
    """Ranks are exact and every score is the correctly rounded float32 of the
    exact value (of the stated float32 sum for the sparse channel), so another
    correct implementation gives the same bits."""
    return "exact"


def _ranked(corpus, queries, ranks, dead):
    """Binary64 scores of each query's first ranks, best first, and their ids."""
    dead = None if dead is None else torch.from_numpy(dead).to(DEVICE)
    n = corpus.shape[0]
    count = min(n, ranks + 256)   # float32 scores are off by far less than 256 ranks here
    ids, scores = [], []
    for q in queries:
        approx = corpus @ q
        if dead is not None:
            approx[dead] = -math.inf
        top = torch.topk(approx, count).indices
        s = corpus[top].double() @ q.double()
        if dead is not None:
            s[torch.isinf(approx[top])] = -math.inf
        order = np.lexsort((top.cpu().numpy(), -s.float().cpu().numpy()))[:ranks]
        order = torch.from_numpy(order).to(DEVICE)
        ids.append(top[order])
        scores.append(s[order])
    return torch.stack(ids), torch.stack(scores)


def _sparse_scores(post, terms, n):
    off, docs, imps = post
    s = torch.zeros(n, dtype=torch.float64, device=DEVICE)
    for t in terms:
        a, b = int(off[t]), int(off[t + 1])
        s[docs[a:b].long()] += imps[a:b].double()
    return s


def exact(case, seed):
    """Scores in binary64 (ranks of equal float32 scores by id).  The fused
    lists are left out: their values are rationals of integer ranks, and
    which of them a pass reports is part of its contract, not a rounding."""
    kind = case["kind"]
    if kind in ("fuse", "hybrid"):
        return None
    if kind == "sparse":
        post = _postings(case["n"], seed)
        s = _sparse_scores(post, _sparse_terms(case, seed, post[0]), case["n"])
        top = torch.topk(s, min(case["ranks"], int((s > 0).sum())))
        return dict(ids=None, scores=top.values)
    corpus, _ = _corpus(case, seed)
    nq = case.get("requests", case.get("queries", 1))
    queries, _ = _queries(case, seed, nq)
    ranks = case.get("ranks", case.get("top", 20))
    ids, scores = _ranked(corpus, queries, ranks, _deleted(case, seed))
    if kind in ("query", "rerank", "build"):
        return dict(ids=ids[0], scores=scores[0])
    if kind == "batch":
        shape = (nq, case["pulls"], ranks // case["pulls"])
        ids, scores = (x.reshape(shape).transpose(0, 1).contiguous() for x in (ids, scores))
    return dict(ids=ids, scores=scores, n_out=None, status=None)
