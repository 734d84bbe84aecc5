"""Performance cases of the retrieval hot path: the calls that a program built
on this package makes, over the sizes that it makes them with.

A case is a dict of plain values:
  kind    "dense"  device queries, exact top-k (with "upsert" rows overwritten
                   first when that is not 0: an index refreshed between batches)
          "host"   the same search with pinned host queries and results
          "two"    one ranking over a knowledge index and a memory index
          "hybrid" dense + BM25 fusion over the whole corpus
          "rerank" dense top-"cand", then the fusion of those candidates
          "embed"  masked mean pool + L2 normalisation of hidden states
  dtype   storage type of the index (embed: of the hidden states)
  n d q k corpus rows, dimension, queries, results; the other keys per kind.

Embeddings are L2-normalised Gaussian directions, or draws around cluster
centres ("clusters" > 0), chunk texts are Zipf(1.1) token bags of 150 to 250
terms over a vocabulary of 30522, queries hold Zipf-drawn terms.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2608_08340_gb300.index import Index, embed_pool, search_two

_DT = {"bf16": torch.bfloat16, "f32": torch.float32}
_VOCAB = 30522
_ZIPF = 1.1
_LEN = (150, 250)
_K1, _B = 1.2, 0.75
# Share of a padded batch's tokens that are real: lengths uniform in [T/4, T].
_REAL = 0.625


def listed():
    return [
        # The smallest call: a small float32 index and a handful of queries.
        dict(name="tiny_f32", kind="dense", dtype="f32", n=1024, d=384, q=16, k=5, clusters=0,
             upsert=0),
        # One user question against 32K chunks: latency of a single query.
        dict(name="one_query", kind="dense", dtype="bf16", n=32768, d=768, q=1, k=5, clusters=0,
             upsert=0),
        # A small serving batch that comes from, and goes back to, host memory.
        dict(name="host_batch", kind="host", dtype="bf16", n=32768, d=768, q=32, k=5, clusters=0),
        # An ordinary serving batch on the device.
        dict(name="batch256", kind="dense", dtype="bf16", n=32768, d=768, q=256, k=5, clusters=0,
             upsert=0),
        # Odd sizes throughout, and more results than one register list holds.
        dict(name="ragged", kind="dense", dtype="bf16", n=50021, d=392, q=300, k=50, clusters=0,
             upsert=0),
        # Bulk search near cluster centres (many near ties), wide rows.
        dict(name="clustered", kind="dense", dtype="bf16", n=32768, d=1024, q=4096, k=10,
             clusters=256, upsert=0),
        # A float32 index (scores are float32 sums) and an ordinary batch.
        dict(name="batch_f32", kind="dense", dtype="f32", n=32768, d=768, q=100, k=10, clusters=0,
             upsert=0),
        # The largest: a million chunks, 4096 of them refreshed before a
        # 2048-query batch that asks for 100 results each.
        dict(name="scale_refresh", kind="dense", dtype="bf16", n=1048576, d=768, q=2048, k=100,
             clusters=0, upsert=4096),
        # Full hybrid retrieval of a scenario's 1024 queries over 32K chunks.
        dict(name="hybrid", kind="hybrid", dtype="bf16", n=32768, d=768, q=1024, k=5, terms=8,
             alpha=0.5),
        # The same scenario with the dense-first policy (top 128, then rerank).
        dict(name="dense_first", kind="rerank", dtype="bf16", n=32768, d=768, q=1024, k=5,
             terms=8, alpha=0.5, cand=128),
        # Knowledge and agent memory in one ranking.
        dict(name="two_indices", kind="two", dtype="bf16", n=32768, m=8192, d=768, q=250, k=8),
        # Embedding tail of a padded ingestion batch.
        dict(name="embed_tail", kind="embed", dtype="bf16", out="bf16", batch=256, tokens=512,
             dim=4096),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["dense", "dense", "dense", "f32", "f32", "host", "two", "hybrid", "hybrid",
                       "rerank", "embed", "embed"])
    if kind == "embed":
        dtype = rng.choice(["bf16", "bf16", "f32"])
        batch, tokens = _log_int(rng, 1, 512), _log_int(rng, 8, 1024)
        dim = 8 * _log_int(rng, 32, 1024 if dtype == "bf16" else 512)
        batch = max(1, min(batch, (1 << 29) // (tokens * dim * (1 if dtype == "bf16" else 2))))
        return dict(kind="embed", dtype=dtype, out=rng.choice(["bf16", "bf16", "f32"]),
                    batch=batch, tokens=tokens, dim=dim)
    d = 8 * rng.randint(8, 160)
    if kind == "f32":
        n, q = _log_int(rng, 1000, 100000), _log_int(rng, 1, 256)
        q = max(1, min(q, int(4e9 / (n * d))))
        return dict(kind="dense", dtype="f32", n=n, d=d, q=q, k=_log_int(rng, 1, 32), clusters=0,
                    upsert=0)
    if kind == "dense":
        n, q = _log_int(rng, 1000, 600000), _log_int(rng, 1, 4096)
        q = max(1, min(q, int(8e11 / (n * d))))
        return dict(kind="dense", dtype="bf16", n=n, d=d, q=q, k=_log_int(rng, 1, 128),
                    clusters=rng.choice([0, 0, 256]), upsert=rng.choice([0, 0, min(n // 4, 1000)]))
    if kind == "host":
        return dict(kind="host", dtype="bf16", n=_log_int(rng, 1000, 100000), d=d,
                    q=_log_int(rng, 1, 512), k=_log_int(rng, 1, 32), clusters=0)
    if kind == "two":
        return dict(kind="two", dtype="bf16", n=_log_int(rng, 1000, 100000),
                    m=_log_int(rng, 100, 20000), d=d, q=_log_int(rng, 1, 1024),
                    k=_log_int(rng, 1, 32))
    n, q = _log_int(rng, 1000, 50000), _log_int(rng, 1, 1200)
    case = dict(kind=kind, dtype="bf16", n=n, d=d, q=q, k=rng.randint(1, 20),
                terms=rng.randint(2, 16), alpha=rng.choice([0.3, 0.5, 0.7]))
    if kind == "rerank":
        case["cand"] = rng.choice([32, 64, 100, 128, 200])
    return case


# ------------------------------------------------------------------ inputs

def _gen(seed, part):
    return torch.Generator(device="cuda").manual_seed(seed * 16 + part)


def _unit(x):
    return x.div_(x.norm(dim=1, keepdim=True))


def _rows(n, d, seed, part, dtype, clusters=0):
    """n unit rows in the index's dtype; with clusters, around shared centres."""
    g = _gen(seed, part)
    centres = None
    if clusters:
        centres = torch.randn(clusters, d, generator=_gen(seed, 15), device="cuda")
    out = torch.empty(n, d, dtype=dtype, device="cuda")
    for lo in range(0, n, 1 << 17):
        hi = min(n, lo + (1 << 17))
        x = torch.randn(hi - lo, d, generator=g, device="cuda")
        if clusters:
            at = torch.randint(clusters, (hi - lo,), generator=g, device="cuda")
            x = x.mul_(0.05).add_(centres[at])
        out[lo:hi] = _unit(x).to(dtype)
    return out


def _zipf(count, g):
    p = torch.arange(1, _VOCAB + 1, dtype=torch.float64, device="cuda").pow(-_ZIPF)
    cdf = torch.cumsum(p, 0) / p.sum()
    u = torch.rand(count, generator=g, device="cuda", dtype=torch.float64)
    return torch.searchsorted(cdf, u, right=True).clamp_(max=_VOCAB - 1).to(torch.int32)


def _bags(n, seed):
    """Token bags of n chunks, CSR on the device: (indptr int32, terms int32)."""
    g = _gen(seed, 6)
    lens = torch.randint(_LEN[0], _LEN[1] + 1, (n,), generator=g, device="cuda")
    indptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(lens, 0, out=indptr[1:])
    return indptr.to(torch.int32), _zipf(int(indptr[-1]), g)


def _query_terms(q, per_query, seed):
    indptr = torch.arange(q + 1, device="cuda", dtype=torch.int32) * per_query
    return indptr, _zipf(q * per_query, _gen(seed, 7))


def _refresh(case, seed):
    """Ids (host int64, distinct) and rows (device) of the upsert batch."""
    g = torch.Generator().manual_seed(seed * 16 + 8)
    ids = torch.randperm(case["n"], generator=g)[:case["upsert"]].numpy().astype(np.int64)
    return ids, _rows(case["upsert"], case["d"], seed, 9, _DT[case["dtype"]], case["clusters"])


def _hidden(case, seed):
    g = _gen(seed, 1)
    b, t, d = case["batch"], case["tokens"], case["dim"]
    x = torch.empty(b, t, d, dtype=_DT[case["dtype"]], device="cuda")
    for i in range(0, b, 32):
        x[i:i + 32] = torch.randn(min(32, b - i), t, d, generator=g, device="cuda")
    lens = torch.randint(max(1, t // 4), t + 1, (b,), generator=g, device="cuda")
    mask = (torch.arange(t, device="cuda")[None] < lens[:, None]).to(torch.uint8)
    return x, mask


def _corpus(case, seed):
    return _rows(case["n"], case["d"], seed, 1, _DT[case["dtype"]], case.get("clusters", 0))


def _queries(case, seed):
    return _rows(case["q"], case["d"], seed, 2, _DT[case["dtype"]], case.get("clusters", 0))


# ------------------------------------------------------------------ the path

def prepare(case, seed):
    kind = case["kind"]
    if kind == "embed":
        x, mask = _hidden(case, seed)
        return dict(kind=kind, x=x, mask=mask, out=_DT[case["out"]])
    corpus = _corpus(case, seed)
    torch.cuda.synchronize()       # an index is made on a stream of its own
    s = dict(kind=kind, k=case["k"], index=Index(corpus), queries=_queries(case, seed))
    if kind == "dense":
        s["refresh"] = _refresh(case, seed) if case["upsert"] else None
    elif kind == "host":
        s["queries"] = s["queries"].cpu().pin_memory()
        s["out"] = (torch.empty(case["q"], case["k"], dtype=torch.int64).pin_memory(),
                    torch.empty(case["q"], case["k"], dtype=torch.float32).pin_memory())
    elif kind == "two":
        corpus = _rows(case["m"], case["d"], seed, 3, _DT[case["dtype"]])
        torch.cuda.synchronize()
        s["memory"] = Index(corpus)
    else:
        indptr, terms = _bags(case["n"], seed)
        s["index"].set_sparse(indptr.cpu().numpy(), terms.cpu().numpy(), _VOCAB, _K1, _B)
        s["terms"] = _query_terms(case["q"], case["terms"], seed)
        s["alpha"] = case["alpha"]
        s["cand"] = max(case.get("cand", 0), case["k"])
    return s


def run(s):
    kind = s["kind"]
    if kind == "embed":
        return embed_pool(s["x"], s["mask"], s["out"])
    if kind == "host":
        return s["index"].search_host(s["queries"], s["k"], out=s["out"])
    if kind == "two":
        return search_two(s["index"], s["memory"], s["queries"], s["k"])
    if kind == "hybrid":
        return s["index"].hybrid_search(s["queries"], *s["terms"], s["alpha"], s["k"])
    if kind == "rerank":
        return s["index"].hybrid_search_dense_first(s["queries"], *s["terms"], s["alpha"],
                                                    s["cand"], s["k"])
    if s["refresh"] is not None:
        s["index"].upsert(*s["refresh"])
    return s["index"].search(s["queries"], s["k"])


def work(case):
    e = 2 if case["dtype"] == "bf16" else 4
    if case["kind"] == "embed":
        real = _REAL * case["batch"] * case["tokens"]
        return {"bytes": real * case["dim"] * e + case["batch"] * case["tokens"] +
                case["batch"] * case["dim"] * (2 if case["out"] == "bf16" else 4),
                "flops": real * case["dim"]}
    n = case["n"] + case.get("m", 0)
    nbytes = (n + case["q"]) * case["d"] * e + case["q"] * case["k"] * 12
    nbytes += 2 * case.get("upsert", 0) * case["d"] * e
    if case["kind"] == "hybrid":
        # the lexical index once: about 100 distinct terms a chunk, 8 bytes each
        nbytes += case["n"] * 100 * 8 + case["q"] * case["terms"] * 4
    if case["kind"] == "rerank":
        nbytes += case["q"] * case["terms"] * (4 + case["cand"] * 4)
    return {"bytes": nbytes, "flops": 2.0 * n * case["q"] * case["d"]}


def tolerance(case):
    if case["kind"] == "embed":
        # float32 sums in another order move a mean by about 1e-7; rounded to
        # bf16, a few values in a hundred thousand then take the neighbouring
        # value (1.3e-5 in the 2-norm for 256 x 512 x 4096, one ulp at most).
        return {"rel": 1e-4, "max": 2e-2} if case["out"] == "bf16" else {"rel": 2e-6, "max": 1e-5}
    if case["dtype"] == "f32":
        # float32 products and sums (5e-8 from 64 bits).
        return {"rel": 5e-7, "max": 2e-6, "differ": 0.01}
    # bf16 products summed by the tensor cores: 2e-6 from 64 bits where scores
    # are near 1 (clusters), 1e-6 and less elsewhere; there 1 id in 100 is at
    # a near tie and may change places.
    return {"rel": 1e-5, "max": 1e-4, "differ": 0.01}


# ---------------------------------------------------------- 64-bit references

def _topk64(E, Q, k):
    """Top-k of Q E^T in float64, over slices of the corpus."""
    Q64 = Q.double()
    best_s = best_i = None
    step = max(4096, (1 << 28) // Q.shape[0])
    for lo in range(0, E.shape[0], step):
        s = Q64 @ E[lo:lo + step].double().T
        v, i = torch.topk(s, min(k, s.shape[1]), dim=1)
        i = i + lo
        if best_s is not None:
            v, i = torch.cat([best_s, v], 1), torch.cat([best_i, i], 1)
            v, at = torch.topk(v, min(k, v.shape[1]), dim=1)
            i = i.gather(1, at)
        best_s, best_i = v, i
    return best_i, best_s


def _bm25_64(case, seed):
    """BM25 of every (query, chunk) pair in float64 (q x n)."""
    n = case["n"]
    indptr, terms = _bags(n, seed)
    lens = (indptr[1:] - indptr[:-1]).long()
    doc = torch.repeat_interleave(torch.arange(n, device="cuda"), lens)
    pair, tf = torch.unique(doc * _VOCAB + terms.long(), return_counts=True)
    doc, term = pair // _VOCAB, pair % _VOCAB
    df = torch.bincount(term, minlength=_VOCAB).double()
    idf = torch.log(1.0 + (n - df + 0.5) / (df + 0.5))
    tf, dl = tf.double(), lens.double()
    w = idf[term] * tf * (_K1 + 1) / (tf + _K1 * (1 - _B + _B * dl[doc] / dl.mean()))
    W = torch.sparse_coo_tensor(torch.stack([doc, term]), w, (n, _VOCAB)).to_sparse_csr()
    qp, qt = _query_terms(case["q"], case["terms"], seed)
    owner = torch.arange(case["q"], device="cuda").repeat_interleave(case["terms"])
    counts = torch.zeros(_VOCAB, case["q"], dtype=torch.float64, device="cuda")
    counts.index_put_((qt.long(), owner), torch.ones_like(owner, dtype=torch.float64),
                      accumulate=True)
    return (W @ counts).T.contiguous()


def exact(case, seed):
    kind = case["kind"]
    if kind == "embed":
        x, mask = _hidden(case, seed)
        out = torch.empty(case["batch"], case["dim"], dtype=torch.float64, device="cuda")
        for i in range(case["batch"]):
            m = x[i][mask[i].bool()].double().mean(0)
            out[i] = m / m.norm()
        return out
    E, Q = _corpus(case, seed), _queries(case, seed)
    if kind == "two":
        E = torch.cat([E, _rows(case["m"], case["d"], seed, 3, _DT[case["dtype"]])])
        ids, s = _topk64(E, Q, case["k"])
        second = ids >= case["n"]
        return torch.where(second, ids - case["n"], ids), second.to(torch.int32), s
    if kind in ("hybrid", "rerank"):
        a = case["alpha"]
        lex = _bm25_64(case, seed)
        if kind == "hybrid":
            top = lex.amax(1, keepdim=True)
            lex = torch.where(top > 0, lex / top, torch.zeros_like(lex))
            s, ids = torch.topk(a * (Q.double() @ E.double().T) + (1 - a) * lex, case["k"], dim=1)
            return ids, s
        cand, dense = _topk64(E, Q, max(case["cand"], case["k"]))
        lex = lex.gather(1, cand)
        top = lex.amax(1, keepdim=True)
        lex = torch.where(top > 0, lex / top, torch.zeros_like(lex))
        s, at = torch.topk(a * dense + (1 - a) * lex, case["k"], dim=1)
        return cand.gather(1, at), s
    if case.get("upsert", 0):
        ids, rows = _refresh(case, seed)
        E[torch.from_numpy(ids).cuda()] = rows
    return _topk64(E, Q, case["k"])
