"""GPU parity of the BM25 pass (one warp per query and 1024-chunk tile) at its
edges: corpora around the tile size, batches below and above the number of
queries from which a CTA looks terms up and stages dense rows for all, queries longer than one round
of 32 terms, corpora without dense terms and with more dense terms than the
shared memory holds, terms with more postings than one batch of loads."""
import numpy as np
import pytest
import torch

import oracle
from oracle import check
from paper_2608_08340_gb300 import workloads
from paper_2608_08340_gb300.index import Index

from _gpu import TOL, dev_tensor

pytestmark = pytest.mark.gpu


def _check(n, q, vocab, zipf, terms, alpha, k=7, lens=(20, 60), seed=1):
    w = workloads.make_dense("bm", n, 64, q, k, "bf16", seed)
    workloads.add_sparse(w, seed, vocab=vocab, s=zipf, len_lo=lens[0], len_hi=lens[1],
                         terms_per_query=terms)
    idx = Index(dev_tensor(w.E_data))
    idx.set_sparse(w.doc_indptr, w.doc_terms, vocab, w.k1, w.b)
    args = (dev_tensor(w.Q_data), torch.from_numpy(w.q_indptr), torch.from_numpy(w.q_terms), alpha)
    o_ids, o_sc, _ = oracle.hybrid_search(w.E_data, w.Q_data, w.doc_indptr, w.doc_terms, vocab,
                                          w.q_indptr, w.q_terms, alpha, min(n, k + 200), w.k1, w.b)
    for gather in (False, True):
        idx.gather_lexical(gather)
        ids, sc = idx.hybrid_search(*args, k)
        check.check_topk(ids.cpu().numpy(), sc.cpu().numpy(), o_ids, o_sc, k, TOL, n=n,
                         label=f"n={n} q={q} vocab={vocab} terms={terms} gather={gather}")
    idx.gather_lexical(False)
    if n <= 256:                # every chunk a candidate: the rerank sums alike
        r_ids, r_sc = idx.hybrid_search_dense_first(*args, n, k)
        h_ids, h_sc = idx.hybrid_search(*args, k)
        assert torch.equal(r_ids, h_ids) and torch.equal(r_sc, h_sc)


@pytest.mark.parametrize("n,q", [(10, 1), (250, 40), (1023, 3), (1024, 9), (1025, 200), (5001, 7)])
def test_tile_and_batch_edges(n, q):
    _check(n, q, vocab=500, zipf=1.1, terms=5, alpha=0.3)


def test_long_queries_span_several_rounds():
    _check(200, 12, vocab=300, zipf=1.0, terms=70, alpha=0.2)


def test_no_dense_terms():
    _check(3000, 30, vocab=5000, zipf=0.2, terms=6, alpha=0.5)


def test_more_dense_terms_than_staged():
    _check(2100, 60, vocab=90, zipf=0.1, terms=9, alpha=0.4, lens=(150, 250))


def test_postings_longer_than_a_batch_of_loads():
    # terms in up to half of the chunks: hundreds of postings per tile
    _check(4000, 20, vocab=120, zipf=0.3, terms=6, alpha=0.4, lens=(30, 60))


# More than 160 queries: the terms of a tile's queries are looked up together
# (up to 2048 of them), the dense rows copied to shared memory.
@pytest.mark.parametrize("n,vocab,zipf,terms,lens", [
    (1024, 500, 1.1, 5, (20, 60)),
    (300, 300, 1.0, 70, (20, 60)),
    (3000, 5000, 0.2, 6, (20, 60)),
    (2100, 90, 0.1, 9, (150, 250)),
    (4000, 120, 0.3, 6, (30, 60)),
])
def test_many_queries(n, vocab, zipf, terms, lens):
    _check(n, 161, vocab, zipf, terms, alpha=0.3, lens=lens)


@pytest.mark.parametrize("n", [1000, 1025, 30000, 200000])
def test_a_query_scores_the_same_in_any_batch(n):
    w = workloads.make_dense("bm", n, 64, 200, 9, "bf16", 2)
    workloads.add_sparse(w, 2, vocab=900, s=1.0, len_lo=10, len_hi=30, terms_per_query=7)
    idx = Index(dev_tensor(w.E_data))
    idx.set_sparse(w.doc_indptr, w.doc_terms, 900, w.k1, w.b)
    Q, ptr, terms = dev_tensor(w.Q_data), torch.from_numpy(w.q_indptr), torch.from_numpy(w.q_terms)
    ids, sc = idx.hybrid_search(Q, ptr, terms, 0.0, 9)
    for q in (1, 19, 160, 161):
        i, s = idx.hybrid_search(Q[:q], ptr[:q + 1], terms, 0.0, 9)
        assert torch.equal(i, ids[:q]) and torch.equal(s, sc[:q])
