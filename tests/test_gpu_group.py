"""GPU parity of searches with k > 32, whose floors come from a group pass:
corpora with fewer groups than k, strides 1, 2, 3 and more, groups of 8 and of
32, every CTA mode, both lexical forms, two stacked corpora, and scores that
make every group maximum equal."""
import numpy as np
import pytest
import torch

import oracle
from oracle import check
from paper_2608_08340_gb300 import workloads
from paper_2608_08340_gb300.index import Index, search_two

from _gpu import TOL, check_dense, dev_tensor

pytestmark = pytest.mark.gpu


def _rows(rng, n, d):
    return workloads.to_bf16_bits(workloads._normalise(rng.standard_normal((n, d)).astype(np.float32)))


@pytest.mark.parametrize("n,d,q,k,mode", [
    (40, 64, 3, 40, None),           # 5 groups of 8 for k = 40: no floor
    (300, 64, 130, 33, None),        # as many groups as k, about
    (4096, 64, 257, 256, None),      # groups of 8, k = K_MAX
    (8300, 72, 5, 100, "single"),    # stride 1, groups of 8, ragged last tile
    (17000, 64, 300, 64, "dual"),    # stride 1, a dual-mode group pass
    (20000, 64, 1100, 37, None),     # stride 2, CTA pairs
    (20000, 64, 1100, 37, "single"),
    (40000, 64, 40, 50, None),       # stride 3
    (90000, 64, 150, 40, None),      # stride 8: counted floors
])
def test_floors(n, d, q, k, mode):
    rng = np.random.default_rng(n + q + k)
    E, Q = _rows(rng, n, d), _rows(rng, q, d)
    idx = Index(dev_tensor(E))
    idx.force_pair(mode)
    Qd = dev_tensor(Q)
    rows = rng.choice(q, min(q, 150), replace=False)
    for _ in range(2):
        ids, sc = idx.search(Qd, k)
        check_dense(ids, sc, E, Q, k, f"n={n} q={q} k={k} {mode}", rows=np.sort(rows))
    idx.check()


@pytest.mark.parametrize("n,k", [(5000, 40), (70000, 100)])
def test_equal_scores(n, k):
    """Every score reaches the floor: lists compact, the lowest ids win."""
    E = oracle.round_bf16(np.ones((n, 64), np.float32))
    idx = Index(dev_tensor(E))
    ids, sc = idx.search(dev_tensor(oracle.round_bf16(np.ones((5, 64), np.float32))), k)
    assert ids.cpu().tolist() == [list(range(k))] * 5
    assert (sc.cpu().numpy() == 64).all()


@pytest.mark.parametrize("reps,k,q", [(30, 40, 3), (80, 100, 3), (80, 100, 300)])
def test_ties_at_rank_k_with_counted_floors(reps, k, q):
    """1500 distinct rows, each stored `reps` times, a group pass over every
    fourth tile: rank k falls inside a group of equal scores, and the merge,
    which drops keys below the best counted floor, must keep its lowest ids."""
    rng = np.random.default_rng(reps)
    base = _rows(rng, 1500, 128)
    E = np.ascontiguousarray(np.tile(base, (reps, 1)))
    Q = np.ascontiguousarray(base[rng.choice(1500, q, replace=False)])
    scores = oracle.bf16_to_f32(Q).astype(np.float64) @ oracle.bf16_to_f32(base).astype(np.float64).T
    order = np.argsort(-scores, axis=1)
    best = np.take_along_axis(scores, order, axis=1)
    apart = (-np.diff(best[:, :k // reps + 2], axis=1)).min(axis=1) > 10 * TOL
    assert apart.sum() >= q // 2             # only ties within a group are ambiguous there
    want = (order[:, :k // reps + 1, None] + 1500 * np.arange(reps)).reshape(q, -1)[:, :k]
    idx = Index(dev_tensor(E))
    ids, _ = idx.search(dev_tensor(Q), k)
    assert (ids.cpu().numpy()[apart] == want[apart]).all()
    idx.check()


@pytest.mark.parametrize("gather", [False, True])
def test_hybrid(gather):
    w = workloads.config(3, n=9000, batch=70)
    idx = Index(dev_tensor(w.E_data))
    idx.set_sparse(w.doc_indptr, w.doc_terms, w.vocab, w.k1, w.b)
    idx.gather_lexical(gather)
    k = 60
    ids, sc = idx.hybrid_search(dev_tensor(w.Q_data), torch.from_numpy(w.q_indptr),
                                torch.from_numpy(w.q_terms), w.alpha, k)
    o_ids, o_sc, _ = oracle.hybrid_search(w.E_data, w.Q_data, w.doc_indptr, w.doc_terms, w.vocab,
                                          w.q_indptr, w.q_terms, w.alpha, k + 200, w.k1, w.b)
    check.check_topk(ids.cpu().numpy(), sc.cpu().numpy(), o_ids, o_sc, k, TOL, n=w.n,
                     label=f"hybrid gather={gather}")


def test_two_stacked_corpora():
    rng = np.random.default_rng(3)
    A, B, Q = _rows(rng, 5001, 64), _rows(rng, 3002, 64), _rows(rng, 200, 64)
    k = 77
    ids, src, sc = search_two(Index(dev_tensor(A)), Index(dev_tensor(B)), dev_tensor(Q), k)
    stacked = ids + 5001 * (src == 1)
    check_dense(stacked, sc, np.concatenate([A, B]), Q, k, "two")


@pytest.mark.parametrize("q,k", [(1, 256), (130, 100), (1500, 40)])
def test_reserve_covers_the_group_pass(q, k):
    rng = np.random.default_rng(q)
    idx = Index(dev_tensor(_rows(rng, 12000, 64)))
    idx.reserve(q, k)
    before = idx.buffer_bytes()
    for kk in {33, k}:
        idx.search(dev_tensor(_rows(rng, q, 64)), kk)
    assert idx.buffer_bytes() == before


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("few", [False, True])
@pytest.mark.parametrize("q,k", [(3, 5), (40, 12), (100, 30), (40, 50), (300, 200)])
def test_scores_that_are_not_a_number_prove_no_floor(q, k, few, dtype):
    """Hybrid with a dense weight of 0: overflowed products give 0 * inf, not a
    number.  Such chunks are no results, and whole groups of them push no other
    chunk out."""
    n = 4000
    E = np.zeros((n, 64), np.float32)
    bad = np.arange(64, 224) if few else np.arange(64, 3000)
    E[bad] = 3e38
    # Term 1 once in every chunk; its weight falls with the chunk's length, and
    # each group of eight chunks holds one of the shortest.
    lens = 1 + np.arange(n) % 8 * 500 + np.arange(n) // 16
    indptr = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    terms = np.full(indptr[-1], 2, np.int32)
    terms[indptr[:-1]] = 1
    Q = np.ones((q, 64), np.float32)
    if dtype == "bf16":
        E, Q = oracle.round_bf16(E), oracle.round_bf16(Q)
    idx = Index(dev_tensor(E))
    idx.set_sparse(indptr, terms, 8)
    ids, sc = idx.hybrid_search(dev_tensor(Q), torch.arange(q + 1, dtype=torch.int32),
                                torch.ones(q, dtype=torch.int32), 0.0, k)
    want = np.argsort(lens, kind="stable")
    want = want[~np.isin(want, bad)][:k]
    assert ids.cpu().tolist() == [want.tolist()] * q
    assert torch.isfinite(sc).all()
