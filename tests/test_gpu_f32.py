"""GPU parity of the fp32 search (register-tiled FMA kernel) at the edges of
its tile shapes: query counts around every tile size, corpora around the tile
height and the slice count, d around the 32-float K block, k around the list
lengths; ties that fill the candidate buffers; the fused hybrid form."""
import numpy as np
import pytest
import torch

import oracle
from oracle import check
from paper_2608_08340_gb300 import workloads
from paper_2608_08340_gb300.index import Index

from _gpu import TOL, check_dense, dev_tensor

pytestmark = pytest.mark.gpu


# fp32 error bound of a score of unit vectors (the sum of |products| is at most
# 1), in units of 2^-24: a chain of at most eight products, three joins, the
# compensated sum (two, and terms of d / 32 times 2^-24 that one more covers).
BOUND = (8 + 3 + 3) * 2.0 ** -24


@pytest.mark.parametrize("n,d,q,k", [
    (1, 8, 1, 1),               # one row, one query, a quarter of a K block
    (17, 32, 4, 17),            # k = n, one K block, TM = 1
    (255, 40, 5, 5),            # TM = 2, a partial second K block
    (3000, 64, 31, 32),         # TM = 8 of 4, the last k of 32-key lists
    (40000, 72, 32, 5),         # several tiles a slice
    (4097, 96, 33, 16),         # TY = 8, TM = 5
    (5000, 128, 64, 33),        # k > 32: query tiles of 32
    (33000, 200, 64, 32),       # TY = 8, TM = 8, k = W
    (9000, 136, 65, 16),        # TY = 16, TM = 5, k = W
    (9000, 136, 65, 32),        # floors from all 32 scores of a warp
    (70000, 24, 100, 10),       # d below one K block, many tiles a slice
    (2000, 384, 128, 1),
    (2000, 264, 129, 8),        # two tiles of 80
    (300, 64, 700, 100),        # k > 32 with many query tiles
    (3000, 512, 3, 256),        # K_MAX
])
def test_tile_edges(n, d, q, k):
    rng = np.random.default_rng(n + d + q + k)
    E = workloads._normalise(rng.standard_normal((n, d)).astype(np.float32))
    Q = workloads._normalise(rng.standard_normal((q, d)).astype(np.float32))
    idx = Index(dev_tensor(E))
    Qd = dev_tensor(Q)
    for _ in range(2):          # the second search reuses the shared bounds
        ids, sc = idx.search(Qd, k)
        check_dense(ids, sc, E, Q, k, f"f32 n={n} d={d} q={q} k={k}")
        i = ids.cpu().numpy()
        want = np.einsum("qkd,qd->qk", E.astype(np.float64)[i], Q.astype(np.float64))
        assert np.abs(sc.cpu().numpy() - want).max() <= BOUND


def _lane_sums(a, b):
    """Inner products of the rows as 32 lanes form them: lane l sums the groups
    of four products l, l + 32, ... in one chain, then the lanes add up in pairs
    (fused multiply-adds through float64)."""
    m, d = a.shape
    lanes = np.zeros((m, 32), np.float32)
    for g in range(d // 4):
        for e in range(4 * g, 4 * g + 4):
            lanes[:, g % 32] = a[:, e].astype(np.float64) * b[:, e] + lanes[:, g % 32]
    for o in (16, 8, 4, 2, 1):
        lanes = lanes + lanes[:, np.arange(32) ^ o]
    return lanes[:, 0]


@pytest.mark.parametrize("q", [16, 50, 100])        # the three tile shapes
@pytest.mark.parametrize("d", [16, 32, 64, 128, 136, 1280, 8192])
def test_error_is_no_larger_than_of_lane_sums(d, q):
    """The root mean square error of the best scores against 64 bits, next to
    the sums of the streaming kernel for bf16 indices.  At d = 16 the two have
    the same chains and joins; 3000 scores then differ by 2 % at most."""
    rng = np.random.default_rng(d)
    E = workloads._normalise(rng.standard_normal((6000, d)).astype(np.float32))
    Q = workloads._normalise(rng.standard_normal((q, d)).astype(np.float32))
    k = 3000 // q
    ids, sc = Index(dev_tensor(E)).search(dev_tensor(Q), k)
    a, b = E[ids.cpu().numpy().ravel()], np.repeat(Q, k, axis=0)
    exact = np.einsum("md,md->m", a.astype(np.float64), b.astype(np.float64))
    err = np.sqrt(np.mean((sc.cpu().numpy().ravel() / exact - 1) ** 2))
    lane = np.sqrt(np.mean((_lane_sums(a, b) / exact - 1) ** 2))
    assert err <= 1.04 * lane, (err, lane)
    assert np.abs(sc.cpu().numpy().ravel() - exact).max() <= BOUND


@pytest.mark.parametrize("q,k", [(3, 7), (40, 20), (90, 16), (20, 100)])
def test_equal_scores_fill_every_buffer(q, k):
    """Every row reaches the floor, so every tile compacts every buffer."""
    E = np.ones((20000, 16), np.float32)
    idx = Index(dev_tensor(E))
    ids, sc = idx.search(dev_tensor(np.ones((q, 16), np.float32)), k)
    assert ids.cpu().tolist() == [list(range(k))] * q
    assert (sc.cpu().numpy() == 16).all()


def test_rising_scores_replace_every_candidate():
    """Scores rise with the id: each tile displaces all that came before."""
    n = 30000
    E = np.zeros((n, 8), np.float32)
    E[:, 0] = np.arange(n)
    Q = np.zeros((70, 8), np.float32)
    Q[:, 0] = 1 + np.arange(70)
    ids, sc = Index(dev_tensor(E)).search(dev_tensor(Q), 10)
    assert ids.cpu().tolist() == [list(range(n - 1, n - 11, -1))] * 70
    assert (sc.cpu().numpy() == (1 + np.arange(70))[:, None] *
            np.arange(n - 1, n - 11, -1)[None]).all()


@pytest.mark.parametrize("q", [3, 40, 100])        # the three tile shapes
@pytest.mark.parametrize("d", [32, 64, 256, 1000])
@pytest.mark.parametrize("k", [5, 40])
def test_overflowing_scores_keep_their_infinity(q, d, k):
    """Finite rows whose product with a query passes the fp32 range rank first,
    whether the sum overflows in the first, a middle or the last K block, and a
    partial sum of the other sign that overflows later does not remove them."""
    n = 3000
    rng = np.random.default_rng(d)
    E = rng.standard_normal((n, d)).astype(np.float32)
    Q = np.ones((q, d), np.float32)
    top = [5, 700, 1500, 2999]
    E[top] = 0
    E[5] = 3e38
    E[700, :8] = 3e38
    E[1500, d // 2:d // 2 + 4] = 3e38
    E[2999, -2:] = 3e38
    if d >= 256:                 # both signs, blocks apart
        top.append(2000)
        E[2000] = np.where(np.arange(d) < d // 2, 3e38, -3e38)
    low = 1111
    E[low] = -3e38
    idx = Index(dev_tensor(E))
    ids, sc = idx.search(dev_tensor(Q), k)
    m = min(k, len(top))
    assert ids.cpu()[:, :m].tolist() == [sorted(top)[:m]] * q
    assert torch.isposinf(sc[:, :m]).all() and torch.isfinite(sc[:, m:]).all()
    assert not (ids == low).any()
    rest = np.setdiff1d(np.arange(n), top + [low])
    want = np.sort((E[rest].astype(np.float64).sum(1)))[::-1][:k - m]
    np.testing.assert_allclose(sc.cpu().numpy()[:, m:], np.broadcast_to(want, (q, k - m)),
                               rtol=0, atol=2.0 ** -20 * d)
    idx.check()
    E[:] = 3e38                  # every score overflows: the lowest ids win
    ids, sc = Index(dev_tensor(E)).search(dev_tensor(Q), k)
    assert ids.cpu().tolist() == [list(range(k))] * q and torch.isposinf(sc).all()


@pytest.mark.parametrize("q", [3, 100])
def test_overflowing_scores_in_the_hybrid_search(q):
    n, d = 2000, 96
    rng = np.random.default_rng(q)
    E = rng.standard_normal((n, d)).astype(np.float32)
    E[[3, 1100, 1999]] = 3e38
    E[700] = -3e38
    terms = rng.integers(0, 40, 5 * n).astype(np.int32)
    idx = Index(dev_tensor(E))
    idx.set_sparse(np.arange(n + 1, dtype=np.int32) * 5, terms, 40)
    ids, sc = idx.hybrid_search(dev_tensor(np.ones((q, d), np.float32)),
                                torch.arange(q + 1, dtype=torch.int32),
                                torch.arange(q, dtype=torch.int32) % 40, 0.5, 12)
    assert ids.cpu()[:, :3].tolist() == [[3, 1100, 1999]] * q
    assert torch.isposinf(sc[:, :3]).all() and torch.isfinite(sc[:, 3:]).all()
    assert not (ids == 700).any()


@pytest.mark.parametrize("q", [3, 40, 100])
@pytest.mark.parametrize("n", [20, 30000])
def test_scores_of_minus_infinity_are_no_results(q, n):
    """Up to 32 results, as with a bf16 index; above, they rank last."""
    E = np.full((n, 64), -3e38, np.float32)
    keep = np.linspace(0, n - 1, 7).astype(int)
    E[keep] = 0
    E[keep, 0] = np.arange(7) - 3
    idx = Index(dev_tensor(E))
    Q = dev_tensor(np.ones((q, 64), np.float32))
    low = np.setdiff1d(np.arange(n), keep)
    for k in (5, 12, 20) if n == 20 else (5, 16, 32, 40):
        want = (keep[::-1].tolist() + ([-1] * k if k <= 32 else low.tolist()))[:k]
        ids, sc = idx.search(Q, k)
        assert ids.cpu().tolist() == [want] * q
        assert sc.cpu().tolist() == [([3.0, 2, 1, 0, -1, -2, -3] + [-np.inf] * k)[:k]] * q


@pytest.mark.parametrize("q", [6, 70])
def test_fused_hybrid(q):
    w = workloads.make_dense("f32h", 3000, 64, q, 9, "f32", 7)
    workloads.add_sparse(w, 7)
    idx = Index(dev_tensor(w.E_data))
    idx.set_sparse(w.doc_indptr, w.doc_terms, w.vocab, w.k1, w.b)
    ids, sc = idx.hybrid_search(dev_tensor(w.Q_data), torch.from_numpy(w.q_indptr),
                                torch.from_numpy(w.q_terms), w.alpha, w.k)
    o_ids, o_sc, _ = oracle.hybrid_search(w.E_data, w.Q_data, w.doc_indptr, w.doc_terms, w.vocab,
                                          w.q_indptr, w.q_terms, w.alpha, w.k + 48, w.k1, w.b)
    check.check_topk(ids.cpu().numpy(), sc.cpu().numpy(), o_ids, o_sc, w.k, TOL, n=w.n,
                     label=f"f32 hybrid q={q}")


@pytest.mark.parametrize("q,k", [(1, 256), (40, 32), (130, 5), (500, 16)])
def test_reserve_covers_smaller_batches(q, k):
    rng = np.random.default_rng(q)
    idx = Index(dev_tensor(rng.standard_normal((6000, 32)).astype(np.float32)))
    idx.reserve(q, k)
    before = idx.buffer_bytes()
    for qq in {1, q // 3 + 1, q // 2 + 1, q}:
        for kk in {1, k}:
            idx.search(dev_tensor(rng.standard_normal((qq, 32)).astype(np.float32)), kk)
    assert idx.buffer_bytes() == before
