"""GPU parity of the small-batch search (up to 32 queries, k <= 16) at its
edges: one to many tiles a slice, slices that end inside a tile, query counts
around the MMA widths and the inline merge, k around its limits, ties, and
agreement with the general kernel."""
import numpy as np
import pytest
import torch

import oracle
from paper_2608_08340_gb300 import workloads
from paper_2608_08340_gb300.index import Index

from _gpu import check_dense, dev_tensor

pytestmark = pytest.mark.gpu


def _rows(rng, n, d):
    return workloads.to_bf16_bits(workloads._normalise(rng.standard_normal((n, d)).astype(np.float32)))


@pytest.mark.parametrize("n,d,q,k", [
    (1, 8, 1, 1),              # one row
    (31, 64, 3, 16),           # one CTA, one partial tile
    (5000, 72, 6, 8),          # slices of 33 rows, the last inline merge
    (5000, 72, 7, 8),          # merged by the merge kernel
    (5000, 72, 6, 9),
    (19456, 64, 16, 5),        # 128 rows a CTA: one full tile
    (19457, 64, 17, 5),        # 129: two tiles of 65
    (38912, 64, 32, 10),       # two full tiles
    (39000, 64, 31, 16),       # three tiles: floors and compactions
    (150000, 40, 32, 16),      # eight tiles, the largest batch
    (5000, 64, 33, 16),        # one query too many: the general kernel
    (150000, 40, 1, 3),
])
def test_edges(n, d, q, k):
    rng = np.random.default_rng(n + q + k)
    E, Q = _rows(rng, n, d), _rows(rng, q, d)
    idx = Index(dev_tensor(E))
    Qd = dev_tensor(Q)
    for _ in range(3):          # the CTA counter returns to zero
        ids, sc = idx.search(Qd, k)
        check_dense(ids, sc, E, Q, k, f"small n={n} d={d} q={q} k={k}")
    idx.force_pair("single")
    g_ids, g_sc = idx.search(Qd, k)
    check_dense(g_ids, g_sc, E, Q, k, "general kernel")
    idx.check()


@pytest.mark.parametrize("q,k", [(1, 5), (30, 16)])
def test_equal_and_rising_scores(q, k):
    n = 60000
    Q = oracle.round_bf16(np.ones((q, 64), np.float32))
    idx = Index(dev_tensor(oracle.round_bf16(np.ones((n, 64), np.float32))))
    ids, sc = idx.search(dev_tensor(Q), k)
    assert ids.cpu().tolist() == [list(range(k))] * q
    E = np.zeros((n, 64), np.float32)
    E[:, 0] = np.arange(n) // 256              # exact in bf16, rising, ties of 256
    idx = Index(dev_tensor(oracle.round_bf16(E)))
    ids, sc = idx.search(dev_tensor(Q), k)
    top = (n - 1) // 256 * 256
    assert ids.cpu().tolist() == [list(range(top, top + k))] * q


@pytest.mark.parametrize("n", [20, 30000, 60000])         # one, two and four tiles a slice
@pytest.mark.parametrize("q,k", [(3, 5), (3, 8), (30, 16)])
def test_scores_of_minus_infinity_are_no_results(n, q, k):
    """Finite rows whose score overflows to -inf: as in the general kernel, they
    leave empty results behind the finite scores."""
    E = np.full((n, 64), -3e38, np.float32)
    keep = np.linspace(0, n - 1, 7).astype(int)
    E[keep] = 0
    E[keep, 0] = np.arange(7) - 3
    idx = Index(dev_tensor(oracle.round_bf16(E)))
    Q = dev_tensor(oracle.round_bf16(np.ones((q, 64), np.float32)))
    want = (keep[::-1].tolist() + [-1] * k)[:k]
    for mode in (None, "single"):
        idx.force_pair(mode)
        ids, sc = idx.search(Q, k)
        assert ids.cpu().tolist() == [want] * q
        assert sc.cpu().tolist() == [([3.0, 2, 1, 0, -1, -2, -3] + [-np.inf] * k)[:k]] * q
