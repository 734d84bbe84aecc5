"""GPU parity of the merges.  Head by head, k above the prefetched keys: top-k
lists drawn from one partial list (every key refetched), spread evenly, and
short of keys.  Unsorted lists (k > 32): buffers that are cut, ranked and empty."""
import numpy as np
import pytest

import oracle
from paper_2608_08340_gb300.index import Index

from _gpu import dev_tensor

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,path", [("f32", None), ("bf16", "simt"), ("bf16", "tc")])
@pytest.mark.parametrize("k", [7, 17, 32, 100, 256])
@pytest.mark.parametrize("spread", [False, True])
def test_skewed_lists(dtype, path, k, spread):
    n, q = 20000, 5
    score = np.zeros(n, np.float32)
    at = np.arange(256) * 78 if spread else 9000 + np.arange(256)
    score[at] = 256 - np.arange(256)              # exact in bf16
    E = np.zeros((n, 64), np.float32)
    E[:, 3] = score
    Q = np.zeros((q, 64), np.float32)
    Q[:, 3] = 2.0 ** np.arange(q)
    if dtype == "bf16":
        E, Q = oracle.round_bf16(E), oracle.round_bf16(Q)
    idx = Index(dev_tensor(E))
    if path:
        idx.force_path(path)
    ids, sc = idx.search(dev_tensor(Q), k)
    assert ids.cpu().tolist() == [at[:k].tolist()] * q
    assert (sc.cpu().numpy() == (2.0 ** np.arange(q))[:, None] * score[at[:k]][None]).all()


def test_fewer_rows_than_lists_hold():
    E = np.zeros((300, 32), np.float32)
    E[:, 0] = np.arange(300)
    ids, _ = Index(dev_tensor(E)).search(dev_tensor(np.ones((3, 32), np.float32)), 256)
    assert ids.cpu().tolist() == [list(range(299, 43, -1))] * 3


@pytest.mark.parametrize("q", [3, 130, 1520, 1521])      # four and two warps a query
@pytest.mark.parametrize("k", [33, 64, 112, 113, 200, 256])
def test_unsorted_lists(q, k):
    """k > 32: rows in the order of their scores fill and cut the merge's
    buffer (queries of the other sign find them in the reverse order); scores
    are row numbers, exact in bf16 halves."""
    n = 20011
    E = np.zeros((n, 64), np.float32)
    E[:, 3], E[:, 40] = np.arange(n) // 256, np.arange(n) % 256
    scale = 2.0 ** (np.arange(q) % 8) * np.where(np.arange(q) % 3 == 1, -1, 1)
    Q = np.zeros((q, 64), np.float32)
    Q[:, 3], Q[:, 40] = 256 * scale, scale
    idx = Index(dev_tensor(oracle.round_bf16(E)))
    ids, sc = idx.search(dev_tensor(oracle.round_bf16(Q)), k)
    best = np.where(scale[:, None] > 0, n - 1 - np.arange(k)[None], np.arange(k)[None])
    assert (ids.cpu().numpy() == best).all()
    assert (sc.cpu().numpy() == scale[:, None] * best).all()


@pytest.mark.parametrize("q", [2, 1600])
@pytest.mark.parametrize("n,k", [(60, 60), (300, 256), (9000, 256)])
def test_unsorted_lists_of_equal_scores(n, k, q):
    E = oracle.round_bf16(np.ones((n, 64), np.float32))
    ids, sc = Index(dev_tensor(E)).search(dev_tensor(oracle.round_bf16(np.ones((q, 64), np.float32))), k)
    assert (ids.cpu().numpy() == np.arange(k)[None]).all()
    assert (sc.cpu().numpy() == 64).all()
