"""GPU parity of the head-by-head merge for k above its prefetched keys: top-k
lists drawn from one partial list (every key refetched), spread evenly, and
short of keys."""
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
