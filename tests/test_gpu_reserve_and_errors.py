"""Two guarantees of the index around its kernels.

reserve: after oprag_index_reserve(q_max, k_max) a search of up to q_max
queries and k_max results allocates nothing (its scratch, the group pass of
k > 32 and the shared per-query bounds were sized and cleared there).

bounded waits: every barrier wait of the search kernels gives up after a spin
limit, records a device error, drains and returns.  A test hook
shortens the limit so that the waits of a real search run out; the index then
reports OPRAG_ERR_DEVICE once, and the next search with the normal limit is
exact again."""
import time

import numpy as np
import pytest
import torch

from paper_2608_08340_gb300 import workloads
from paper_2608_08340_gb300._lib import OpragError
from paper_2608_08340_gb300.index import Index

from _gpu import check_dense, dev_tensor

pytestmark = pytest.mark.gpu


def test_reserve_covers_later_searches():
    # 40000 rows: 313 corpus tiles of 128, so k = 100 runs a group pass
    w = workloads.config(1, n=40000, batch=256)
    idx = Index(dev_tensor(w.E_data))
    idx.reserve(256, 100)
    before = idx.buffer_bytes()
    assert before["scratch"] > 0 and before["bounds"] >= 256 * 8
    Q = dev_tensor(w.Q_data)
    idx.enable_timing(True)
    for k in (5, 16, 32, 100):
        for q in (1, 100, 256):
            ids, sc = idx.search(Q[:q], k)
            t = idx.last_timing()
            if k == 100 and q == 256:
                assert t["sample_ms"] > 0.0          # the group pass ran
                check_dense(ids, sc, w.E_data, w.Q_data[:q], k, "reserved k=100",
                            rows=np.arange(0, 256, 37))
    idx.check()
    assert idx.buffer_bytes() == before


@pytest.mark.parametrize("q,mode", [(64, "single"), (256, "dual")])
def test_bounded_wait_gives_up_and_the_index_recovers(q, mode):
    w = workloads.config(1, n=8192, batch=q)
    idx = Index(dev_tensor(w.E_data))
    idx.force_pair(mode)
    Q = dev_tensor(w.Q_data)
    ref_ids, ref_sc = idx.search(Q, 5)
    idx.check()
    idx.set_wait_limit(1)                 # every wait that is not already complete gives up
    idx.search(Q, 5)
    torch.cuda.synchronize()              # the kernel returned: the context is usable
    with pytest.raises(OpragError) as err:
        idx.check()
    assert err.value.code == -6
    idx.check()                           # reported once, then cleared
    idx.set_wait_limit(0)
    ids, sc = idx.search(Q, 5)
    idx.check()
    assert idx.last_launch["tiles"] == (2 if mode == "dual" else 1)
    assert torch.equal(ids, ref_ids) and torch.equal(sc, ref_sc)
    check_dense(ids, sc, w.E_data, w.Q_data, 5, f"after abort ({mode})")
    idx.close()


# Every kernel with bounded waits: the fp32 search over many K blocks with ring
# stages whose number does not divide the warps' turns, the small-batch kernel
# with its merge inside (a CTA counter that has to return to zero) and behind
# it, the group pass, and the hybrid search's copies of the BM25 block.
@pytest.mark.parametrize("limit", [1, 2500])    # the first wait, or one in mid-run
@pytest.mark.parametrize("kind,d,q,k", [
    ("f32", 768, 100, 10), ("f32", 768, 33, 5), ("f32", 104, 20, 40), ("f32", 1000, 7, 20),
    ("bf16", 768, 3, 5), ("bf16", 768, 30, 16), ("bf16", 256, 150, 60),
    ("hybrid", 768, 20, 5), ("hybrid", 768, 300, 5), ("hybrid", 256, 150, 40),
])
def test_every_kernel_gives_up_in_time_and_the_index_recovers(kind, d, q, k, limit):
    rng = np.random.default_rng(d + q)
    n = 40000
    E = torch.from_numpy(rng.standard_normal((n, d)).astype(np.float32)).cuda()
    Q = torch.from_numpy(rng.standard_normal((q, d)).astype(np.float32)).cuda()
    if kind != "f32":
        E, Q = E.bfloat16(), Q.bfloat16()
    torch.cuda.synchronize()
    idx = Index(E)
    if kind == "hybrid":
        terms = rng.integers(0, 50, n * 6).astype(np.int32)
        idx.set_sparse(np.arange(n + 1, dtype=np.int32) * 6, terms, 50)
        q_ptr = torch.arange(q + 1, dtype=torch.int32, device="cuda") * 3
        q_terms = torch.from_numpy(rng.integers(0, 50, 3 * q).astype(np.int32)).cuda()
        search = lambda: idx.hybrid_search(Q, q_ptr, q_terms, 0.5, k)    # noqa: E731
    else:
        search = lambda: idx.search(Q, k)                                # noqa: E731
    ref_ids, ref_sc = search()
    idx.check()
    for _ in range(3):
        idx.set_wait_limit(limit)
        start = time.perf_counter()
        search()
        torch.cuda.synchronize()          # the kernels returned: the context is usable
        # nothing waited for the default limit of about a second
        assert time.perf_counter() - start < 0.5
        if limit == 1:
            with pytest.raises(OpragError) as err:
                idx.check()
            assert err.value.code == -6
        else:
            try:
                idx.check()
            except OpragError as e:
                assert e.code == -6
        idx.set_wait_limit(0)
        ids, sc = search()
        idx.check()
        assert torch.equal(ids, ref_ids) and torch.equal(sc, ref_sc)
    idx.close()
