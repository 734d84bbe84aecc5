"""The table of where each term's postings enter the tiles of 1024 chunks: with a
large vocabulary its rows have wider cells, and a cell's postings belong to
several tiles.  The same texts under spread-out term ids have the same weights
and sums, so every result is the same to the bit; and the table's memory stays
within 8 bytes per term and 8192 chunks."""
import numpy as np
import pytest
import torch

import oracle
from oracle import check
from paper_2608_08340_gb300.index import Index

from _gpu import TOL, dev_tensor

pytestmark = pytest.mark.gpu


def _texts(n, rng):
    """Bags over 60 terms: common ones, rare ones, and ones in a run of chunks."""
    bags = []
    for i in range(n):
        bag = list(rng.integers(0, 8, 3))                            # in many chunks
        bag += [t for t in range(8, 24) if rng.random() < 0.02]      # 2 % each
        bag += [t for t in range(24, 44) if rng.random() < 4 / n]    # a few chunks
        bag += [t for t in range(44, 59) if (t - 44) * n // 16 <= i < (t - 44) * n // 16 + 5 * t]
        bags.append(bag)                                             # term 59: nowhere
    indptr = np.concatenate([[0], np.cumsum([len(b) for b in bags])]).astype(np.int32)
    return indptr, np.concatenate(bags).astype(np.int32)


@pytest.mark.parametrize("n", [1024, 1025, 20000, 33000])
@pytest.mark.parametrize("q", [5, 200])
def test_wider_cells_give_the_same_bits(n, q):
    rng = np.random.default_rng(n + q)
    E = oracle.round_bf16(rng.standard_normal((n, 64)).astype(np.float32))
    Q = dev_tensor(oracle.round_bf16(rng.standard_normal((q, 64)).astype(np.float32)))
    indptr, terms = _texts(n, rng)
    q_terms = rng.integers(0, 60, 9 * q).astype(np.int32)
    q_ptr = np.arange(q + 1, dtype=np.int32) * 9
    got = []
    for spread, vocab in ((1, 60), (2500, 150000), (20000, 1200000)):
        idx = Index(dev_tensor(E))
        idx.set_sparse(indptr, terms * spread, vocab)
        args = torch.from_numpy(q_ptr).cuda(), torch.from_numpy(q_terms * spread).cuda(), 0.3
        got.append([idx.hybrid_search(Q, *args, 12), idx.hybrid_search(Q, *args, 50),
                    idx.hybrid_search_dense_first(Q, *args, 130, 20),
                    idx.hybrid_search_dense_first(Q, *args, 100, 5)])
        if spread > 1:
            idx.append(dev_tensor(E[:100]))          # rebuilt with the same rule
            idx.hybrid_search(Q, *args, 12)
            idx.check()
        idx.close()
    for other in got[1:]:
        for (ids, sc), (ref_ids, ref_sc) in zip(other, got[0]):
            assert torch.equal(ids, ref_ids) and torch.equal(sc, ref_sc)
    o_ids, o_sc, _ = oracle.hybrid_search(E, Q.view(torch.int16).cpu().numpy().view(np.uint16),
                                          indptr, terms, 60, q_ptr, q_terms, 0.3, 60, 1.2, 0.75)
    check.check_topk(got[0][0][0].cpu().numpy(), got[0][0][1].cpu().numpy(), o_ids, o_sc, 12, TOL,
                     n=n, label="hybrid")


def test_memory_of_a_large_vocabulary():
    n, vocab = 200000, 200000
    idx = Index(torch.zeros(n, 8, dtype=torch.bfloat16, device="cuda"))
    torch.cuda.synchronize()
    free, _ = torch.cuda.mem_get_info()
    rng = np.random.default_rng(0)
    idx.set_sparse(np.arange(n + 1, dtype=np.int32) * 4, rng.integers(0, vocab, 4 * n), vocab)
    used = free - torch.cuda.mem_get_info()[0]
    postings, per_chunk = 4 * n * 8, 128 * n          # and the split head-term weights
    per_term = vocab * (8 + 4 + 4)
    table = vocab * (n // 8192 + 2) * 8
    # (ten allocations, in steps of 2 MiB)
    assert used <= postings + per_chunk + per_term + table + 10 * (2 << 20), used
