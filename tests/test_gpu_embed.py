"""GPU parity of the embedding tail (Sec. 4.3: masked mean pool of hidden
states, L2 normalisation, cast to the index dtype) against the fp64 oracle.
A bf16 output must be a correct rounding of a value within 2e-6 of the exact
result (the kernel accumulates in fp32); an fp32 output must lie within 2e-6."""
import numpy as np
import pytest
import torch

import oracle
from paper_2608_08340_gb300 import workloads
from paper_2608_08340_gb300.index import Index, embed_pool

from _golden import load
from _gpu import check_dense, dev_tensor

pytestmark = pytest.mark.gpu

ERR = 2e-6


def _bf16_ok(got_bits, exact):
    got = oracle.bf16_to_f32(got_bits).astype(np.float64)
    # half a bf16 ulp of the exact value (8 bits of mantissa), plus the fp32 error
    ulp = np.where(exact != 0, 2.0 ** (np.floor(np.log2(np.abs(exact) + 1e-300)) - 7), 2.0 ** -133)
    return np.abs(got - exact) <= 0.5 * ulp + ERR


def test_embed_pool_golden_padded_to_eight_dims():
    g = load("embed_pool_2tok.json")
    h = np.zeros((3, 2, 8), np.float32)
    h[:, :, :2] = np.array(g["hidden"], np.float32)
    out = embed_pool(torch.from_numpy(h).cuda(), torch.tensor(g["mask"], dtype=torch.uint8).cuda())
    bits = out.view(torch.int16).cpu().numpy().view(np.uint16)
    assert bits[:, :2].tolist() == g["bf16_bits"]
    assert (bits[:, 2:] == 0).all()


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("dim", [768, 4096, 136])
@pytest.mark.parametrize("out_dtype", [torch.bfloat16, torch.float32])
def test_embed_pool_matches_oracle(dtype, dim, out_dtype):
    rng = np.random.default_rng(dim + (dtype == "bf16"))
    b, t = 37, 50
    h = rng.standard_normal((b, t, dim)).astype(np.float32)
    lens = rng.integers(1, t + 1, b)
    mask = (np.arange(t)[None, :] < lens[:, None]).astype(np.uint8)
    mask[3] = 0                                            # a row with no real token
    mask[5] = (rng.random(t) < 0.3)                        # a row with holes
    h_in = oracle.round_bf16(h) if dtype == "bf16" else h
    exact = oracle.embed_pool(h_in, mask)
    out = embed_pool(dev_tensor(h_in), torch.from_numpy(mask).cuda(), out_dtype)
    torch.cuda.synchronize()
    if out_dtype == torch.bfloat16:
        bits = out.view(torch.int16).cpu().numpy().view(np.uint16)
        ok = _bf16_ok(bits, exact)
        assert ok.all(), f"{(~ok).sum()} of {ok.size} values off"
    else:
        np.testing.assert_allclose(out.cpu().numpy(), exact, rtol=0, atol=ERR)
    assert (out[3] == 0).all()


@pytest.mark.parametrize("dtype,dim", [("bf16", 12272), ("bf16", 12280), ("bf16", 12288),
                                       ("bf16", 12296), ("bf16", 16384), ("f32", 8192)])
def test_embed_pool_of_wide_rows_in_small_batches(dtype, dim):
    """Partial sums of a row around 48 KB, where the shared memory opt-in begins."""
    rng = np.random.default_rng(dim)
    h = rng.standard_normal((3, 130, dim)).astype(np.float32)
    h_in = oracle.round_bf16(h) if dtype == "bf16" else h
    mask = np.ones((3, 130), np.uint8)
    mask[1, 77:] = 0
    out = embed_pool(dev_tensor(h_in), torch.from_numpy(mask).cuda(), torch.float32)
    np.testing.assert_allclose(out.cpu().numpy(), oracle.embed_pool(h_in, mask), rtol=0, atol=ERR)


# Batches whose rows one CTA takes alone (400 rows, or fewer than 16 tokens), and
# two, four and eight share; widths whose groups do not divide among them.
@pytest.mark.parametrize("b,t", [(400, 9), (3, 15), (152, 40), (60, 33), (20, 70), (1, 512)])
@pytest.mark.parametrize("dtype,dim", [("bf16", 8), ("bf16", 136), ("bf16", 2056), ("bf16", 4104),
                                       ("f32", 8), ("f32", 1032), ("f32", 2056)])
def test_embed_pool_at_every_split(b, t, dtype, dim):
    rng = np.random.default_rng(b + dim)
    h = rng.standard_normal((b, t, dim)).astype(np.float32)
    h_in = oracle.round_bf16(h) if dtype == "bf16" else h
    mask = (rng.random((b, t)) < 0.7).astype(np.uint8)
    mask[:, 0] = 1
    out = embed_pool(dev_tensor(h_in), torch.from_numpy(mask).cuda(), torch.float32)
    np.testing.assert_allclose(out.cpu().numpy(), oracle.embed_pool(h_in, mask), rtol=0, atol=ERR)


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("dim,tokens", [(768, 70), (1000, 300), (4096, 128), (8192, 40)])
def test_a_row_does_not_depend_on_its_batch(dtype, dim, tokens):
    """The same bits alone, in batches of every split and with more padding."""
    g = torch.Generator(device="cuda").manual_seed(dim)
    h = torch.randn(400, tokens, dim, generator=g, device="cuda").to(dtype)
    mask = (torch.rand(400, tokens, generator=g, device="cuda") < 0.8).to(torch.uint8)
    whole = embed_pool(h, mask, torch.float32)
    for b in (1, 2, 19, 40, 80, 160, 310):
        assert torch.equal(embed_pool(h[:b], mask[:b], torch.float32), whole[:b]), b
    wide = torch.zeros(5, tokens + 90, dim, dtype=dtype, device="cuda")
    wide[:, :tokens] = h[:5]
    wide_mask = torch.zeros(5, tokens + 90, dtype=torch.uint8, device="cuda")
    wide_mask[:, :tokens] = mask[:5]
    assert torch.equal(embed_pool(wide, wide_mask, torch.float32), whole[:5])


def test_embed_pool_feeds_the_search():
    w = workloads.config(1, n=8000, batch=4)
    rng = np.random.default_rng(11)
    h = oracle.round_bf16(rng.standard_normal((64, 20, w.d)).astype(np.float32))
    mask = np.ones((64, 20), np.uint8)
    mask[:, 15:] = 0
    Q = embed_pool(dev_tensor(h), torch.from_numpy(mask).cuda())
    idx = Index(dev_tensor(w.E_data))
    ids, sc = idx.search(Q, 10)
    q_bits = Q.view(torch.int16).cpu().numpy().view(np.uint16)
    check_dense(ids, sc, w.E_data, q_bits, 10, "pooled queries")


def test_embed_pool_argument_errors():
    h = torch.zeros((2, 3, 12), dtype=torch.bfloat16, device="cuda")       # dim not % 8
    with pytest.raises(RuntimeError):
        embed_pool(h, torch.ones((2, 3), dtype=torch.uint8, device="cuda"))
    h = torch.zeros((2, 3, 16), dtype=torch.bfloat16, device="cuda")
    with pytest.raises(ValueError):
        embed_pool(h, torch.ones((2, 4), dtype=torch.uint8, device="cuda"))
