"""Layers of at most 9216 chunks a head that keep more of them than a CTA lists (8192): either side of that line, into packed and
paged outputs, and a whole-model call, which runs layer by layer there. A layer of other inputs goes ahead, whose scores lie in scratch."""
import numpy as np
import pytest
import torch

from oracle import chunkkv_oracle as ora
from tests.helpers import assert_gather_exact, assert_selection_matches, bits_of, rand_bits, to_dev

pytestmark = pytest.mark.gpu


# one and four KV heads, and one whose 136 rows are two scoring heads
@pytest.mark.parametrize("Hq,Hkv,w,c", [(4, 1, 16, 5), (16, 4, 4, 8), (8, 1, 17, 10)])
@pytest.mark.parametrize("C,k", [(8193, 8192), (9000, 8193), (9000, 8999), (9216, 8500), (9000, 9000)])
def test_layers_that_keep_most_chunks(Hq, Hkv, w, c, C, k):
    import paper_2502_00299_b200 as ck
    d, page = 64, 32
    L, budget = C * c + w - 2, w + c * k                  # (a clipped last chunk)
    rng = np.random.default_rng(C + k + Hkv)
    xs = [(rand_bits(rng, (Hq, w, d)), rand_bits(rng, (Hkv, L, d)), rand_bits(rng, (Hkv, L, d))) for _ in range(2)]
    dev = [tuple(map(to_dev, x)) for x in xs]
    want = [ora.chunk_scores(ora.token_scores(q, K, Hq, Hkv, w), c) for q, K, _ in xs]
    ck.compress_layer(*dev[1], Hq, w, c, w + c)           # (the other inputs' scores)
    ck.compress_layer(*dev[1], Hq, w, c, budget)
    outs = [ck.compress_layer(*x, Hq, w, c, budget) for x in dev]
    assert ck.device_status() == 0
    for (oK, oV, idx), s, (_, K, V) in zip(outs, want, xs):
        assert_selection_matches(idx.cpu().numpy(), s, L, w, c, budget)
        assert_gather_exact(bits_of(oK), bits_of(oV), idx.cpu().numpy(), K, V)
    # paged: the same rows through a block table
    n_pages = -(-(w + c * k) // page)
    table = torch.arange(n_pages, dtype=torch.int32, device="cuda").flip(0).contiguous()
    cache = [torch.zeros(n_pages, page, Hkv, d, dtype=torch.bfloat16, device="cuda") for _ in range(2)]
    ck.compress_layer(*dev[1], Hq, w, c, budget)
    idx = ck.compress_layer_paged(*dev[0], Hq, w, c, budget, table, *cache)
    assert ck.device_status() == 0 and torch.equal(idx, outs[0][2])
    for out, pages in zip(outs[0], cache):
        rows = pages[table.long()].reshape(n_pages * page, Hkv, d)[:w + c * k].transpose(0, 1)
        kept = (idx >= 0)[..., None]
        assert torch.equal(torch.where(kept, rows, 0), out)
    # the model call, two computed layers and two that reuse their indices
    model = ck.compress_model([dev[0], dev[1], dev[1], dev[0]], Hq, w, c, budget, 2)
    assert ck.device_status() == 0
    for l in (0, 2):
        assert all(torch.equal(a, b) for a, b in zip(model[l], outs[0 if l == 0 else 1]))
        assert torch.equal(model[l + 1][2], model[l][2])
