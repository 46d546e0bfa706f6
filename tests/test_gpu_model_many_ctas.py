"""Whole-model calls with many CTAs a head, whose row records every epilogue thread merges by itself (18 at a time): counts at and beside
multiples of 18, the most there are, and heads whose last CTA has few keys."""
import numpy as np
import pytest
import torch

from oracle import chunkkv_oracle as ora
from tests.helpers import assert_gather_exact, assert_selection_matches, bits_of, rand_bits, to_dev

pytestmark = pytest.mark.gpu


# key tiles of 120: 36, 37, 54, 55, 72 (of at most 73, 72, 48 and 147 CTAs a head), 300
@pytest.mark.parametrize("Hq,Hkv,w,c", [(8, 1, 16, 10), (8, 2, 32, 5), (2, 1, 33, 20), (9, 3, 4, 10)])
@pytest.mark.parametrize("L", [36 * 120, 36 * 120 + 1, 54 * 120, 54 * 120 + 7, 72 * 120, 36000])
def test_model_call(Hq, Hkv, w, c, L):
    import paper_2502_00299_b200 as ck
    d, budget = 64, w + c * (L // (8 * c))
    rng = np.random.default_rng(L + Hq)
    xs = [(rand_bits(rng, (Hq, w, d)), rand_bits(rng, (Hkv, L, d)), rand_bits(rng, (Hkv, L, d))) for _ in range(2)]
    for x in xs:                                                    # (a sink: row maxima that differ from CTA to CTA)
        x[1][:, 2] = x[0][0, 0]
    dev = [tuple(map(to_dev, x)) for x in xs]
    outs = ck.compress_model([dev[i % 2] for i in range(5)], Hq, w, c, budget, 1)
    assert ck.device_status() == 0
    for i, (oK, oV, idx) in enumerate(outs):
        q, K, V = xs[i % 2]
        if i < 2:
            idx = idx.cpu().numpy()
            assert_selection_matches(idx, ora.chunk_scores(ora.token_scores(q, K, Hq, Hkv, w), c), L, w, c, budget)
            assert_gather_exact(bits_of(oK), bits_of(oV), idx, K, V)
        else:
            assert all(torch.equal(a, b) for a, b in zip(outs[i], outs[i - 2]))
