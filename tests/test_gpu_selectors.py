"""Whole-model calls with as many selector CTAs as heads, 16 at most: heads that share a selector unevenly, heads beyond 16, and
lengths at which the number of selectors changes."""
import numpy as np
import pytest

from oracle import chunkkv_oracle as ora
from tests.helpers import assert_gather_exact, assert_selection_matches, bits_of, rand_bits, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Hq,Hkv,d,L,w,c,budget,reuse", [
    (8, 8, 64, 1000, 8, 10, 100, 1), (8, 8, 64, 8200, 8, 10, 4000, 3), (64, 8, 64, 4100, 32, 10, 400, 1),
    (12, 12, 64, 700, 8, 5, 150, 2), (16, 16, 64, 1500, 8, 16, 300, 1), (20, 20, 64, 900, 8, 10, 120, 1), (33, 33, 64, 600, 8, 20, 100, 2),
    (140, 140, 64, 300, 4, 10, 50, 1),
    # either side of a change: 8 -> 4, twice
    (64, 8, 64, 4080, 32, 10, 400, 1), (64, 8, 64, 4081, 32, 10, 400, 1), (8, 8, 64, 10200, 8, 10, 100, 1), (8, 8, 64, 10201, 8, 10, 100, 1),
])
def test_model_call(Hq, Hkv, d, L, w, c, budget, reuse):
    import paper_2502_00299_b200 as ck
    rng = np.random.default_rng(Hkv * L)
    n = 2 * reuse
    xs = [(rand_bits(rng, (Hq, w, d)), rand_bits(rng, (Hkv, L, d)), rand_bits(rng, (Hkv, L, d))) for _ in range(n)]
    outs = ck.compress_model([tuple(map(to_dev, x)) for x in xs], Hq, w, c, budget, reuse)
    assert ck.device_status() == 0
    for l, (oK, oV, idx) in enumerate(outs):
        q, K, V = xs[l // reuse * reuse]
        idx = idx.cpu().numpy()
        if l % reuse == 0:
            assert_selection_matches(idx, ora.chunk_scores(ora.token_scores(q, K, Hq, Hkv, w), c), L, w, c, budget)
        else:
            assert np.array_equal(idx, outs[l // reuse * reuse][2].cpu().numpy())
        assert_gather_exact(bits_of(oK), bits_of(oV), idx, xs[l][1], xs[l][2])
