"""The layer kernel's hand-overs between the CTAs of a head, as tagged words (records of few and many CTAs a head, one and two scoring
heads, an odd number of chunk scores, the most that fit) and by counters (more chunk scores than fit). Launches of different
inputs follow one another, so that every launch meets the words of the one before."""
import numpy as np
import pytest
import torch

from oracle import chunkkv_oracle as ora
from tests.helpers import assert_gather_exact, assert_selection_matches, bits_of, rand_bits, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Hq,Hkv,d,L,w,c", [
    (8, 2, 64, 300, 16, 10),                     # 3 CTAs a head
    (4, 1, 64, 3000, 16, 10),                    # 25 CTAs, 64 rows: eight slices
    (4, 1, 64, 148 * 120 + 5, 16, 20),           # 148
    (5, 1, 64, 3000, 16, 10),                    # 25 CTAs, 80 rows: four slices, more than one round
    (64, 8, 128, 32 + 1009, 32, 10),             # two scoring heads, 101 chunks, the last clipped
    (64, 32, 128, 4 * 128 * 33 + 65, 128, 32),   # two query tiles
    (16, 16, 64, 5 * 4096 + 4, 4, 5),            # 65536 chunk scores
    (16, 16, 64, 5 * 4096 + 5, 4, 5),            # one more a head
])
def test_launches_in_turn(Hq, Hkv, d, L, w, c):
    import paper_2502_00299_b200 as ck
    rng = np.random.default_rng(L)
    budget = w + c * max(1, (L - w) // (5 * c))
    xs = [(rand_bits(rng, (Hq, w, d)), rand_bits(rng, (Hkv, L, d)), rand_bits(rng, (Hkv, L, d))) for _ in range(2)]
    dev = [tuple(map(to_dev, x)) for x in xs]
    outs = [ck.compress_layer(*dev[i % 2], Hq, w, c, budget) for i in range(5)]
    assert ck.device_status() == 0
    for i, (oK, oV, idx) in enumerate(outs):
        q, K, V = xs[i % 2]
        if i < 2:
            s = ora.chunk_scores(ora.token_scores(q, K, Hq, Hkv, w), c)
            assert_selection_matches(idx.cpu().numpy(), s, L, w, c, budget)
            assert_gather_exact(bits_of(oK), bits_of(oV), idx.cpu().numpy(), K, V)
        else:
            assert all(torch.equal(a, b) for a, b in zip(outs[i], outs[i - 2]))
