"""Keys that no query attends to (an infinite component gives every row the logit -inf): their score is 0, and the other
keys' scores and the selection are what they are without them. Tolerances as in test_gpu_parity.py."""
import numpy as np
import pytest
import torch

from oracle import chunkkv_oracle as ora
from tests.helpers import assert_gather_exact, assert_scores_close, assert_selection_matches, bits_of, rand_bits, to_dev

pytestmark = pytest.mark.gpu

MINUS_INF = np.uint16(0xFF80)


@pytest.fixture(scope="module")
def ck():
    import paper_2502_00299_b200 as ck
    assert torch.cuda.is_available()
    return ck


def _inputs(Hq, Hkv, d, L, w, hidden, seed):
    rng = np.random.default_rng(seed)
    q, K, V = rand_bits(rng, (Hq, w, d)), rand_bits(rng, (Hkv, L, d)), rand_bits(rng, (Hkv, L, d))
    q[..., 0] = np.uint16(0x3F80)                 # 1: the product with the infinite component is -inf for every row
    K[:, hidden, 0] = MINUS_INF
    return q, K, V


def _check(ck, Hq, Hkv, d, L, w, c, hidden):
    q, K, V = _inputs(Hq, Hkv, d, L, w, hidden, seed=L + c)
    t = ora.token_scores(q, K, Hq, Hkv, w)
    s = ora.chunk_scores(t, c)
    assert np.all(t[:, [j for j in hidden if j < L - w]] == 0) and np.isfinite(t).all()
    R, (dq, dK, dV) = w * Hq // Hkv, map(to_dev, (q, K, V))
    cs, ts = ck.score(dq, dK, w, c, want_token_scores=True)
    alone, _ = ck.score(dq, dK, w, c)
    budget = w + c * max(1, (L - w) // (4 * c))
    oK, oV, idx = ck.compress_layer(dq, dK, dV, Hq, w, c, budget)
    assert ck.device_status() == 0
    for got, want, what in ((ts, t, "token scores"), (cs, s, "chunk scores beside token scores"), (alone, s, "chunk scores")):
        assert torch.isfinite(got).all(), f"{what}: {int((~torch.isfinite(got)).sum())} are not finite"
        assert_scores_close(got.cpu().numpy(), want, R, L, what)
    idx = idx.cpu().numpy()
    assert_selection_matches(idx, s, L, w, c, budget)
    assert_gather_exact(bits_of(oK), bits_of(oV), idx, K, V)


# rows per scoring head of the token-score kernel: 112, 128 + 96, 8, 1, 86, 64, 128, 256
@pytest.mark.parametrize("Hq,Hkv,d,w", [(28, 4, 128, 16), (28, 4, 128, 32), (4, 4, 64, 8), (2, 2, 64, 1), (10, 5, 64, 43), (32, 8, 64, 16),
                                        (32, 8, 128, 32), (64, 8, 128, 32)])
@pytest.mark.parametrize("c", [1, 7])
def test_single_keys_without_attention_at_token_level(ck, Hq, Hkv, d, w, c):
    _check(ck, Hq, Hkv, d, 1500, w, c, [3, 77, 300, 301, 640, 1499 - w])


# runs that cover whole panels (60 or 64 keys of a row): a CTA's first panel, panels between others, everything up to the window
@pytest.mark.parametrize("Hq,Hkv,d,L,w", [(32, 8, 128, 1500, 32), (64, 8, 64, 9000, 32), (4, 4, 64, 700, 8), (32, 32, 64, 4 * 128 * 17 + 1, 8)])
@pytest.mark.parametrize("c", [1, 5, 7, 8, 10, 16, 20, 32])
def test_runs_of_keys_without_attention(ck, Hq, Hkv, d, L, w, c):
    _check(ck, Hq, Hkv, d, L, w, c, [*range(200, 520), *range(L - w - 150, L - w)])


@pytest.mark.parametrize("c", [5, 8, 10, 16, 20, 32])
@pytest.mark.parametrize("Hq", [8, 64])
def test_model_call_with_runs_of_keys_without_attention(ck, Hq, c):
    Hkv, d, L, w = 8, 64, 6000, 32
    hidden = [*range(200, 520), *range(L - w - 150, L - w)]
    xs = [_inputs(Hq, Hkv, d, L, w, hidden, seed=c + i) for i in range(3)]
    budget = w + c * ((L - w) // (4 * c))
    outs = ck.compress_model([tuple(map(to_dev, x)) for x in xs], Hq, w, c, budget, 1)
    assert ck.device_status() == 0
    for (q, K, V), (oK, oV, idx) in zip(xs, outs):
        s = ora.chunk_scores(ora.token_scores(q, K, Hq, Hkv, w), c)
        assert_selection_matches(idx.cpu().numpy(), s, L, w, c, budget)
        assert_gather_exact(bits_of(oK), bits_of(oV), idx.cpu().numpy(), K, V)
