"""The selection bodies that the one-launch layer kernel and the persistent model kernel dispatch to, over their ranges of chunk
counts: keys in registers (8 and 16 a thread), keys in shared memory, and 8 bits at a time where the keys do not fit or very
many chunks are kept. Each against the oracle, and with ties that the lower chunk id has to win."""
import numpy as np
import pytest
import torch

from oracle import chunkkv_oracle as ora
from tests.helpers import assert_gather_exact, assert_selection_matches, bits_of, rand_bits, to_dev

pytestmark = pytest.mark.gpu

# The layer kernel has 576 threads: 16 keys a thread up to 9216 chunks, then keys in the K ring's shared memory (29994 chunks do
# not fit beside two query tiles, and more than 8192 kept ones are not staged).
LAYER = [(4, 1, 64, 30000, 16, 5, 700), (8, 2, 64, 46000, 16, 8, 500), (4, 1, 64, 60000, 16, 5, 700), (16, 2, 64, 100000, 32, 10, 900),
         (8, 1, 128, 150000, 32, 5, 700), (2, 1, 64, 60000, 8, 5, 9000)]
# A selector of the model kernel has 640: 10240 chunks, then shared memory; 59999 chunks do not fit.
MODEL = [(4, 1, 64, 30000, 16, 5, 700), (4, 1, 64, 60000, 16, 5, 700), (2, 1, 64, 300000, 8, 5, 700)]


@pytest.fixture(scope="module")
def ck():
    import paper_2502_00299_b200 as ck
    assert torch.cuda.is_available()
    return ck


def _random(Hq, Hkv, d, L, w, seed):
    rng = np.random.default_rng(seed)
    return rand_bits(rng, (Hq, w, d)), rand_bits(rng, (Hkv, L, d)), rand_bits(rng, (Hkv, L, d))


def _tied(Hq, Hkv, d, L, w, c, k, seed):
    """Two kinds of keys by whole chunks: all tokens of a marked chunk have one key, all others another with a smaller logit
    (one query for all rows). The marked chunks' scores are equal to the bit, and there are more of them than are kept."""
    rng = np.random.default_rng(seed)
    q, K = rand_bits(rng, (Hq, w, d)), np.empty((Hkv, L, d), dtype=np.uint16)
    q[:] = q[:1, :1]
    C = -(-(L - w) // c)
    hot = np.zeros((Hkv, C), dtype=bool)
    for h in range(Hkv):
        # (none in the last 200 tokens, whose panels add a chunk's terms in another order)
        hot[h, rng.permutation(C - 200 // c)[:k + k // 2 + 3]] = True
        on = np.zeros(L, dtype=bool)
        on[:L - w] = np.repeat(hot[h], c)[:L - w]
        K[h] = np.where(on[:, None], q[0, 0], np.uint16(0))                       # logit |q|^2 / sqrt(d) or 0
    return q, K, rand_bits(rng, (Hkv, L, d)), hot


def _expect_tied(idx, hot, L, w, c, k):
    for h in range(idx.shape[0]):
        chunks = np.flatnonzero(hot[h])[:k]
        want = np.concatenate([(chunks[:, None] * c + np.arange(c)).ravel(), np.arange(L - w, L)])
        assert np.array_equal(idx[h], want), f"head {h}: ties must go to the lower chunk ids"


@pytest.mark.parametrize("Hq,Hkv,d,L,w,c,k", LAYER)
def test_layer_selection(ck, Hq, Hkv, d, L, w, c, k):
    budget = w + c * k
    q, K, V = _random(Hq, Hkv, d, L, w, seed=L + c)
    s = ora.chunk_scores(ora.token_scores(q, K, Hq, Hkv, w), c)
    oK, oV, idx = ck.compress_layer(*map(to_dev, (q, K, V)), Hq, w, c, budget)
    assert ck.device_status() == 0
    assert_selection_matches(idx.cpu().numpy(), s, L, w, c, budget)
    assert_gather_exact(bits_of(oK), bits_of(oV), idx.cpu().numpy(), K, V)
    q, K, V, hot = _tied(Hq, Hkv, d, L, w, c, k, seed=L + c)
    oK, oV, idx = ck.compress_layer(*map(to_dev, (q, K, V)), Hq, w, c, budget)
    assert ck.device_status() == 0
    _expect_tied(idx.cpu().numpy(), hot, L, w, c, k)
    assert_gather_exact(bits_of(oK), bits_of(oV), idx.cpu().numpy(), K, V)


@pytest.mark.parametrize("Hq,Hkv,d,L,w,c,k", MODEL)
def test_model_selection(ck, Hq, Hkv, d, L, w, c, k):
    budget = w + c * k
    q, K, V = _random(Hq, Hkv, d, L, w, seed=L + c)
    tq, tK, tV, hot = _tied(Hq, Hkv, d, L, w, c, k, seed=L + c)
    s = ora.chunk_scores(ora.token_scores(q, K, Hq, Hkv, w), c)
    outs = ck.compress_model([tuple(map(to_dev, x)) for x in ((q, K, V), (tq, tK, tV))], Hq, w, c, budget, 1)
    assert ck.device_status() == 0
    assert_selection_matches(outs[0][2].cpu().numpy(), s, L, w, c, budget)
    _expect_tied(outs[1][2].cpu().numpy(), hot, L, w, c, k)
    for (oK, oV, idx), (k_, v_) in zip(outs, ((K, V), (tK, tV))):
        assert_gather_exact(bits_of(oK), bits_of(oV), idx.cpu().numpy(), k_, v_)


@pytest.mark.parametrize("C,k", [(4, 2), (2047, 600), (2049, 600), (4096, 4095), (4097, 800), (9000, 700), (30000, 9000), (65535, 4000), (65537, 300)])
def test_select_with_all_scores_equal_and_with_two_values(ck, C, k):
    # register, cluster, shared-memory and 8-bits-at-a-time bodies of chunkkv_select
    L, w, c = 2 * C + 3, 3, 2
    x = torch.full((2, C), 0.25, device="cuda")
    g = torch.Generator(device="cuda").manual_seed(C)
    hot = torch.randperm(C, device="cuda", generator=g)[:max(1, k // 2)]
    x[1, hot] = 0.5
    idx = ck.select(x, L, w, c, w + c * k).cpu().numpy()
    for h in range(2):
        want = ora.select_chunks(x[h].double().cpu().numpy(), k)
        assert np.array_equal(idx[h][:k * c], (want[:, None] * c + np.arange(c)).ravel())
        assert idx[h][k * c:].tolist() == list(range(L - w, L))


# Chunk counts at the ends of the runs of ids that a thread holds (2, 4, 8, 16, 24): 576 threads in the layer kernel, 512 in chunkkv_select
@pytest.mark.parametrize("C,k", [(1, 1), (31, 30), (575, 1), (1152, 100), (1153, 1152), (2304, 700), (2305, 300), (4608, 4000),
                                 (4609, 900), (9216, 1), (9217, 800), (13824, 600), (13825, 700)])
def test_layer_selection_at_the_ends_of_runs(ck, C, k):
    w, c, d = 16, 5, 64
    L = C * c + w - (3 if C > 1 else 0)                 # (a clipped last chunk)
    q, K, V = _random(4, 1, d, L, w, seed=C)
    s = ora.chunk_scores(ora.token_scores(q, K, 4, 1, w), c)
    oK, oV, idx = ck.compress_layer(*map(to_dev, (q, K, V)), 4, w, c, w + c * k)
    assert ck.device_status() == 0
    assert_selection_matches(idx.cpu().numpy(), s, L, w, c, w + c * k)
    assert_gather_exact(bits_of(oK), bits_of(oV), idx.cpu().numpy(), K, V)


@pytest.mark.parametrize("C", [2, 33, 511, 1024, 1025, 2048, 2049, 4095, 4096])
def test_select_at_the_ends_of_runs(ck, C):
    L, w, c = 2 * C + 3, 3, 2
    g = torch.Generator(device="cuda").manual_seed(C)
    x = torch.randn(4, C, device="cuda", generator=g)                                  # head 0: all different
    x[1] = torch.randint(0, 3, (C,), device="cuda", generator=g).float()               # many ties
    x[2] = torch.where(torch.rand(C, device="cuda", generator=g) < 0.9, -float("inf"), x[0])
    x[3] = torch.where(torch.rand(C, device="cuda", generator=g) < 0.1, 1e30 * x[0], 1e-30 * x[0])
    for k in sorted({1, C // 3 + 1, C - 1, C}):
        idx = ck.select(x, L, w, c, w + c * k).cpu().numpy()
        for h in range(4):
            want = ora.select_chunks(x[h].double().cpu().numpy(), k)
            assert np.array_equal(idx[h][:k * c], (want[:, None] * c + np.arange(c)).ravel())


# The same with the scores of two scoring heads added (136 rows of an even group of heads)
@pytest.mark.parametrize("C,k", [(575, 3), (1152, 700), (1153, 1), (2304, 90), (2305, 2300), (4608, 500), (4609, 1000)])
def test_layer_selection_of_two_scoring_heads_at_the_ends_of_runs(ck, C, k):
    w, c, d = 17, 10, 64
    L = C * c + w - 4
    q, K, V = _random(8, 1, d, L, w, seed=C)
    s = ora.chunk_scores(ora.token_scores(q, K, 8, 1, w), c)
    oK, oV, idx = ck.compress_layer(*map(to_dev, (q, K, V)), 8, w, c, w + c * k)
    assert ck.device_status() == 0
    assert_selection_matches(idx.cpu().numpy(), s, L, w, c, w + c * k)
    assert_gather_exact(bits_of(oK), bits_of(oV), idx.cpu().numpy(), K, V)


# A selector of the model kernel has 640 threads: runs of 2 and 4 ids, 8 and 16 keys a thread, then shared memory; small and big (two
# query tiles) variants, the big one for chunks of 8 without runs
@pytest.mark.parametrize("Hq,c", [(4, 5), (16, 10), (16, 8)])
@pytest.mark.parametrize("C,k", [(1280, 300), (1281, 1280), (2560, 1), (2561, 800), (5120, 5000), (5121, 400), (10240, 700), (10241, 900)])
def test_model_selection_at_the_ends_of_runs(ck, Hq, c, C, k):
    w, d = 10, 64
    L = C * c + w - 3
    q, K, V = _random(Hq, 1, d, L, w, seed=C + c)
    s = ora.chunk_scores(ora.token_scores(q, K, Hq, 1, w), c)
    x = tuple(map(to_dev, (q, K, V)))
    outs = ck.compress_model([x, x], Hq, w, c, w + c * k)
    assert ck.device_status() == 0
    assert_selection_matches(outs[0][2].cpu().numpy(), s, L, w, c, w + c * k)
    assert_gather_exact(bits_of(outs[0][0]), bits_of(outs[0][1]), outs[0][2].cpu().numpy(), K, V)
    assert all(torch.equal(a, b) for a, b in zip(*outs))
