"""The one-launch layer kernel over its whole range: every chunk size it is built for, one and two query tiles,
key ranges whose partial sums do not fit on chip, last tiles and chunks of any length, strided inputs, paged outputs.
Tolerances as in test_gpu_parity.py."""
import numpy as np
import pytest
import torch

from oracle import chunkkv_oracle as ora
from tests.helpers import (assert_gather_exact, assert_scores_close, assert_selection_matches, bits_of, guarded_outputs,
                           to_dev)
from workloads import CONFIGS, make_layer, scaled

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ck():
    import paper_2502_00299_b200 as ck
    assert torch.cuda.is_available()
    return ck


def _layer(Hq, Hkv, d, L, w, c, budget, seed=0):
    wl = scaled(CONFIGS[1], Hq=Hq, Hkv=Hkv, d=d, L=L, w=w, c=c, budget=budget, seed=900 + seed, planted_count=2,
                sink_tokens=1)
    return wl, make_layer(wl)


# a CTA takes ceil(ceil(L / tile) / (148 / Hkv)) key tiles (tile = 120 keys, 128 for c = 8, 16, 32); partial sums beyond
# 256 / (chunks per half tile) panels go to scratch
CASES = [
    (8, 2, 64, 2048, 16, 5), (8, 2, 64, 121, 16, 8), (8, 2, 64, 129, 16, 16), (4, 4, 128, 33, 32, 32), (2, 1, 128, 20, 16, 5),
    (28, 4, 128, 3000, 32, 10), (28, 4, 128, 1500, 16, 32),          # 224 rows: tiles of 128 and 96; 112 rows
    (15, 3, 64, 1203, 43, 20), (64, 8, 128, 2047, 32, 16),           # 215 rows (odd); 256 rows
    (64, 16, 64, 9 * 120 * 11 + 7, 16, 5),                           # 64 rows, 22 panels of which 21 fit
    (64, 16, 64, 9 * 120 * 22, 16, 10), (32, 32, 64, 4 * 128 * 17 + 1, 8, 8), (32, 32, 64, 4 * 128 * 33 - 3, 8, 16),
    (128, 32, 64, 4 * 120 * 23 + 61, 64, 20), (64, 32, 128, 4 * 128 * 33 + 65, 128, 32),     # 256 rows, in scratch from panel 86 / 129
]


@pytest.mark.parametrize("Hq,Hkv,d,L,w,c", CASES)
def test_layer_and_chunk_scores(ck, Hq, Hkv, d, L, w, c):
    budget = w + c * max(1, (L - w) // (4 * c)) + 1
    wl, x = _layer(Hq, Hkv, d, L, w, c, budget, seed=L)
    q, K, V = to_dev(x.q_obs), to_dev(x.K), to_dev(x.V)
    t = ora.token_scores(x.q_obs, x.K, Hq, Hkv, w)
    s = ora.chunk_scores(t, c)
    cs, _ = ck.score(q, K, w, c)
    assert_scores_close(cs.cpu().numpy(), s, w * Hq // Hkv, L, "chunk scores")
    gK, gV, gI = guarded_outputs(Hkv, ck.out_len(L, w, c, budget), d)
    oK, oV, idx = ck.compress_layer(q, K, V, Hq, w, c, budget, out_K=gK.t, out_V=gV.t, out_idx=gI.t)
    assert ck.device_status() == 0
    for g in (gK, gV, gI):
        g.check()
    idx = idx.cpu().numpy()
    assert_selection_matches(idx, s, L, w, c, budget)
    assert_gather_exact(bits_of(oK), bits_of(oV), idx, x.K, x.V)
    # token-major inputs: same scores and so the same selection and rows
    Kt, Vt = (a.permute(1, 0, 2).contiguous().permute(1, 0, 2) for a in (K, V))
    sK, sV, sidx = ck.compress_layer_strided(q, Kt, Vt, Hq, w, c, budget)
    assert np.array_equal(sidx.cpu().numpy(), idx) and torch.equal(sK, oK) and torch.equal(sV, oV)


# More than 128 rows: two scoring heads of half the rows where all their panels stay on chip, else two query tiles. Odd numbers of
# rows, the last length of the one form and the first of the other (32 KV heads: two CTAs a half, 21 tiles each hold 252 chunk slots),
# more KV heads than a hand-over counter per half leaves room for.
@pytest.mark.parametrize("Hq,Hkv,d,L,w,c", [
    (3, 1, 64, 900, 43, 10), (5, 1, 128, 1003, 51, 5), (14, 2, 128, 130, 32, 16), (128, 32, 64, 2 * 21 * 120, 64, 10),
    (128, 32, 64, 2 * 21 * 120 + 1, 64, 10), (160, 80, 64, 700, 65, 20), (64, 8, 128, 300, 32, 32),
])
def test_layer_with_more_than_128_rows(ck, Hq, Hkv, d, L, w, c):
    test_layer_and_chunk_scores(ck, Hq, Hkv, d, L, w, c)


# a model call's CTA takes ceil(ceil(L / tile) / (144 / Hkv)) key tiles of every layer; its ring of partial sums continues in
# scratch where a layer and eight panels more do not fit on chip, and always has both forms with two query tiles
MODEL_CASES = [
    (8, 2, 64, 2048, 16, 5, 3, 1), (28, 4, 128, 3000, 32, 10, 4, 2), (4, 4, 128, 1300, 32, 32, 5, 2),
    (64, 16, 64, 9 * 120 * 11 + 7, 16, 5, 3, 2), (64, 16, 64, 9 * 128 * 18, 16, 8, 3, 1), (64, 16, 64, 9 * 120 * 23 - 50, 16, 10, 4, 1),
    (128, 32, 64, 4 * 120 * 15 + 61, 64, 20, 4, 1), (128, 32, 64, 4 * 128 * 12, 64, 16, 3, 1), (64, 32, 128, 4 * 128 * 20, 128, 32, 2, 1),
    (8, 2, 64, 600, 16, 10, 100, 98),                     # a reuse group longer than a launch
]


@pytest.mark.parametrize("Hq,Hkv,d,L,w,c,n_layers,n_reuse", MODEL_CASES)
def test_model_call(ck, Hq, Hkv, d, L, w, c, n_layers, n_reuse):
    budget = w + c * max(1, (L - w) // (4 * c)) + 1
    wl = scaled(CONFIGS[1], Hq=Hq, Hkv=Hkv, d=d, L=L, w=w, c=c, budget=budget, seed=950 + L, planted_count=2, sink_tokens=1)
    xs = [make_layer(wl, layer=i) for i in range(min(n_layers, 5))]
    pick = [min(i, 4) for i in range(n_layers)]
    on = [(to_dev(x.q_obs), to_dev(x.K), to_dev(x.V)) for x in xs]
    dev = [on[p] for p in pick]
    guards = [guarded_outputs(Hkv, ck.out_len(L, w, c, budget), d) for _ in range(n_layers)]
    for _ in range(2):                                    # the second call finds the counters and scratch of the first
        outs = ck.compress_model(dev, Hq, w, c, budget, n_reuse, outs=[tuple(g.t for g in gs) for gs in guards])
        assert ck.device_status() == 0
    for gs in guards:
        for g in gs:
            g.check()
    for l, (oK, oV, idx) in enumerate(outs):
        x, src = xs[pick[l]], l // n_reuse * n_reuse
        if l == src:
            t = ora.token_scores(x.q_obs, x.K, Hq, Hkv, w)
            assert_selection_matches(idx.cpu().numpy(), ora.chunk_scores(t, c), L, w, c, budget)
        else:
            assert torch.equal(idx, outs[src][2])
        if l < 5 or l > n_layers - 3:
            assert_gather_exact(bits_of(oK), bits_of(oV), idx.cpu().numpy(), x.K, x.V)
    major = [(q, *(a.permute(1, 0, 2).contiguous().permute(1, 0, 2) for a in (K, V))) for q, K, V in on]
    for a, b in zip(ck.compress_model_strided([major[p] for p in pick], Hq, w, c, budget, n_reuse), outs):
        assert all(torch.equal(s, t) for s, t in zip(a, b))


# token scores: 128-key tiles, one or two scoring heads per KV head (128 rows and the rest), two passes
@pytest.mark.parametrize("Hq,Hkv,d,L,w,c", [
    (8, 2, 64, 2048, 16, 7), (28, 4, 128, 1500, 32, 13), (15, 3, 64, 1203, 43, 300), (4, 1, 128, 129, 1, 100), (64, 8, 128, 20 * 128, 32, 64),
    (32, 8, 64, 18 * 128 * 5 + 1, 16, 3), (4, 2, 128, 40, 32, 65), (256, 1, 64, 700, 1, 1), (4, 4, 64, 127 + 16, 16, 2),
])
def test_token_scores_and_chunk_scores_with_and_without_them(ck, Hq, Hkv, d, L, w, c):
    wl, x = _layer(Hq, Hkv, d, L, w, c, w, seed=L + c)
    q, K = to_dev(x.q_obs), to_dev(x.K)
    t = ora.token_scores(x.q_obs, x.K, Hq, Hkv, w)
    s = ora.chunk_scores(t, c)
    cs, ts = ck.score(q, K, w, c, want_token_scores=True)
    alone, none = ck.score(q, K, w, c)
    assert ck.device_status() == 0 and none is None
    R = w * Hq // Hkv
    assert_scores_close(ts.cpu().numpy(), t, R, L, "token scores")
    assert_scores_close(cs.cpu().numpy(), s, R, L, "chunk scores beside token scores")
    assert_scores_close(alone.cpu().numpy(), s, R, L, "chunk scores alone")


# Up to 64 rows and more than 20 CTAs a head read the head's row statistics in a variant of their own: its first row and CTA counts,
# the last ones before it, one round trip of records (40) and its first beyond, every CTA of the GPU for one head.
@pytest.mark.parametrize("Hq,w,d,tiles", [(1, 1, 64, 21), (3, 11, 64, 20), (4, 16, 128, 21), (4, 16, 64, 40), (2, 32, 64, 41), (5, 13, 64, 41),
                                          (4, 16, 64, 148), (1, 64, 128, 81)])
def test_layer_with_few_rows_and_many_ctas(ck, Hq, w, d, tiles):
    test_layer_and_chunk_scores(ck, Hq, 1, d, 120 * tiles - 7, w, 10)


# Five to eight heads have a selector CTA each up to six tiles a scoring CTA (28, 23, 20 and 17 CTAs a head), six and eight only while
# few chunks and rows are copied for a selection: the last length of the one form and the first of the other, one and two query
# tiles, either side of 15 and 22 chunks a CTA (indices shared or not) and of 27 % of the rows.
@pytest.mark.parametrize("Hq,Hkv,L,w,c,n_layers,n_reuse,kept", [
    (5, 5, 28 * 6 * 120, 8, 10, 3, 1, 0.05), (5, 5, 28 * 6 * 120 + 1, 8, 10, 3, 1, 0.05), (6, 6, 23 * 6 * 120, 8, 10, 3, 1, 0.05),
    (6, 6, 23 * 6 * 120 + 1, 8, 10, 3, 1, 0.05), (14, 7, 20 * 6 * 128, 32, 16, 3, 2, 0.1), (14, 7, 20 * 6 * 128 + 1, 32, 16, 3, 2, 0.1),
    (64, 8, 17 * 6 * 120, 32, 20, 2, 1, 0.05), (64, 8, 17 * 6 * 120 + 1, 32, 20, 2, 1, 0.05), (7, 7, 600, 16, 5, 3, 1, 0.3), (6, 6, 121, 8, 8, 2, 1, 0.5),
    (16, 8, 17 * 3 * 120 - 5, 16, 10, 4, 2, 0.205), (16, 8, 17 * 3 * 120 - 5, 16, 10, 4, 2, 0.22), (16, 8, 17 * 4 * 120, 16, 20, 4, 1, 0.26),
    (16, 8, 17 * 4 * 120, 16, 20, 4, 1, 0.28), (16, 8, 17 * 2 * 120, 16, 32, 4, 3, 0.25), (8, 8, 17 * 2 * 120, 16, 5, 4, 3, 0.25),
    (40, 8, 17 * 4 * 128, 26, 8, 3, 50, 0.1),
])
def test_model_call_with_five_to_eight_heads(ck, Hq, Hkv, L, w, c, n_layers, n_reuse, kept):
    budget = w + c * int(kept * L / c)
    x = [_layer(Hq, Hkv, 64, L, w, c, budget, seed=i)[1] for i in range(2)]
    on = [tuple(to_dev(t) for t in (a.q_obs, a.K, a.V)) for a in x]
    outs = ck.compress_model([on[i % 2] for i in range(n_layers)], Hq, w, c, budget, n_reuse)
    assert ck.device_status() == 0
    for l, (oK, oV, idx) in enumerate(outs):
        src = l // n_reuse * n_reuse
        assert_gather_exact(bits_of(oK), bits_of(oV), idx.cpu().numpy(), x[l % 2].K, x[l % 2].V)
        if l != src:
            assert torch.equal(idx, outs[src][2])
        elif l < 2:
            s = ora.chunk_scores(ora.token_scores(x[l].q_obs, x[l].K, Hq, Hkv, w), c)
            assert_selection_matches(idx.cpu().numpy(), s, L, w, c, budget)
        else:                                             # (the layers of a pair have the same inputs)
            assert torch.equal(idx, outs[l - 2][2] if n_reuse == 1 else ck.compress_layer(*on[l % 2], Hq, w, c, budget)[2])


# Up to 64 rows and more than nine CTAs a head read the head's row statistics in a variant of their own (148 SMs, four selectors)
@pytest.mark.parametrize("Hq,Hkv,L,w", [(64, 16, 9 * 120, 16), (56, 14, 10 * 120, 16), (70, 14, 10 * 120 - 3, 13), (14, 14, 10 * 120 - 119, 1),
                                        (56, 14, 9 * 120, 16), (3, 1, 2500, 21)])
def test_model_call_with_few_rows(ck, Hq, Hkv, L, w):
    test_model_call(ck, Hq, Hkv, 64, L, w, 10, 2, 1)


# d = 128: a ring stage is 64 dims of a tile up to ten tiles a CTA (four CTAs a head of 32) and for two scoring heads, else a whole tile
@pytest.mark.parametrize("Hq,Hkv,L,w", [(32, 32, 40 * 128, 4), (32, 32, 40 * 128 + 1, 4), (64, 32, 4 * 23 * 128 - 77, 16), (160, 32, 2 * 11 * 128 + 5, 32)])
def test_token_scores_with_either_ring_stage(ck, Hq, Hkv, L, w):
    test_token_scores_and_chunk_scores_with_and_without_them(ck, Hq, Hkv, 128, L, w, 7)
