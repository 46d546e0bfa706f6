"""Scratch of the one-launch layer kernel and of the persistent model kernel where their partial sums do not all stay on chip:
how much a shape asks for, and that a call writes nothing outside it."""
import ctypes

import pytest
import torch

from tests.helpers import Guarded

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ck():
    import paper_2502_00299_b200 as ck
    assert torch.cuda.is_available()
    yield ck
    ck.set_workspace(None)


def _layer(Hq, Hkv, d, L, w, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    q = torch.randn(Hq, w, d, device="cuda", generator=g).to(torch.bfloat16)
    K, V = (torch.randn(Hkv, L, d, device="cuda", dtype=torch.bfloat16, generator=g) for _ in range(2))
    return q, K, V


def test_scratch_grows_with_the_rows_that_exist(ck):
    # off-chip records are as wide as the rows: a few rows ask for a few MB, whatever 128 rows ask for
    for Hq, Hkv, d, L, w, c, limit in ((8, 8, 128, 131072, 8, 10, 7.0), (8, 8, 128, 131072, 8, 5, 14.0), (8, 8, 128, 131072, 16, 5, 22.0),
                                       (32, 32, 64, 16000, 8, 10, 4.2), (32, 32, 64, 65536, 8, 10, 12.0), (8, 8, 128, 131072, 1, 5, 6.5)):
        assert ck.workspace_bytes(L, Hq, Hkv, d, w, c) <= limit * 2 ** 20, (Hq, Hkv, L, w, c)


# shapes with off-chip records: one and two query tiles, rows no multiple of 4 or 32, few rows
SPILL = [(64, 16, 64, 9 * 120 * 22, 16, 10), (64, 32, 64, 4 * 120 * 30 + 7, 5, 5), (32, 32, 64, 4 * 128 * 33 - 3, 8, 8), (32, 32, 64, 4 * 120 * 23 + 1, 1, 5),
         (128, 32, 64, 4 * 120 * 23 + 61, 64, 20), (96, 32, 64, 4 * 128 * 40, 64, 16), (28 * 8, 32, 64, 4 * 120 * 20, 32, 10)]


@pytest.mark.parametrize("Hq,Hkv,d,L,w,c", SPILL)
def test_layer_and_model_calls_stay_inside_their_scratch(ck, Hq, Hkv, d, L, w, c):
    budget = w + c * ((L - w) // (5 * c))
    xs = [_layer(Hq, Hkv, d, L, w, seed=L + i) for i in range(3)]
    ck.set_workspace(None)
    free = [ck.compress_layer(*x, Hq, w, c, budget) for x in xs]           # (scratch with room to spare)
    scores = [ck.score(x[0], x[1], w, c)[0] for x in xs]
    ws = Guarded((ck.workspace_bytes(L, Hq, Hkv, d, w, c),), torch.uint8)
    ck.set_workspace(ws.t)
    for x, want, s in zip(xs, free, scores):
        got = ck.compress_layer(*x, Hq, w, c, budget)
        assert all(torch.equal(a, b) for a, b in zip(got, want))
        assert torch.equal(ck.score(x[0], x[1], w, c)[0], s)
    assert ck.device_status() == 0
    ws.check("layer scratch")
    ws = Guarded((int(ck.lib.chunkkv_model_workspace_bytes(len(xs), L, Hq, Hkv, d, w, c, budget, 1)),), torch.uint8)
    ck.set_workspace(ws.t)
    for _ in range(2):
        for got, want in zip(ck.compress_model(xs, Hq, w, c, budget, 1), free):
            assert all(torch.equal(a, b) for a, b in zip(got, want))
    assert ck.device_status() == 0
    ws.check("model scratch")


@pytest.mark.parametrize("Hq,Hkv,w,c", [(32, 8, 32, 20), (64, 8, 32, 10), (64, 8, 32, 5), (8, 8, 8, 5), (28, 4, 32, 16), (32, 8, 32, 32)])
def test_model_scratch_never_shrinks_for_a_longer_sequence(ck, Hq, Hkv, w, c):
    # so that a buffer sized for the longest prompt holds every shorter one
    lens = [*range(129400, 129700, 4), *range(w, 140000, 97)]
    need = [ck.lib.chunkkv_model_workspace_bytes(32, L, Hq, Hkv, 128, w, c, 4096, 1) for L in sorted(lens)]
    assert all(a <= b for a, b in zip(need, need[1:])), [L for L, a, b in zip(sorted(lens)[1:], need, need[1:]) if a > b][:5]


# Either side of lengths at which a tile more a CTA is due, and with it more or fewer selector CTAs: 6 heads 6 -> 4, 8 heads 8 -> 4 and back, 12
# heads 12 -> 4, 16 heads 16 -> 4 (5 and 7 heads keep as many)
@pytest.mark.parametrize("Hkv,L", [(5, 20160), (6, 16560), (7, 14400), (8, 12240), (8, 10200), (8, 10698), (12, 14520), (16, 15360)])
def test_model_call_in_scratch_sized_for_a_longer_sequence(ck, Hkv, L):
    d, w, c = 64, 8, 10
    budget = w + c * (L // (12 * c))
    ws = Guarded((int(ck.lib.chunkkv_model_workspace_bytes(2, L + 1, Hkv, Hkv, d, w, c, budget, 1)),), torch.uint8)
    for n in (L, L + 1):
        xs = [_layer(Hkv, Hkv, d, n, w, seed=n + i) for i in range(2)]
        ck.set_workspace(None)
        want = [ck.compress_layer(*x, Hkv, w, c, budget) for x in xs]
        n_max = ck.out_len(n, w, c, budget)
        outs = [(torch.empty(Hkv, n_max, d, dtype=torch.bfloat16, device="cuda"), torch.empty(Hkv, n_max, d, dtype=torch.bfloat16, device="cuda"),
                 torch.empty(Hkv, n_max, dtype=torch.int32, device="cuda")) for _ in xs]
        arr = ctypes.c_void_p * 2
        ck.set_workspace(ws.t)
        st = ck.lib.chunkkv_compress_model(2, *[arr(*[x[j].data_ptr() for x in xs]) for j in range(3)], n, Hkv, Hkv, d, w, c, budget, 1,
                                           *[arr(*[o[j].data_ptr() for o in outs]) for j in range(3)], None)
        assert st == 0 and ck.device_status() == 0
        assert all(torch.equal(a, b) for o, v in zip(outs, want) for a, b in zip(o, v))
    ws.check("model scratch")


@pytest.mark.parametrize("Hq,c,L,refused", [(8, 10, 20000, True), (8, 20, 20000, True), (8, 16, 20000, False), (8, 5, 9000, False),
                                            (8, 10, 120000, False)])
def test_model_call_on_a_scratch_of_the_layer_calls(ck, Hq, c, L, refused):
    # chunk sizes 10 and 20 need the model's scratch, as they always have, unless a CTA's key range is too long; the others
    # run layer by layer on the layer calls' scratch
    Hkv, d, w, n = 8, 64, 4, 96
    budget = w + c * (L // (6 * c))
    x = _layer(Hq, Hkv, d, L, w, seed=L + c)
    n_max = ck.out_len(L, w, c, budget)
    need, layers = (int(ck.lib.chunkkv_model_workspace_bytes(n, L, Hq, Hkv, d, w, c, budget, 3)), ck.workspace_bytes(L, Hq, Hkv, d, w, c))
    assert layers < need
    ck.set_workspace(None)
    want = ck.compress_layer(*x, Hq, w, c, budget)
    out = (torch.empty(n, Hkv, n_max, d, dtype=torch.bfloat16, device="cuda"), torch.empty(n, Hkv, n_max, d, dtype=torch.bfloat16, device="cuda"),
           torch.full((n, Hkv, n_max), -7, dtype=torch.int32, device="cuda"))
    arr = ctypes.c_void_p * n
    ptrs = [arr(*[t.data_ptr()] * n) for t in x] + [arr(*[o[l].data_ptr() for l in range(n)]) for o in out]

    def call(ws):
        ck.set_workspace(ws)
        return ck.lib.chunkkv_compress_model(n, *ptrs[:3], L, Hq, Hkv, d, w, c, budget, 3, *ptrs[3:], None)

    def same():
        assert ck.device_status() == 0
        return all(torch.equal(o[l], v) for o, v in zip((out[0], out[1], out[2]), want) for l in (0, 1, n - 1))

    ws = Guarded((layers,), torch.uint8)
    assert call(ws.t) == (-4 if refused else 0)
    assert bool((out[2] == -7).all()) if refused else same()
    ws.check("layer scratch")
    out[2].fill_(-7)
    assert call(Guarded((need,), torch.uint8).t) == 0 and same()
    assert call(torch.empty(4096, dtype=torch.uint8, device="cuda")) == -4
