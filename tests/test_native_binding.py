"""The binding's native calls (csrc/native.cpp): what they decline goes the general way, and both ways give the same results."""
import os
import subprocess
import sys

import numpy as np
import pytest
import torch
from torch.utils._python_dispatch import TorchDispatchMode

import paper_2502_00299_b200 as ck
from paper_2502_00299_b200 import binding, build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CALLS = ("layer", "layer_strided", "layer_alg1", "layer_paged", "window_queries", "score", "model")


def test_declined_arguments_raise_what_the_general_way_raises():
    x = torch.zeros(2, 64, 64, dtype=torch.bfloat16)               # not on a GPU
    for call in (lambda: ck.compress_layer(x, x, x, 4, 16, 8, 32), lambda: ck.compress_layer_strided(x, x, x, 4, 16, 8, 32),
                 lambda: ck.compress_layer_paged(x, x, x, 4, 16, 8, 32, x, x[None], x[None]),
                 lambda: ck.compress_layer_alg1(x, x, x, 4, 16, 8, 32), lambda: ck.score(x, x, 16, 8),
                 lambda: ck.compress_model([(x, x, x)], 4, 16, 8, 32), lambda: ck.compress_model_strided([(x, x, x)], 4, 16, 8, 32),
                 lambda: ck.window_queries(x[0], 1, 1, 64, 16, x[0], x[0])):
        with pytest.raises(ValueError):
            call()
    with pytest.raises(AttributeError):
        ck.compress_layer(None, None, None, 4, 16, 8, 32)
    for name in CALLS:
        with pytest.raises(TypeError):
            getattr(binding._native, name)(1, 2, 3)


class Fake:
    """What the general way looks at of a CUDA tensor; nothing is behind it."""

    def __init__(self, *shape, dtype=torch.bfloat16, cuda=True, contiguous=True):
        self.shape, self.dtype, self.is_cuda, self.device, self._contiguous = torch.Size(shape), dtype, cuda, torch.device("cuda"), contiguous

    def is_contiguous(self):
        return self._contiguous

    def numel(self):
        return self.shape.numel()

    def dim(self):
        return len(self.shape)

    def stride(self, i):
        return self.shape[i + 1:].numel()

    def data_ptr(self):
        raise AssertionError("the pointer of a tensor that should have been refused")


def _refused(call, good, bad):
    """`good` passes the checks (and ends where a device is asked for, in data_ptr where there is one); each of `bad` in its place does not."""
    with pytest.raises((RuntimeError, AssertionError)):
        call(**good)
    for name, values in bad.items():
        for v in values:
            with pytest.raises(ValueError, match=name):
                call(**{**good, name: v})


def test_paged_layer_call_checks_its_tensors():
    Hq, Hkv, d, L, w, c, budget, page = 8, 2, 64, 300, 16, 10, 100, 16
    n = ck.out_len(L, w, c, budget)
    i32 = torch.int32
    good = dict(q_obs=Fake(Hq, w, d), K=Fake(Hkv, L, d), V=Fake(Hkv, L, d), block_table=Fake(-(-n // page), dtype=i32),
                cache_K=Fake(9, page, Hkv, d), cache_V=Fake(9, page, Hkv, d))
    kinds = lambda *s: [Fake(*s, cuda=False), Fake(*s, dtype=torch.float16), Fake(*s, contiguous=False)]
    bad = {"q_obs": kinds(Hq, w, d) + [Fake(Hq, w - 1, d)], "K": kinds(Hkv, L, d), "V": kinds(Hkv, L, d) + [Fake(Hkv, L - 1, d)],
           "block_table": [Fake(9, dtype=torch.int64), Fake(9, dtype=i32, cuda=False), Fake(-(-n // page) - 1, dtype=i32)],
           "cache_K": kinds(9, page, Hkv, d) + [Fake(9, page, 1, d)], "cache_V": kinds(9, page, Hkv, d) + [Fake(8, page, Hkv, d)]}
    call = lambda **k: ck.compress_layer_paged(k.pop("q_obs"), k.pop("K"), k.pop("V"), Hq, w, c, budget, **k)
    _refused(call, good, bad)
    idx = Fake(Hkv, n, dtype=i32)
    _refused(call, {**good, "q_obs": None, "reuse_idx": idx}, {"reuse_idx": [Fake(Hkv, n, dtype=torch.int64), Fake(Hkv, n - 1, dtype=i32)]})


def test_given_outputs_are_checked():
    Hq, Hkv, d, L, w, c, budget = 8, 2, 64, 300, 16, 10, 100
    i32 = torch.int32
    q, K, V = Fake(Hq, w, d), Fake(Hkv, L, d), Fake(Hkv, L, d)
    for call, n in ((ck.compress_layer, ck.out_len(L, w, c, budget)), (ck.compress_layer_strided, ck.out_len(L, w, c, budget)),
                    (ck.compress_layer_alg1, ck.out_len_alg1(L, w, c, budget)), (ck.compress_model, ck.out_len(L, w, c, budget)),
                    (ck.compress_model_strided, ck.out_len(L, w, c, budget))):
        rows = lambda: Fake(Hkv, n, d)
        kinds = lambda *s: [Fake(*s, cuda=False), Fake(*s, dtype=torch.float32), Fake(*s, contiguous=False), Fake(s[0], s[1] - 1, *s[2:])]
        bad = {"out_K": kinds(Hkv, n, d), "out_V": kinds(Hkv, n, d), "out_idx": [Fake(Hkv, n, dtype=torch.int64), Fake(Hkv, n - 1, dtype=i32), Fake(Hkv, n, dtype=i32, cuda=False)]}
        if call in (ck.compress_model, ck.compress_model_strided):
            one = lambda out_K, out_V, out_idx: call([(q, K, V)] * 2, Hq, w, c, budget, 2, outs=[(rows(), rows(), Fake(Hkv, n, dtype=i32)), (out_K, out_V, out_idx)])
        else:
            one = lambda **k: call(q, K, V, Hq, w, c, budget, **k)
        _refused(one, dict(out_K=rows(), out_V=rows(), out_idx=Fake(Hkv, n, dtype=i32)), bad)
    n = 40
    _refused(lambda **k: ck.gather(K, V, Fake(Hkv, n, dtype=i32), **k), dict(out_K=Fake(Hkv, n, d), out_V=Fake(Hkv, n, d)),
             {"out_K": [Fake(Hkv, n - 1, d)], "out_V": [Fake(Hkv, n, d, cuda=False)]})


def test_inputs_that_are_too_small_are_refused():
    Hq, Hkv, d, L, w, c, budget, n = 8, 2, 64, 300, 16, 10, 100, 96
    assert ck.out_len(L, w, c, budget) == n
    i32, f32 = torch.int32, torch.float32
    good = dict(q_obs=Fake(Hq, w, d), K=Fake(Hkv, L, d), V=Fake(Hkv, L, d))
    bad = {"q_obs": [Fake(Hq, w - 1, d)], "V": [Fake(Hkv, L - 1, d), Fake(1, L, d)]}
    sizes = (Hq, w, c, budget)
    for call in (ck.compress_layer, ck.compress_layer_strided, ck.compress_layer_alg1):
        _refused(lambda q_obs, K, V: call(q_obs, K, V, *sizes), good, bad)
    for call in (ck.compress_layer, ck.compress_layer_strided):
        _refused(lambda reuse_idx: call(None, good["K"], good["V"], *sizes, reuse_idx=reuse_idx), dict(reuse_idx=Fake(Hkv, n, dtype=i32)),
                 {"reuse_idx": [Fake(Hkv, n - 1, dtype=i32)]})
    for call in (ck.compress_model, ck.compress_model_strided):
        _refused(lambda q_obs, K, V: call([(q_obs, K, V)], *sizes), good, {"q_obs": bad["q_obs"]})
    _refused(lambda q_obs, K: ck.score(q_obs, K, w, c), dict(q_obs=good["q_obs"], K=good["K"]), {"q_obs": bad["q_obs"], "K": [Fake(Hkv, L, d - 1)]})
    _refused(lambda V, idx: ck.gather(good["K"], V, idx), dict(V=good["V"], idx=Fake(Hkv, n, dtype=i32)), {"V": bad["V"], "idx": [Fake(1, n, dtype=i32)]})
    _refused(lambda cos_rows, sin_rows: ck.window_queries(Fake(L, (Hq + 2 * Hkv) * d), Hq, Hkv, d, w, cos_rows, sin_rows),
             dict(cos_rows=Fake(w, d // 2, dtype=f32), sin_rows=Fake(w, d // 2, dtype=f32)),
             {"cos_rows": [Fake(w - 1, d // 2, dtype=f32)], "sin_rows": [Fake(w - 1, d // 2, dtype=f32)]})
    table, cache = Fake(6, dtype=i32), lambda h=Hkv: Fake(9, 16, h, d)
    _refused(lambda V, block_table, cache_V: ck.gather_paged(good["K"], V, Fake(Hkv, n, dtype=i32), block_table, cache(), cache_V),
             dict(V=good["V"], block_table=table, cache_V=cache()), {"V": bad["V"], "block_table": [Fake(5, dtype=i32)], "cache_V": [cache(1)]})
    _refused(lambda V, block_table, cache_V: ck.compress_model_paged([(good["q_obs"], good["K"], V)], *sizes, [block_table], [(cache(), cache_V)]),
             dict(V=good["V"], block_table=table, cache_V=cache()), {"V": bad["V"], "block_table": [Fake(5, dtype=i32)], "cache_V": [cache(1)]})


@pytest.mark.gpu
def test_native_calls_decline_inputs_that_are_too_small():
    Hq, Hkv, d, L, w, c, budget = 8, 2, 64, 300, 16, 10, 100
    n, bf = ck.out_len(L, w, c, budget), torch.bfloat16
    ck.set_workspace(torch.empty(64 << 20, dtype=torch.uint8, device="cuda"))
    z = lambda *s, dtype=bf: torch.zeros(*s, dtype=dtype, device="cuda")
    q, K, V, sizes, N = z(Hq, w, d), z(Hkv, L, d), z(Hkv, L, d), (Hq, w, c, budget), binding._native
    idx, ang = z(Hkv, n, dtype=torch.int32), z(w, d // 2, dtype=torch.float32)
    less = lambda t: t.flatten()[:-1].contiguous()
    few = z(Hq, w - 1, d)
    for call, args in ((lambda *a: N.layer(*a, *sizes, None, None, None, None, None), (q, K, V)), (lambda *a: N.layer_alg1(*a, *sizes, None, None, None, None), (q, K, V)),
                       (lambda r: N.layer(None, K, V, *sizes, r, None, None, None, None), (idx,)), (lambda q: N.score(q, K, w, c, True, None), (q,)),
                       (lambda a, b: N.window_queries(z(L, (Hq + 2 * Hkv) * d), Hq, Hkv, d, w, a, b, None), (ang, ang))):
        assert call(*args) is not None
        for i, t in enumerate(args):
            if t is not K:
                small = few if t is q else less(t)
                assert call(*[small if j == i else x for j, x in enumerate(args)]) is None, i
    for strided in (False, True):
        assert N.model([(q, K, V)], *sizes, 1, None, None, strided) is not None and N.model([(few, K, V)], *sizes, 1, None, None, strided) is None
    assert N.layer_strided(q, K, V[:, 1:], *sizes, None, None, None, None, None) is None
    assert ck.device_status() == 0


@pytest.mark.gpu
def test_native_calls_decline_outputs_that_the_general_way_refuses():
    Hq, Hkv, d, L, w, c, budget = 8, 2, 64, 300, 16, 10, 100
    n, n1, bf, i32 = ck.out_len(L, w, c, budget), ck.out_len_alg1(L, w, c, budget), torch.bfloat16, torch.int32
    ck.set_workspace(torch.empty(64 << 20, dtype=torch.uint8, device="cuda"))
    z = lambda *s, dtype=bf: torch.zeros(*s, dtype=dtype, device="cuda")
    q, K, V, sizes = z(Hq, w, d), z(Hkv, L, d), z(Hkv, L, d), (Hq, w, c, budget)
    N = binding._native
    calls = [(lambda *o: N.layer(q, K, V, *sizes, None, *o, None), n), (lambda *o: N.layer_strided(q, K, V, *sizes, None, *o, None), n),
             (lambda *o: N.layer_alg1(q, K, V, *sizes, *o, None), n1), (lambda *o: N.model([(q, K, V)], *sizes, 1, None, [o], False), n),
             (lambda *o: N.model([(q, K, V)], *sizes, 1, None, [o], True), n)]
    for call, m in calls:
        good = [z(Hkv, m, d), z(Hkv, m, d), z(Hkv, m, dtype=i32)]
        assert call(*good) is not None
        for i, t in ((0, z(Hkv, m, d).cpu()), (0, z(Hkv, m - 1, d)), (0, z(Hkv, d, m).transpose(1, 2)), (1, z(Hkv, m, d, dtype=torch.float16)), (1, z(Hkv, m - 1, d)),
                     (2, z(Hkv, m, dtype=torch.int64)), (2, z(Hkv, m - 1, dtype=i32)), (2, z(Hkv, m, dtype=i32).cpu())):
            assert call(*[t if j == i else x for j, x in enumerate(good)]) is None, i
    assert ck.device_status() == 0


@pytest.mark.gpu
def test_native_paged_layer_call_declines_what_the_general_way_refuses():
    Hq, Hkv, d, L, w, c, budget = 8, 2, 64, 300, 16, 10, 100
    n, bf = ck.out_len(L, w, c, budget), torch.bfloat16
    ck.ensure_workspace(L, Hq, Hkv, d, w, c)
    z = lambda *s, dtype=bf: torch.zeros(*s, dtype=dtype, device="cuda")
    good = [z(Hq, w, d), z(Hkv, L, d), z(Hkv, L, d), Hq, w, c, budget, torch.arange(9, dtype=torch.int32, device="cuda"), z(9, 16, Hkv, d), z(9, 16, Hkv, d),
            None, None, None]
    assert binding._native.layer_paged(*good) is not None
    for i, t in ((0, z(Hq, w - 1, d)), (1, z(Hkv, d, L).transpose(1, 2)), (1, z(Hkv, L, d).cpu()), (2, z(Hkv, L - 1, d)), (2, z(Hkv, L, d, dtype=torch.float16)),
                 (7, torch.arange(9, device="cuda")), (7, good[7][:5]), (7, good[7].cpu()), (8, z(9, 16, 1, d)), (9, z(8, 16, Hkv, d)),
                 (9, z(9, Hkv, 16, d).transpose(1, 2)), (10, z(Hkv, n, dtype=torch.int64)), (10, z(Hkv, n - 1, dtype=torch.int32))):
        assert binding._native.layer_paged(*[t if j == i else x for j, x in enumerate(good)]) is None, i
    assert ck.device_status() == 0


def _general(monkeypatch):
    for name in CALLS:
        monkeypatch.setattr(binding._native, name, lambda *a: None)


def _cases(g):
    Hq, Hkv, d, L, w, c, budget = 8, 2, 64, 1111, 16, 10, 200
    bf = torch.bfloat16
    q, K, V = (torch.randn(*s, device="cuda", generator=g).to(bf) for s in ((Hq, w, d), (Hkv, L, d), (Hkv, L, d)))
    n = ck.out_len(L, w, c, budget)
    tm = [t.permute(1, 0, 2).contiguous().permute(1, 0, 2) for t in (K, V)]
    idx = torch.stack([torch.randperm(L, device="cuda", generator=g)[:n].sort().values for _ in range(Hkv)]).to(torch.int32)
    outs = lambda: (torch.zeros(Hkv, n, d, dtype=bf, device="cuda"), torch.zeros(Hkv, n, d, dtype=bf, device="cuda"),
                    torch.zeros(Hkv, n, dtype=torch.int32, device="cuda"))
    kw = lambda o: dict(out_K=o[0], out_V=o[1], out_idx=o[2])
    table = torch.randperm(20, device="cuda", generator=g)[:-(-n // 16)].to(torch.int32)
    qkv = torch.randn(300, (Hq + 2 * Hkv) * d, device="cuda", generator=g).to(bf)
    ang = torch.rand(w, d // 2, device="cuda", generator=g)
    side = torch.cuda.Stream()

    def paged(**more):
        cache = [torch.zeros(20, 16, Hkv, d, dtype=bf, device="cuda") for _ in range(2)]
        return [ck.compress_layer_paged(q, K, V, Hq, w, c, budget, table, *cache, **more), *cache]

    def on_side():
        o = outs()
        side.wait_stream(torch.cuda.current_stream())
        r = ck.compress_layer(q, K, V, Hq, w, c, budget, stream=side, **kw(o))
        torch.cuda.current_stream().wait_stream(side)
        return r
    layers = [(q, K, V), (None, V, K), (q, V, K)]
    strided = [(q, tm[0], tm[1]), (None, tm[1], tm[0])]
    return [lambda: ck.compress_layer(q, K, V, Hq, w, c, budget), lambda: ck.compress_layer(q, K, V, Hq, w, c, budget, **kw(outs())),
            lambda: ck.compress_layer(None, K, V, Hq, w, c, budget, reuse_idx=idx), lambda: ck.compress_layer(q, K, V, Hq, w, 1, budget),
            lambda: ck.compress_layer(q, K, V, np.int64(Hq), w, c, np.int32(budget)), on_side,
            lambda: ck.compress_layer_strided(q, *tm, Hq, w, c, budget), lambda: ck.compress_layer_strided(None, *tm, Hq, w, c, budget, reuse_idx=idx),
            lambda: ck.compress_layer_alg1(q, K, V, Hq, w, c, budget), lambda: paged(), lambda: paged(reuse_idx=idx),
            lambda: [ck.window_queries(qkv, Hq, Hkv, d, w, ang.cos(), ang.sin())], lambda: ck.score(q, K, w, c)[:1],
            lambda: ck.score(q, K, w, c, want_token_scores=True),
            lambda: sum(ck.compress_model(layers, Hq, w, c, budget, 2), ()),
            lambda: sum(ck.compress_model(layers, Hq, w, c, budget, 2, outs=[outs() for _ in layers]), ()),
            lambda: sum(ck.compress_model(tuple(layers), Hq, w, c, budget, 2, outs=tuple(list(outs()) for _ in layers)), ()),
            lambda: sum(ck.compress_model_strided(strided, Hq, w, c, budget, 2), ())]


DECLINED = (4, 16)      # of these: numpy ints, outputs as lists


@pytest.mark.gpu
def test_native_and_general_results_are_the_same(monkeypatch):
    cases = _cases(torch.Generator(device="cuda").manual_seed(5))
    for call in cases:                                    # (the scratch grows in the general way)
        call()
    answers = []
    with monkeypatch.context() as m:
        for name in CALLS:
            def spy(*a, f=getattr(binding._native, name)):
                answers.append(f(*a))
                return answers[-1]
            m.setattr(binding._native, name, spy)
        native = []
        for i, call in enumerate(cases):
            answers.clear()
            native.append(call())
            assert [a is None for a in answers] == [i in DECLINED], i
    _general(monkeypatch)
    for i, (got, call) in enumerate(zip(native, cases)):
        want = call()
        assert len(got) == len(want), i
        for x, y in zip(got, want):
            assert x.shape == y.shape and x.dtype == y.dtype and x.device == y.device and torch.equal(x, y), i
    assert ck.device_status() == 0


@pytest.mark.gpu
def test_native_errors_and_growing_scratch():
    g = torch.Generator(device="cuda").manual_seed(6)
    q, K, V = (torch.randn(*s, device="cuda", generator=g).to(torch.bfloat16) for s in ((8, 16, 64), (2, 900, 64), (2, 900, 64)))
    for bad in (dict(budget=4), dict(c=0), dict(w=901)):             # sizes
        with pytest.raises(ck.ChunkKVError) as e:
            ck.compress_layer(q, K, V, 8, **{**dict(w=16, c=10, budget=100), **bad})
        assert e.value.status == -2
    with pytest.raises(ck.ChunkKVError) as e:                        # a status of the C ABI
        ck.compress_layer(None, K, V, 8, 16, 10, 100)
    assert e.value.status == -1 and "chunkkv_compress_layer" in str(e.value)
    with pytest.raises(ValueError):
        ck.compress_layer(q, K.transpose(0, 1), V, 8, 16, 10, 100)
    ck.set_workspace(torch.empty(8192, dtype=torch.uint8, device="cuda"))
    want = ck.compress_layer(q, K, V, 8, 16, 10, 100)                # too small: replaced by a larger one
    assert binding._workspaces[torch.cuda.current_device()].numel() > 8192
    for x, y in zip(ck.compress_layer(q, K, V, 8, 16, 10, 100), want):
        assert torch.equal(x, y)
    assert ck.device_status() == 0


class _Empties(TorchDispatchMode):
    """Empties a list when a tensor is allocated."""

    def __init__(self, victim):
        super().__init__()
        self.victim, self.hits = victim, 0

    def __torch_dispatch__(self, func, types, args=(), kwargs=None):
        if "empty" in str(func):
            self.hits += 1
            self.victim.clear()
        return func(*args, **(kwargs or {}))


@pytest.mark.gpu
def test_layers_list_that_changes_while_outputs_are_allocated():
    g = torch.Generator(device="cuda").manual_seed(7)
    make = lambda *s: torch.randn(*s, device="cuda", generator=g).to(torch.bfloat16)
    xs = [(make(8, 16, 64), make(2, 900, 64), make(2, 900, 64)) for _ in range(3)]
    ck.set_workspace(torch.empty(64 << 20, dtype=torch.uint8, device="cuda"))
    want = ck.compress_model(xs, 8, 16, 10, 100)
    layers = [list(x) for x in xs]
    with _Empties(layers) as mode:
        got = binding._native.model(layers, 8, 16, 10, 100, 1, None, None, False)
    assert mode.hits == 9 and layers == [] and len(got) == 3
    assert all(torch.equal(a, b) for x, y in zip(got, want) for a, b in zip(x, y))
    assert ck.device_status() == 0


def test_scratch_is_looked_up_where_the_binding_keeps_it():
    # (loaded again, the binding has no scratch, and the native calls must not take the old one for granted)
    code = ("import importlib; from paper_2502_00299_b200 import binding as b; t = b._native.scratch(); assert t is b._workspaces; "
            "b = importlib.reload(b); assert b._native.scratch() is b._workspaces is not t")
    subprocess.run([sys.executable, "-c", code], check=True, cwd=ROOT)


def test_without_the_native_part_calls_go_the_general_way(monkeypatch):
    monkeypatch.setattr(torch, "__version__", "0.0.1")              # built for another torch
    assert not build.is_current()
    with pytest.warns(RuntimeWarning, match="paper_2502_00299_b200.build"):
        none = binding._load_native()
    for name in CALLS:
        assert getattr(none, name)(1, 2, 3) is None
    monkeypatch.undo()
    assert binding._load_native().scratch.__name__ == "scratch" and build.is_current()
