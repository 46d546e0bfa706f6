"""What this library's users have it do, as cases that can be timed.

Compressing the KV cache at the end of a prefill: one layer at a time as an engine's layer loop calls it, whole
models in one call (with and without layer-wise index reuse), from token-major caches, into paged caches, with
the chunk sizes of the method's own ablation and at token level, and the scores alone for analysis. Lengths run from a
2K prompt to a 128K document; most are ragged, as real prompts are.
"""
import math

import torch

import paper_2502_00299_b200 as ck

# (query heads, KV heads, head dim): a small model, 8B-class and 70B-class grouped-query shapes, and an odd group of 7
SHAPES = ((8, 2, 64), (32, 8, 128), (64, 8, 128), (28, 4, 128))
SPAN = 12            # tokens that share one topic, and so one strength of attention
SINKS = 4            # the first tokens draw attention whatever they say


def _case(kind, name=None, Hq=32, Hkv=8, d=128, L=32768, w=32, c=10, budget=3276, layers=1, reuse=1, page=16):
    case = dict(kind=kind, Hq=Hq, Hkv=Hkv, d=d, L=L, w=w, c=c, budget=budget, layers=layers, reuse=reuse, page=page)
    return case if name is None else dict(case, name=name)


def listed():
    return [
        # the smallest call: a 2K prompt of a small model, where latency and the host path count
        _case("layer", "layer 2k", Hq=8, Hkv=2, d=64, L=2048, w=16, budget=256),
        # an ordinary prompt of an 8B-class model, one layer of the prefill loop
        _case("layer", "layer 8k", L=8192, budget=819),
        # the same model on a 32K document
        _case("layer", "layer 32k"),
        # a 128K document with a longer window and larger chunks: 256 score rows per KV head
        _case("layer", "layer 128k", L=131072, w=64, c=20, budget=4096),
        # a ragged prompt of a 70B-class model with chunks of 16 tokens (one cache page each)
        _case("layer", "layer 30k c16", Hq=64, L=29695, c=16, budget=2048),
        # token-level selection, as the later layers of a hybrid model use it
        _case("layer", "token level 32k", c=1),
        # a layer that reuses its neighbour's indices
        _case("reuse", "reuse 32k"),
        # a serving engine's layer: window queries out of the fused QKV activation, kept rows into a paged decode cache
        _case("serve", "serve paged 10k", Hq=64, L=10248, budget=2048),
        # a whole 32-layer model in one call
        _case("model", "model 32k x32", layers=32),
        # an 80-layer 70B-class model on a ragged prompt, indices shared by three layers
        _case("model", "model 42k x80 reuse 3", Hq=64, L=42450, budget=2048, layers=80, reuse=3),
        # a 32-layer model whose prefill cache is token-major, indices shared by two layers
        _case("token_major", "token-major 20k x32 reuse 2", L=19854, budget=1985, layers=32, reuse=2),
        # chunk and token scores of a layer, for analysis
        _case("scores", "scores 62k", L=62261, budget=2048),
    ]


def draw(rng):
    """One more case of these ranges."""
    kind = rng.choice(("layer", "layer", "layer", "layer", "reuse", "serve", "model", "model", "token_major", "scores"))
    Hq, Hkv, d = rng.choice(SHAPES)
    w = rng.choice((16, 32, 64) if Hq // Hkv <= 4 else (16, 32))
    c = rng.choice((5, 8, 10, 10, 10, 16, 20, 20, 32))
    whole = kind in ("model", "token_major")
    L = int(round(math.exp(rng.uniform(math.log(2048), math.log(32768 if whole else 131072)))))
    if kind == "layer" and rng.random() < 0.15:
        c, L = 1, min(L, 65536)
    budget = max(w + 4 * c, int(L * rng.uniform(0.03, 0.25)))
    case = _case(kind, Hq=Hq, Hkv=Hkv, d=d, L=L, w=w, c=c, budget=budget)
    if whole:
        case.update(layers=rng.randint(4, 32), reuse=rng.randint(1, 3))
    return case


def _layer(case, g, computes=True, token_major=False):
    """q_obs, K, V of one layer. Keys have a component along a direction that their head's window queries share;
    its strength varies from topic to topic, so the attention a token receives spreads over orders of magnitude."""
    Hq, Hkv, d, L, w = (case[k] for k in ("Hq", "Hkv", "d", "L", "w"))
    dev, bf16 = "cuda", torch.bfloat16
    u = torch.nn.functional.normalize(torch.randn(Hkv, 1, d, device=dev, generator=g), dim=-1)
    strength = torch.randn(Hkv, -(-L // SPAN), device=dev, generator=g).mul_(2.0 * math.sqrt(d) / 4.0)
    strength = strength.repeat_interleave(SPAN, 1)[:, :L].contiguous()
    strength[:, :SINKS] = 10.0 * math.sqrt(d) / 4.0
    lead = u.to(bf16) * strength.to(bf16)[:, :, None]
    if token_major:
        K = torch.randn(L, Hkv, d, device=dev, dtype=bf16, generator=g).permute(1, 0, 2)
        V = torch.randn(L, Hkv, d, device=dev, dtype=bf16, generator=g).permute(1, 0, 2)
    else:
        K = torch.randn(Hkv, L, d, device=dev, dtype=bf16, generator=g)
        V = torch.randn(Hkv, L, d, device=dev, dtype=bf16, generator=g)
    K += lead
    q = None
    if computes:
        q = torch.randn(Hkv, (Hq // Hkv) * w, d, device=dev, generator=g).add_(4.0 * u).to(bf16).view(Hq, w, d)
    return q, K, V


def prepare(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    Hq, Hkv, d, L, w, c, budget = (case[k] for k in ("Hq", "Hkv", "d", "L", "w", "c", "budget"))
    kind, n_max = case["kind"], ck.out_len(L, w, c, budget)
    s = {"case": case}
    if kind in ("model", "token_major"):
        n = case["layers"]
        s["layers"] = [_layer(case, g, l % case["reuse"] == 0, kind == "token_major") for l in range(n)]
        # the compacted caches that decoding reads afterwards, one allocation for all layers
        s["out"] = [torch.empty(n, Hkv, n_max, d, dtype=torch.bfloat16, device="cuda") for _ in range(2)]
        s["out"].append(torch.empty(n, Hkv, n_max, dtype=torch.int32, device="cuda"))
        s["outs"] = [tuple(o[l] for o in s["out"]) for l in range(n)]
        return s
    s["q"], s["K"], s["V"] = _layer(case, g)
    if kind == "reuse":
        # the neighbour's indices: whole chunks in ascending order, then the window
        k = (n_max - w) // c
        chunks = torch.rand(Hkv, (L - w) // c, device="cuda", generator=g).topk(k, dim=1).indices.sort(dim=1).values
        toks = (chunks[:, :, None] * c + torch.arange(c, device="cuda")).flatten(1)
        s["idx"] = torch.cat([toks, torch.arange(L - w, L, device="cuda").expand(Hkv, w)], 1).to(torch.int32).contiguous()
    elif kind == "serve":
        # the layer's QKV projection before the rotary embedding; the keys above are those of the cache, after it
        inv = 1.0 / (500000.0 ** (torch.arange(0, d, 2, device="cuda", dtype=torch.float64) / d))
        ang = torch.arange(L - w, L, device="cuda", dtype=torch.float64)[:, None] * inv[None, :]
        s["cos"], s["sin"] = ang.cos().float(), ang.sin().float()
        q = s.pop("q").float()
        half = d // 2
        cos, sin = s["cos"], s["sin"]
        un = torch.cat([q[..., :half] * cos + q[..., half:] * sin, q[..., half:] * cos - q[..., :half] * sin], -1)
        s["qkv"] = torch.randn(L, (Hq + 2 * Hkv) * d, device="cuda", dtype=torch.bfloat16, generator=g)
        s["qkv"][L - w:, :Hq * d] = un.transpose(0, 1).reshape(w, Hq * d).to(torch.bfloat16)
        pages = -(-n_max // case["page"])
        total = pages + pages // 4 + 1
        s["table"] = torch.randperm(total, device="cuda", generator=g)[:pages].to(torch.int32)
        s["cache"] = [torch.zeros(total, case["page"], Hkv, d, dtype=torch.bfloat16, device="cuda") for _ in range(2)]
    return s


def run(s):
    case = s["case"]
    kind, Hq, Hkv, d, w, c, budget = (case[k] for k in ("kind", "Hq", "Hkv", "d", "w", "c", "budget"))
    if kind == "layer":
        return ck.compress_layer(s["q"], s["K"], s["V"], Hq, w, c, budget)
    if kind == "reuse":
        return ck.compress_layer(None, s["K"], s["V"], Hq, w, c, budget, reuse_idx=s["idx"])
    if kind == "serve":
        q = ck.window_queries(s["qkv"], Hq, Hkv, d, w, s["cos"], s["sin"])
        idx = ck.compress_layer_paged(q, s["K"], s["V"], Hq, w, c, budget, s["table"], *s["cache"])
        return [q, idx, *s["cache"]]
    if kind == "scores":
        return ck.score(s["q"], s["K"], w, c, want_token_scores=True)
    call = ck.compress_model if kind == "model" else ck.compress_model_strided
    call(s["layers"], Hq, w, c, budget, case["reuse"], outs=s["outs"])
    return s["out"]


def work(case):
    Hq, Hkv, d, L, w, c, budget = (case[k] for k in ("Hq", "Hkv", "d", "L", "w", "c", "budget"))
    n_max = ck.out_len(L, w, c, budget)
    keys, q = Hkv * L * d * 2, Hq * w * d * 2
    rows, idx = 4 * Hkv * n_max * d * 2, Hkv * n_max * 4           # K and V rows read and written; indices written
    flops = 2 * Hq * w * L * d
    if case["kind"] == "reuse":
        return {"bytes": rows + 2 * idx, "flops": 0}
    if case["kind"] == "scores":
        return {"bytes": keys + q + 4 * Hkv * ((L - w) + -(-(L - w) // c)), "flops": flops}
    if case["kind"] == "serve":
        return {"bytes": keys + 2 * q + rows + idx, "flops": flops}
    n = case["layers"]
    computed = -(-n // case["reuse"])
    return {"bytes": computed * (keys + q) + n * (rows + idx), "flops": computed * flops}


def tolerance(case):
    # Scores: fp32 sums of exact bf16 products and of exponentials with a relative error of 2^-22. Against the same
    # sums in 64 bits the kernels differ by up to 4e-7 in the 2-norm and by up to 6.4e-7 in the worst value.
    if case["kind"] == "scores":
        return {"rel": 1.6e-6, "max": 2.6e-6}
    # Everything else is whole numbers and bit copies of rows. Two chunks would have to lie within rounding (1e-7) of
    # the k-th score for a selection to differ; neighbouring scores lie 3e-4 (tokens) to 2e-2 apart there.
    return "exact"


def exact(case, seed):
    """Chunk and token scores in 64 bits; the other calls' outputs are whole numbers and copies of rows."""
    if case["kind"] != "scores":
        return None
    Hq, Hkv, d, L, w, c = (case[k] for k in ("Hq", "Hkv", "d", "L", "w", "c"))
    s = prepare(case, seed)
    P = L - w
    chunks = torch.zeros(Hkv, -(-P // c), dtype=torch.float64, device="cuda")
    tokens = torch.zeros(Hkv, P, dtype=torch.float64, device="cuda")
    hidden = torch.arange(L, device="cuda")[None, :] > P + torch.arange(w, device="cuda")[:, None]
    q = s["q"].view(Hkv, Hq // Hkv, w, d)
    for h in range(Hkv):
        keys = s["K"][h].double()
        for g in range(Hq // Hkv):
            logits = (q[h, g].double() @ keys.T) / math.sqrt(d)
            tokens[h] += logits.masked_fill_(hidden, -math.inf).softmax(-1)[:, :P].sum(0)
    chunks.index_add_(1, torch.arange(P, device="cuda") // c, tokens)
    return chunks, tokens
