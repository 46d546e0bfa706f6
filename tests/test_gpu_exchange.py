"""The tagged words of captured calls: graphs over different scratch run side by side, beside calls on a third."""
import numpy as np
import pytest
import torch

from tests.helpers import rand_bits, to_dev

pytestmark = pytest.mark.gpu


def _inputs(n, Hq, Hkv, d, L, w, seed):
    rng = np.random.default_rng(seed)
    return [tuple(map(to_dev, (rand_bits(rng, (Hq, w, d)), rand_bits(rng, (Hkv, L, d)), rand_bits(rng, (Hkv, L, d))))) for _ in range(n)]


def test_graphs_over_different_scratch_side_by_side():
    # launches of 6 CTAs each, so that those of all three streams are resident together; every one meets words of others before it
    import paper_2502_00299_b200 as ck
    Hq, Hkv, d, L, w, c, budget = 8, 2, 64, 300, 16, 10, 116
    xs = [_inputs(12, Hq, Hkv, d, L, w, seed=i) for i in range(3)]
    want = [[ck.compress_layer(*x, Hq, w, c, budget) for x in part] for part in xs]
    bytes_ = ck.workspace_bytes(L, Hq, Hkv, d, w, c)
    streams = [torch.cuda.Stream() for _ in range(3)]
    graphs, outs, scratch = [], [], [torch.empty(bytes_, dtype=torch.uint8, device="cuda") for _ in range(3)]
    try:
        for i in range(2):
            ck.set_workspace(scratch[i])
            graphs.append(torch.cuda.CUDAGraph())
            with torch.cuda.graph(graphs[i], stream=streams[i]):
                outs.append([ck.compress_layer(*x, Hq, w, c, budget) for x in xs[i]])
        ck.set_workspace(scratch[2])
        for _ in range(40):
            for part in outs:
                for o in part:
                    o[2].fill_(-7)
            torch.cuda.synchronize()
            for i in range(2):
                with torch.cuda.stream(streams[i]):
                    graphs[i].replay()
            with torch.cuda.stream(streams[2]):
                eager = [ck.compress_layer(*x, Hq, w, c, budget) for x in xs[2]]
            torch.cuda.synchronize()
            assert all(int(b[:4].view(torch.int32)) == 0 for b in scratch)       # (their status words)
            for got, ref in zip([*outs, eager], want):
                assert all(torch.equal(a, b) for g, r in zip(got, ref) for a, b in zip(g, r))
    finally:
        ck.set_workspace(None)


BEYOND = """
import numpy as np, torch
import paper_2502_00299_b200 as ck
from oracle import chunkkv_oracle as ora
from tests.helpers import assert_gather_exact, assert_selection_matches, bits_of, rand_bits, to_dev
keep = []
x = [torch.randn(8, 16, 64, device="cuda").bfloat16(), *(torch.randn(2, 300, 64, device="cuda").bfloat16() for _ in range(2))]
for i in range(8):
    keep.append(torch.empty(2 << 20, dtype=torch.uint8, device="cuda"))
    ck.set_workspace(keep[-1])
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        keep.append(ck.compress_layer(*x, 8, 16, 10, 116))
    keep.append(g)
ck.set_workspace(torch.empty(256 << 20, dtype=torch.uint8, device="cuda"))
for Hq, Hkv, d, L, w, c in ((8, 2, 64, 3000, 16, 10), (32, 8, 128, 5000, 32, 20), (64, 16, 64, 23760, 16, 10), (8, 2, 64, 2000, 16, 1)):
    budget = w + c * ((L - w) // (5 * c))
    rng = np.random.default_rng(L)
    xs = [(rand_bits(rng, (Hq, w, d)), rand_bits(rng, (Hkv, L, d)), rand_bits(rng, (Hkv, L, d))) for _ in range(2)]
    outs = [ck.compress_layer(*map(to_dev, xs[i % 2]), Hq, w, c, budget) for i in range(4)]
    assert ck.device_status() == 0
    for i, (oK, oV, idx) in enumerate(outs):
        q, K, V = xs[i % 2]
        assert_selection_matches(idx.cpu().numpy(), ora.chunk_scores(ora.token_scores(q, K, Hq, Hkv, w), c), L, w, c, budget)
        assert_gather_exact(bits_of(oK), bits_of(oV), idx.cpu().numpy(), K, V)
"""


def test_calls_on_a_scratch_that_finds_no_words_left():
    # in a process of its own: the eight that take them keep them
    import os
    import subprocess
    import sys
    r = subprocess.run([sys.executable, "-c", BEYOND], cwd=os.path.dirname(os.path.dirname(os.path.abspath(__file__))), capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-1500:]
