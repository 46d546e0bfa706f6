"""The end of the tags by which launches hand values over: words of old launches are cleared before the tags start over, and the
launches around it agree with those before. The last tag is set near the end, which takes 2^32 - 1 launches otherwise."""
import ctypes

import numpy as np
import pytest
import torch

from tests.helpers import rand_bits, to_dev

pytestmark = pytest.mark.gpu

LAST = 0xffffffff


@pytest.mark.parametrize("c", [10, 1])                  # layer kernel, token kernel
def test_launches_over_the_last_tag(c):
    import paper_2502_00299_b200 as ck
    Hq, Hkv, d, w = 8, 2, 64, 16
    rng = np.random.default_rng(c)

    def inputs(L):
        return tuple(map(to_dev, (rand_bits(rng, (Hq, w, d)), rand_bits(rng, (Hkv, L, d)), rand_bits(rng, (Hkv, L, d)))))

    def layers(xs):
        return [ck.compress_layer(*x, Hq, w, c, 216) for x in xs]

    def same(got, want):
        return ck.device_status() == 0 and all(torch.equal(a, b) for g, r in zip(got, want) for a, b in zip(g, r))

    def last_tag(tag):
        assert ck.lib.chunkkv_test_last_tag(ctypes.c_uint(tag)) == 0

    # twice over the end, then some launches with the first tags. (The layer kernel has few CTAs for `few`, the token kernel always all.)
    many, few, others = [inputs(4000) for _ in range(4)], [inputs(300) for _ in range(3)], [inputs(4000) for _ in range(4)]
    want = [layers(x) for x in (many, few, others)]
    last_tag(LAST - 3)
    assert same(layers(few), want[1])
    assert same(layers(many), want[0])                  # tags 1 to 4
    last_tag(LAST - 3)
    assert same(layers(few), want[1])                   # the last three; the layer kernel leaves words of `many`
    assert same(layers(others), want[2])                # tags 1 to 4 again: those words must be gone
