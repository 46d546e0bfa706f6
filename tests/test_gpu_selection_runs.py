"""The layer kernel's selection at the ends of runs of six and twelve ids a thread (576 threads), random scores and ties."""
import numpy as np
import pytest

from oracle import chunkkv_oracle as ora
from tests.helpers import assert_gather_exact, assert_selection_matches, bits_of, rand_bits, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tied", [False, True])
@pytest.mark.parametrize("C,k", [(3455, 3), (3456, 900), (3457, 3456), (6911, 1), (6912, 4000), (6913, 700)])
def test_layer_selection(C, k, tied):
    import paper_2502_00299_b200 as ck
    w, c, d = 16, 5, 64
    L = C * c + w - 3                                   # (a clipped last chunk)
    rng = np.random.default_rng(C)
    q, K, V = rand_bits(rng, (4, w, d)), rand_bits(rng, (1, L, d)), rand_bits(rng, (1, L, d))
    if tied:
        K[:, :] = K[:, :1]                              # every key the same: all whole chunks score the same, the lowest ids are kept
    oK, oV, idx = ck.compress_layer(*map(to_dev, (q, K, V)), 4, w, c, w + c * k)
    assert ck.device_status() == 0
    idx = idx.cpu().numpy()
    if tied:
        assert idx[0].tolist() == [*range(c * k), *range(L - w, L)]
    else:
        assert_selection_matches(idx, ora.chunk_scores(ora.token_scores(q, K, 4, 1, w), c), L, w, c, w + c * k)
    assert_gather_exact(bits_of(oK), bits_of(oV), idx, K, V)
