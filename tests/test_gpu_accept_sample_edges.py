"""GPU parity of the sampling acceptance where its split of the vocabulary turns: less than a step per warp, exactly one, a
remainder behind the two steps a warp loads together, rows that are not 16-byte aligned, the largest tree."""
import numpy as np
import pytest

from test_gpu_tree_accept_sample import _built, _check, _target_near_draft

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("V,B", [(130, 5), (16384, 31), (16385, 33), (32768, 16), (32769, 16), (49281, 64), (4100, 512)])
def test_splits_of_the_vocabulary(V, B):
    rng = np.random.default_rng(7900 + V)
    logp, token, parent, depth, anc, n = _built(rng, 2, 4, 4, B, V, 3.0)
    logits = _target_near_draft(rng, logp, token, parent, depth, n, B, V, 0.6)
    _check(logits, 0.8, logp, token, parent, depth, anc, n, 4, rng)
