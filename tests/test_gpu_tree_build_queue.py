"""The pending queue of tree construction: one to sixteen registers per lane and the lines between them, chains, queues that run dry,
priorities that tie everywhere, entries of -inf; against the oracle."""
import numpy as np
import pytest

from jet_inputs import make_logp
from test_gpu_tree_build_scored import _compare as compare_scored

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode,alpha", [("accum_logp", 0.0), ("entropy", 0.0), ("hybrid", 0.5), ("hybrid", -3.0)])
@pytest.mark.parametrize("N,W,B", [(12, 7, 225), (12, 7, 226), (12, 7, 449), (12, 7, 450), (20, 2, 257), (20, 2, 258), (30, 2, 512), (64, 1, 512), (64, 1, 40), (1, 32, 512),
                                   (2, 3, 512), (16, 32, 512), (9, 8, 512), (40, 3, 193), (5, 4, 2), (64, 4, 257)])
def test_queue(N, W, B, mode, alpha):
    rng = np.random.default_rng(N * 1000 + B)
    sharp = np.stack([make_logp(rng, N, 997, 3.0, peaked_p=0.7) for _ in range(2)])
    flat = np.full((1, N, 997), -np.log(997.0), dtype=np.float32)        # every priority of a depth ties
    steps = -(1 + np.arange(997, dtype=np.float32) // 2)[None, None, :].repeat(N, axis=1)       # and sums of different paths do
    few = sharp[:1].copy()
    few[0, :, 3:] = -np.inf                                              # fewer finite entries than candidates
    l = np.concatenate([sharp, flat, steps, few]).astype(np.float32)
    compare_scored(l, np.arange(5), N, W, B, mode, alpha)
