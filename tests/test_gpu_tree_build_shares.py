"""Tree construction with a sum over many aligned rows: the scan whose blocks take equal shares that begin and end inside rows
(some thousand rounds of 4096 entries), against the oracle: shares of whole rows, of parts, of several rows, a last round of
four entries, pieces without a finite entry, logits and log-probabilities that the table form does not cover."""
import numpy as np
import pytest

from jet_inputs import make_logp
from test_gpu_tree_build_logits import _compare as compare_logits
from test_gpu_tree_build_scored import _compare as compare_scored

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch,N,V", [(94, 16, 4100), (188, 16, 4), (50, 4, 4096 * 25), (2, 2, 4096 * 1250 + 4), (47, 8, 33000)])
def test_shares(batch, N, V):
    rng = np.random.default_rng(V)
    z = (rng.standard_normal((batch, N, V), dtype=np.float32) * 3).astype(np.float32)
    if V > 4:
        compare_logits(z, np.arange(batch), N, 3, 17, "hybrid", 0.5)
        z = z.astype(np.float64)
        z -= np.log(np.exp(z).sum(axis=2, keepdims=True))
        compare_scored(z.astype(np.float32), np.arange(batch), N, 3, 17, "hybrid", 0.5)
    else:
        compare_logits(z, np.arange(batch), N, 3, 17, "accum_logp", 0.0)


@pytest.mark.parametrize("offset,spread", [(6e4, 1.0), (-6e4, 1.0), (1.05e4, 30.0), (3e7, 1e7), (0.0, 3.0)])
def test_logits_beyond_the_table_form(offset, spread):
    rng = np.random.default_rng(9)
    z = (rng.standard_normal((100, 15, 8196)) * spread + offset).astype(np.float32)
    z[0, 0, 8195] = np.float32(offset + 5 * spread)
    z[:, 1, :4096] = -np.inf
    z[:, 2, 40:] = -np.inf
    z[0, 3, :] = -np.inf
    z[0, 3, 5] = 0.0
    compare_logits(z, np.arange(100), 15, 3, 9, "hybrid", 0.5)
    z[:, 4, 8195] = offset + 700                     # beyond what a reference from the first round can hold
    compare_logits(z, np.arange(100), 15, 3, 9, "accum_logp", 0.0)


def test_log_probabilities_zero_and_above():
    rng = np.random.default_rng(4)
    l = np.stack([make_logp(rng, 15, 8196, 3.0) for _ in range(100)])
    l[0, 0] = -np.inf
    l[0, 0, 17] = 0.0                                # one certain token: entropy exactly zero
    l[1, 2, 4099] = 0.5
    l[2, 3, 4] = -1e-41
    compare_scored(l, np.arange(100), 15, 3, 9, "entropy", 0.0)
