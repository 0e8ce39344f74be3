"""Tree construction where the row scan and the expansion change form: slices and rounds of the scan (rows of 4096 entries
and their edges, few and many rows), group maxima beyond a warp's registers, more qualifying groups or candidates than
the fast form holds, the number of queue registers, logits the table-driven exponential does not cover."""
import numpy as np
import pytest

from jet_inputs import make_draft_logits, make_logp
from test_gpu_tree_build_logits import _compare as compare_logits
from test_gpu_tree_build_scored import _compare as compare_scored

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("V", [127, 128, 129, 4095, 4096, 4097, 8192 + 4, 163840, 163841, 200003])
def test_row_lengths_at_the_edges_of_slices_and_groups(V):
    rng = np.random.default_rng(V)
    compare_scored(np.stack([make_logp(rng, 3, V, 3.0, peaked_p=0.6)]), [7], 3, 7, 40, "hybrid", 0.5)
    compare_logits(np.stack([make_draft_logits(rng, 3, V, 3.0)]), [7], 3, 7, 40, "accum_logp", 0.0)


@pytest.mark.parametrize("batch,N", [(1, 16), (14, 16), (28, 16), (60, 16)])     # one, two and four rounds of the scan per block
def test_rounds_per_block(batch, N):
    rng = np.random.default_rng(batch)
    V = 4096 * 4 + 260
    z = (rng.standard_normal((batch, N, V)) * 3).astype(np.float32)
    compare_logits(z, np.arange(batch), N, 5, 33, "hybrid", 0.5)


@pytest.mark.parametrize("W", [1, 7, 32])
@pytest.mark.parametrize("kind", ["flat", "steps", "one_group", "ramp", "masked"])
def test_rows_with_many_nearly_equal_entries(kind, W):
    rng = np.random.default_rng(5)
    V = 20000
    z = np.zeros((1, 3, V), np.float32)
    if kind == "steps":
        z += rng.integers(0, 3, z.shape).astype(np.float32)
    elif kind == "one_group":                        # a whole group of entries within one rounding step of each other
        z[:, :, 5000:5128] = 9.0 + np.arange(128, dtype=np.float32) * np.float32(1e-7)
        z[:, :, 100] = 24.0
    elif kind == "ramp":
        z += np.arange(V, dtype=np.float32) * np.float32(1e-6)
    elif kind == "masked":
        z[:, :, 40:] = -np.inf
    compare_logits(z, [3], 3, W, 60, "accum_logp", 0.0)
    compare_logits(z, [3], 3, W, 60, "hybrid", 1.0)


@pytest.mark.parametrize("W,B", [(1, 33), (1, 34), (2, 65), (2, 67), (4, 512), (3, 512), (2, 512), (1, 512), (7, 226), (7, 227)])
@pytest.mark.parametrize("mode,alpha", [("accum_logp", 0.0), ("entropy", 0.0), ("hybrid", 2.0)])
def test_queue_sizes(W, B, mode, alpha):
    rng = np.random.default_rng(W * 1000 + B)
    compare_scored(np.stack([make_logp(rng, 64, 300, 2.0, peaked_p=0.9)]), [1], 64, W, B, mode, alpha)


@pytest.mark.parametrize("offset,spread", [(6e4, 1.0), (-6e4, 1.0), (3e7, 1e7), (0.0, 900.0)])
def test_logits_beyond_the_table_form(offset, spread):
    rng = np.random.default_rng(9)
    z = (rng.standard_normal((1, 3, 9000)) * spread + offset).astype(np.float32)
    z[0, 0, 8999] = np.float32(offset + 5 * spread)  # far above everything in an earlier slice
    z[0, 1, :4096] = -np.inf                         # a slice without a finite entry
    compare_logits(z, [2], 3, 6, 30, "accum_logp", 0.0)
    compare_logits(z, [2], 3, 6, 30, "hybrid", 0.5)


@pytest.mark.parametrize("V,W", [(9, 9), (1150, 9), (1350, 9), (4096, 32), (4097, 32), (12160, 5), (16384, 9), (16385, 10)])
def test_rows_of_few_groups(V, W):
    rng = np.random.default_rng(V + W)
    compare_logits(np.stack([make_draft_logits(rng, 4, V, 3.0) for _ in range(2)]), [7, 8], 4, W, 163, "hybrid", 0.5)
    compare_scored(np.stack([make_logp(rng, 1, V, 3.0, peaked_p=0.6)]), [7], 1, W, 20, "accum_logp", 0.0)
    compare_logits(np.zeros((1, 2, V), np.float32), [7], 2, W, 50, "accum_logp", 0.0)
