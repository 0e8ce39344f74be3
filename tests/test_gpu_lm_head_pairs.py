"""LM-head arg-max on CTA pairs (more than 128 rows): row counts at the edges of 128 / 256 / 512-row groups, vocabularies at
the edges of the weight blocks, one K chunk and many.  Integer-valued operands make every logit exact in fp32 and ties
frequent, so the prediction must be the lowest token id among the largest logits, whichever block or CTA pair saw it."""
import numpy as np
import pytest

from jet_inputs import f32_to_bf16_bits
from test_gpu_lm_head import _run

pytestmark = pytest.mark.gpu


def _predictions(rows, d, V, rng, low, high):
    hidden = rng.integers(low, high + 1, (rows, d)).astype(np.float32)
    weight = rng.integers(low, high + 1, (V, d)).astype(np.float32)
    batch = -(-rows // 512)
    B = -(-rows // batch)
    hb = np.zeros((batch * B, d), np.float32)
    hb[:rows] = hidden
    tree = np.full((batch, B), -1, np.int32)          # a star of B nodes; the path selection is not what is tested here
    parent, depth, token = tree.copy(), np.ones_like(tree), np.zeros_like(tree)
    parent[:, 1:], depth[:, 0] = 0, 0
    words = (B + 31) // 32
    anc = np.zeros((batch, B, words), np.uint32)
    for v in range(B):
        anc[:, v, v // 32] |= np.uint32(1 << (v % 32))
        anc[:, v, 0] |= np.uint32(1)
    got = _run(f32_to_bf16_bits(hb), f32_to_bf16_bits(weight), token, parent, depth, anc, np.full(batch, B, np.int32), 4)
    return got["tgt"].reshape(-1)[:rows], hidden.astype(np.float64) @ weight.astype(np.float64).T


@pytest.mark.parametrize("rows", [128, 129, 255, 256, 257, 384, 511, 512, 513, 1024])
@pytest.mark.parametrize("d,V", [(64, 33000), (448, 3001)])
def test_row_groups(rows, d, V):
    got, logits = _predictions(rows, d, V, np.random.default_rng(rows + d), -1, 1)
    assert np.array_equal(got, logits.argmax(axis=1))


@pytest.mark.parametrize("V", [1, 15, 16, 95, 96, 97, 192, 193, 511, 513, 74 * 96, 74 * 96 + 1, 74 * 192 + 5, 50257])
@pytest.mark.parametrize("rows", [200, 300])
def test_vocabulary_edges(V, rows):
    got, logits = _predictions(rows, 128, V, np.random.default_rng(V), -2, 2)
    assert np.array_equal(got, logits.argmax(axis=1))
