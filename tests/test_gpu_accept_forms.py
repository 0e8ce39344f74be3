"""Greedy acceptance on both sides of the limits of its one-launch form, for one sequence and for batches; and a large tree of
short rows is not left to the warps of one CTA."""
import numpy as np
import pytest
import torch

import jet_harness as H
import paper_2606_18394_b200 as jet
from jet_inputs import make_logp, make_target_logits, plant_path
from oracle import tree_accept_ref, tree_build_ref

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch,B,V,launches", [(1, 16, 1024, 1), (1, 16, 1025, 2), (1, 17, 64, 2), (1, 7, 2048, 1), (1, 7, 2049, 2), (19, 17, 100, 2),
                                                (20, 17, 100, 1), (20, 64, 512, 1), (20, 64, 513, 2), (20, 16, 2048, 1), (21, 15, 2049, 2),
                                                (1, 512, 64, 2), (20, 512, 64, 1)])
def test_both_forms(batch, B, V, launches):
    assert jet.jet_tree_accept_launches(batch, B, V) == launches
    rng = np.random.default_rng(batch * 7 + B * 1000 + V)
    N = 6
    trees = [tree_build_ref(make_logp(rng, N, V, 2.0), 0, N, 5, B) for _ in range(batch)]
    logits = np.stack([make_target_logits(rng, B, V, 2.0) for _ in range(batch)])
    logits[:, ::3] = np.round(logits[:, ::3])        # ties: the lowest token wins
    for b, t in enumerate(trees):
        plant_path(logits[b], t["token"], t["parent"], t["depth"], t["n_nodes"], 3, rng)
    stack = lambda k: np.stack([t[k] for t in trees])
    got = H.run_tree_accept(logits, stack("token"), stack("parent"), stack("depth"), stack("anc_mask"),
                            np.array([t["n_nodes"] for t in trees], np.int32), N)
    for b, t in enumerate(trees):
        ref = tree_accept_ref(logits[b], t["token"], t["parent"], t["depth"], t["n_nodes"], N)
        for k in ("tgt", "path", "out_tokens"):
            assert np.array_equal(got[k][b], ref[k]), (b, k)
        assert got["accept_len"][b] == ref["accept_len"]


def _time(B, V):
    N, i32 = 4, dict(dtype=torch.int32, device="cuda:0")
    logits = torch.randn((1, B, V), device="cuda:0")
    parent, depth, token = torch.zeros((1, B), **i32), torch.ones((1, B), **i32), torch.zeros((1, B), **i32)
    anc, n = torch.zeros((1, B, (B + 31) // 32), **i32), torch.full((1,), B, **i32)
    out = [torch.empty((1, B), **i32), torch.empty(1, **i32), torch.empty((1, N + 1), **i32), torch.empty((1, N + 1), **i32)]
    ws = torch.empty(max(256, jet.jet_tree_accept_workspace_bytes(1, B, V)), dtype=torch.uint8, device="cuda:0")

    def calls():
        for _ in range(10):
            jet.jet_tree_accept(logits, V, token, parent, depth, anc, n, 1, B, V, N, *out, ws)

    calls()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):                    # (issued call by call the host would be timed)
        calls()
    times = []
    for _ in range(12):
        start, end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        start.record()
        graph.replay()
        end.record()
        torch.cuda.synchronize()
        times.append(start.elapsed_time(end))
    return min(times)


def test_a_large_tree_of_short_rows():
    """512 rows of 64 logits: 12 times the time of 16 rows when one CTA took them in turns, twice now."""
    assert _time(512, 64) < 5 * _time(16, 64)
