"""Small problems take forms of their own -- tree construction and acceptance in one launch each: both sides of the limits
of these forms, rows that end inside a 16-byte load, one to many rows per warp; and the step entry that restarts seq_len."""
import numpy as np
import pytest

from jet_inputs import make_logp, make_target_logits, plant_path
from oracle import tree_accept_ref, tree_build_ref

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,V", [(1, 1), (6, 4096), (6, 4097), (3, 8192), (3, 8191), (2, 12288), (1, 24576), (1, 24577), (5, 129)])
def test_tree_construction(N, V):
    import jet_harness as H
    rng = np.random.default_rng(N * 100003 + V)
    batch, W, B = 3, 7, 40
    logp = np.stack([make_logp(rng, N, V, 2.0, peaked_p=0.6 if V > 1 else None) for _ in range(batch)])
    logp[1] = np.float32(-3.0)                                   # all equal: token order decides
    got = H.run_tree_build(logp, [5, 6, 7], N, W, B)
    for b in range(batch):
        ref = tree_build_ref(logp[b], 5 + b, N, W, B)
        for k in ("parent", "depth", "token", "anc_mask"):
            assert np.array_equal(got[k][b], ref[k]), (b, k)
        assert np.array_equal(got["score"][b].view(np.uint32), ref["score"].view(np.uint32))


@pytest.mark.parametrize("B,V", [(1, 1), (8, 4096), (9, 4096), (8, 4097), (16, 2048), (17, 1927), (512, 64), (511, 63), (40, 3)])
def test_acceptance(B, V):
    import jet_harness as H
    rng = np.random.default_rng(B * 100003 + V)
    batch, N = 2, 6
    trees = [tree_build_ref(make_logp(rng, N, V, 2.0), 0, N, 5, B) for _ in range(batch)]
    logits = np.stack([make_target_logits(rng, B, V, 2.0) for _ in range(batch)])
    logits[:, ::3] = np.round(logits[:, ::3])                    # ties: the lowest token wins
    for b, t in enumerate(trees):
        if V > 8:
            plant_path(logits[b], t["token"], t["parent"], t["depth"], t["n_nodes"], 3, rng)
    stack = lambda k: np.stack([t[k] for t in trees])
    got = H.run_tree_accept(logits, stack("token"), stack("parent"), stack("depth"), stack("anc_mask"),
                            np.array([t["n_nodes"] for t in trees], np.int32), N)
    for b, t in enumerate(trees):
        ref = tree_accept_ref(logits[b], t["token"], t["parent"], t["depth"], t["n_nodes"], N)
        for k in ("tgt", "path", "out_tokens"):
            assert np.array_equal(got[k][b], ref[k]), (b, k)
        assert got["accept_len"][b] == ref["accept_len"]


@pytest.mark.parametrize("V,score_mode,raw", [(500, "accum_logp", False), (9000, "accum_logp", False), (9000, "hybrid", False),
                                              (9000, "accum_logp", True), (9000, "entropy", True)])
def test_a_step_restarts_the_lengths(V, score_mode, raw):
    import torch
    from paper_2606_18394_b200.step import VerifyStep
    st = VerifyStep(batch=3, layers=1, Hq=4, Hkv=2, D=64, B=12, N=4, W=3, V=V, max_seq_len=40)
    st.score_mode, st.draft_logits = score_mode, raw
    st.seq_len0.copy_(torch.tensor([40, 1, 17], dtype=torch.int32))
    st.logp.copy_(torch.log_softmax(torch.randn_like(st.logp), dim=-1))
    for _ in range(2):
        st.seq_len.fill_(-5)
        st.run_front()
        torch.cuda.synchronize()
        assert torch.equal(st.seq_len, st.seq_len0) and int(st.status.item()) == 0
    st.run_back()
    torch.cuda.synchronize()
    assert torch.equal(st.seq_len, st.seq_len0 + st.accept_len + 1)
