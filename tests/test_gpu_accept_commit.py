"""Acceptance and commit as a step runs them (the path selected by the CTAs that copy) against the separate calls, bit for bit."""
import pytest
import torch

pytestmark = pytest.mark.gpu

RESULTS = ("tgt", "accept_len", "path", "out_tokens", "seq_len", "k_cache", "v_cache")


# batch, layers, B, N, W, V: one CTA per sequence and several; nodes at warp edges, the smallest and largest tree; rows of one key,
# of a few and of more than eight per thread; the one-launch acceptance with both commits
@pytest.mark.parametrize("batch,layers,B,N,W,V", [
    (1, 1, 1, 1, 1, 300), (1, 1, 16, 4, 4, 1000), (3, 2, 31, 4, 3, 8192), (2, 5, 33, 6, 3, 8193), (1, 36, 64, 8, 7, 151936),
    (5, 7, 255, 12, 6, 20001), (1, 4, 257, 16, 5, 151936), (2, 48, 512, 12, 10, 33000), (20, 1, 61, 5, 4, 512), (24, 9, 40, 64, 3, 512),
    (1, 3, 512, 9, 8, 600000),
])
@pytest.mark.parametrize("accept", ["greedy", "hidden", "sample"])
@pytest.mark.parametrize("paged,tail", [(0, 0), (1, 0), (0, 1), (1, 1)])
def test_step_form_equals_the_separate_calls(batch, layers, B, N, W, V, accept, paged, tail):
    from paper_2606_18394_b200.step import VerifyStep
    if accept == "sample" and B * V > 2e7 or accept != "greedy" and V > 2e5:
        pytest.skip("covered by the greedy form")
    dev, L, D = torch.device("cuda"), 77, 64
    gen = torch.Generator(device=dev).manual_seed(batch * 1000 + B)
    reserve = max(N + 1, B) if tail else N + 1
    kw = {}
    if paged:
        need = (L + reserve + 15) // 16
        kw = dict(page_size=16, num_pages=batch * need + 2, max_pages=need + 1)
    st = VerifyStep(batch=batch, layers=layers, Hq=2, Hkv=1, D=D, B=B, N=N, W=W, V=V, max_seq_len=L, device=dev, tail=bool(tail), **kw)
    st.seq_len0.copy_(torch.randint(L // 2, L + 1, (batch,), generator=gen, device=dev))
    st.seq_len.copy_(st.seq_len0)
    for t in (st.tree_k, st.tree_v, st.k_cache, st.v_cache):
        t.normal_(generator=gen)
    if paged:
        pages = torch.randperm(st.num_pages, generator=gen, device=dev)[:batch * need].to(torch.int32).view(batch, need)
        st.page_table.zero_()
        st.page_table[:, :need] = pages
    st.logp.copy_(torch.log_softmax(3.0 * torch.randn(st.logp.shape, generator=gen, device=dev), dim=-1))
    st.root_token.fill_(5)
    st.tree_build()
    st.accept_mode = accept
    if accept == "hidden":
        st.enable_lm_head(64)
        st.hidden.normal_(generator=gen)
        st.lm_head.normal_(generator=gen)
        rows = st.hidden.view(batch, B, -1)
    else:
        st.logits.normal_(generator=gen)
        st.u_accept.uniform_(generator=gen)
        st.u_sample.uniform_(generator=gen)
    parent, token, n = st.parent.tolist(), st.token.tolist(), st.n_nodes.tolist()
    for b in range(batch):                              # the target follows one path as far as it goes
        v = n[b] - 1 - b % max(n[b] // 2, 1)
        while v > 0:
            u = parent[b][v]
            if accept == "hidden":
                rows[b, u] = st.lm_head[token[b][v]] * 4.0
            else:
                st.logits[b, u, token[b][v]] = 60.0
            v = u
    before = {k: getattr(st, k).clone() for k in ("k_cache", "v_cache", "seq_len")}
    {"greedy": st.tree_accept, "hidden": st.tree_accept_hidden, "sample": st.tree_accept_sample}[accept]()
    st.kv_compact()
    want = {k: getattr(st, k).clone() for k in RESULTS}
    if n[0] > 1 and accept != "hidden":
        assert int(want["accept_len"].max()) > 0
    for _ in range(2):                                  # (the second time with the counts the first one left)
        for k, t in before.items():
            getattr(st, k).copy_(t)
        for k in ("tgt", "accept_len", "path", "out_tokens"):
            if accept != "sample" or k != "tgt":
                getattr(st, k).fill_(-7)
        st.run_back()
        for k in RESULTS:
            assert torch.equal(getattr(st, k), want[k]), k
        assert not st.arrived.any()
