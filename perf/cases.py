"""Performance cases of the tree-verification path: what a serving program has it do, over the range it is used in.

A case is one call pattern of the public entry points:

  step    one verification step through ``VerifyStep.run()`` -- tree construction, attention of every layer, acceptance,
          commit -- issued call by call, or (``graph``) replayed from a CUDA graph captured once, as ``bench.py`` does
  attn    the attention calls of a layer stack alone (the draft head's block-causal attention: a chain of rows)
  build   one tree-construction call, as an engine issues it right behind its draft head's forward
  accept  one acceptance call, as an engine issues it behind the target's forward

Sizes are those of the repository's workload table (``jet_inputs.CONFIGS``) and of its tests; inputs are synthetic and
seeded: q / k / v ~ N(0,1) in bf16, draft rows with one confident token per depth (p = 0.7 over N(0, 3) logits), target
logits N(0, 2) whose arg-max follows one random path of the tree.
"""
import math

import torch

import paper_2606_18394_b200 as jet
from paper_2606_18394_b200.step import VerifyStep

QWEN3_8B = dict(Hq=32, Hkv=8, D=128)          # layer shapes of the workload table
MOE_30B = dict(Hq=32, Hkv=4, D=128)
VOCAB = 151936
SCORE_MODES = {"accum_logp": 0, "entropy": 1, "hybrid": 2}


def _step(**kw):
    c = dict(kind="step", batch=1, layers=36, **QWEN3_8B, L=4096, L_min=0, paged=0, tail=0, B=64, N=8, W=7, V=VOCAB,
             draft="logp", score="accum_logp", accept="greedy", d_model=0, plant=5, graph=0)
    c.update(kw)
    c["L_min"] = c["L_min"] or c["L"]
    return c


def listed():
    return [
        # the smallest step there is: one small layer, a 16-node tree; launches and host work are all it costs
        _step(name="tiny_step", layers=1, Hq=8, Hkv=2, D=64, L=512, B=16, N=4, W=4, V=1024, plant=3),
        # the benchmark's own step, captured once and replayed: latency-bound attention launches back to back
        _step(name="qwen3_8b_step_graph", graph=1),
        # an odd-sized step at temperature > 0 issued call by call: tree rows in the cache tail, in-place commit
        _step(name="odd_sample_tail_step", L=2937, B=61, accept="sample", tail=1, plant=4),
        # long generation with the largest budget the paper uses, issued call by call
        _step(name="sweep_16k_b256_step", L=16384, B=256, N=12, plant=8),
        # batched serving: 32 ragged sequences in a paged cache, raw draft logits, a quarter of the layer stack
        _step(name="batched_paged_step", batch=32, layers=8, L=8192, L_min=1024, paged=1, draft="logits"),
        # the largest step: 48 layers, prefix 32768, 512 nodes
        _step(name="moe_b512_step", layers=48, **MOE_30B, L=32768, B=512, N=12, plant=8),
        # eight long sequences at once, acceptance straight from the hidden states (1024 rows through the LM head)
        _step(name="moe_batch8_hidden_step", batch=8, layers=6, **MOE_30B, L=32768, L_min=24001, B=128, N=12, plant=6,
              accept="hidden", d_model=2048, graph=1),
        # the draft head's own attention: a block of 16 chained rows behind a short context, five layers
        dict(name="draft_head_attn", kind="attn", batch=1, layers=5, **QWEN3_8B, L=1000, L_min=1000, B=16),
        # one sequence's tree from raw draft logits, large budget: what stands between draft and target forward
        dict(name="build_logits_b256", kind="build", batch=1, N=16, V=VOCAB, W=7, B=256, draft="logits", score="accum_logp"),
        # hybrid expansion score for a serving batch
        dict(name="build_hybrid_batch32", kind="build", batch=32, N=8, V=VOCAB, W=7, B=64, draft="logp", score="hybrid"),
        # greedy acceptance from hidden states for a small batch: 256 rows through the LM head
        dict(name="accept_hidden_256", kind="accept", batch=4, B=64, N=8, W=7, V=VOCAB, accept="hidden", d_model=4096, plant=5),
        # non-greedy acceptance for a serving batch: 2048 rows of fp32 logits
        dict(name="accept_sample_batch32", kind="accept", batch=32, B=64, N=8, W=7, V=VOCAB, accept="sample", d_model=0, plant=5),
    ]


# ------------------------------------------------------------------------------------------------ what a pass must do
def _lens(c):
    """Prefix lengths: evenly spread over [L_min, L], the longest exactly L (prepare shuffles them)."""
    n = c["batch"]
    return [c["L"] - (c["L"] - c["L_min"]) * i // max(n - 1, 1) for i in range(n)]


def _nodes(c):
    """Nodes a tree of this shape ends up with (the budget, unless W and N cannot fill it)."""
    if c["kind"] == "attn":
        return c["B"]
    total, level = 1, 1
    for _ in range(c["N"]):
        level *= c["W"]
        total += level
        if total >= c["B"]:
            return c["B"]
    return total


def work(case):
    c, nbytes, flops = case, 0.0, 0.0
    n, batch = _nodes(c), c["batch"]
    if c["kind"] in ("step", "attn"):
        Hq, Hkv, D = c["Hq"], c["Hkv"], c["D"]
        for L in _lens(c):
            kv_rows = 2 * (L + n) * Hkv * D * 2                         # K and V: prefix and the tree's own rows
            nbytes += c["layers"] * (kv_rows + 2 * n * Hq * D * 2)      # q in, out out
            flops += c["layers"] * 4.0 * n * Hq * D * (L + 1)
    if c["kind"] in ("step", "build"):
        nbytes += batch * c["N"] * c["V"] * 4 + batch * c["B"] * (16 + 4 * ((c["B"] + 31) // 32))
    if c["kind"] in ("step", "accept"):
        if c["accept"] == "hidden":
            nbytes += c["V"] * c["d_model"] * 2 + batch * n * c["d_model"] * 2
            flops += 2.0 * batch * n * c["d_model"] * c["V"]
        else:
            nbytes += batch * n * c["V"] * 4
    if c["kind"] == "step":                                             # rows of the accepted path, read and written
        nbytes += batch * c["layers"] * (min(c["plant"], c["N"]) + 1) * 2 * 2 * c["Hkv"] * c["D"] * 2
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    """bf16 attention outputs: 1e-2; fp32 scores and log-sum-exps: 1e-5; trees, tokens and lengths: the same.  The LM
    head's fp32 sums may be formed in any order, so the arg-max of a row may differ where its two best logits tie."""
    k, acc = case["kind"], case.get("accept")
    if k in ("step", "attn"):
        return {"rel": 1e-2, "differ": 0.005} if acc == "hidden" else {"rel": 1e-2}
    if k == "build":
        return {"rel": 1e-5}
    if acc == "hidden":
        return {"rel": 0.0, "differ": 0.005}
    return {"rel": 1e-4} if acc == "sample" else "exact"


# ------------------------------------------------------------------------------------------------ more of the same
def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _cost(c):
    w = work(c)
    return w["bytes"] / 4e12 + w["flops"] / 8e14


def draw(rng):
    ceiling = max(_cost(c) for c in listed())
    while True:
        kind = rng.choice(["step"] * 6 + ["attn", "build", "build", "accept"])
        V = VOCAB if rng.random() < 0.6 else _log_int(rng, 1024, VOCAB)
        N, W = rng.randint(4, 16), rng.randint(3, 10)
        B, batch = _log_int(rng, 8, 512), _log_int(rng, 1, 32)
        heads = rng.choice([QWEN3_8B] * 3 + [MOE_30B] * 2 + [dict(Hq=8, Hkv=2, D=64), dict(Hq=16, Hkv=4, D=64)])
        L = _log_int(rng, 64, 32768)
        L_min = L if batch == 1 else max(1, int(L * rng.uniform(0.2, 1.0)))
        accept = rng.choice(["greedy"] * 3 + ["hidden", "sample"])
        d_model = rng.choice([1024, 2048, 2560, 4096]) if accept == "hidden" else 0
        if kind == "build":
            c = dict(kind=kind, batch=batch, N=N, V=V, W=W, B=B, draft=rng.choice(["logp", "logits"]),
                     score=rng.choice(["accum_logp", "accum_logp", "entropy", "hybrid"]))
        elif kind == "accept":
            c = dict(kind=kind, batch=batch, B=B, N=N, W=W, V=V, accept=accept, d_model=d_model, plant=rng.randint(1, N))
        elif kind == "attn":
            c = dict(kind=kind, batch=batch, layers=rng.randint(1, 6), **heads, L=min(L, 8192), L_min=min(L_min, 8192),
                     B=rng.randint(4, 32))
        else:
            c = _step(batch=batch, layers=_log_int(rng, 1, 48), **heads, L=L, L_min=L_min, paged=rng.randint(0, 1),
                      tail=int(rng.random() < 0.3), B=B, N=N, W=W, V=V,
                      draft="logp" if accept == "sample" else rng.choice(["logp", "logits"]),
                      score=rng.choice(["accum_logp"] * 3 + ["entropy", "hybrid"]), accept=accept, d_model=d_model,
                      plant=rng.randint(1, N), graph=rng.randint(0, 1))
        kv = c.get("layers", 0) * sum(_lens(c)) * 4 * c["Hkv"] * c["D"] if "L" in c else 0
        rows = 0 if kind in ("attn", "build") else batch * B * V * 4
        if kv <= 5e9 and rows <= 1.4e9 and batch * B <= 8192 and _cost(c) <= ceiling:
            return c


# ------------------------------------------------------------------------------------------------ inputs and handles
def _draft_rows(gen, batch, N, V, raw, dev):
    """[batch, N, V] fp32: N(0, 3) logits with one token per depth raised to p = 0.7, as they are or log-softmaxed."""
    out = torch.empty((batch, N, V), dtype=torch.float32, device=dev)
    at = torch.arange(N, device=dev)
    for b in range(batch):
        z = torch.randn((N, V), generator=gen, device=dev).double() * 3.0
        top = torch.randint(0, V, (N,), generator=gen, device=dev)
        z[at, top] = -math.inf
        z[at, top] = math.log(0.7 / 0.3) + torch.logsumexp(z, dim=1)
        out[b] = (z if raw else torch.log_softmax(z, dim=1)).float()
    return out


def _planted(gen, token, parent, depth, n_nodes, length, V):
    """One random root path per sequence: lists of (sequence, node, token its target row must prefer)."""
    token, parent, depth, n_nodes = (t.cpu().tolist() for t in (token, parent, depth, n_nodes))
    pick = torch.rand((len(token), 2), generator=gen, device=gen.device).cpu().tolist()
    seqs, nodes, toks = [], [], []
    for b, (u, w) in enumerate(pick):
        n = n_nodes[b]
        eff = min(length, max(depth[b][:n]))
        cands = [v for v in range(n) if depth[b][v] == eff]
        end = cands[int(u * len(cands))]
        taken = {token[b][v] for v in range(n) if parent[b][v] == end}
        t = int(w * V)
        while t in taken:
            t = (t + 1) % V
        v = end
        while v >= 0:
            seqs.append(b)
            nodes.append(v)
            toks.append(t)
            t, v = token[b][v], parent[b][v]
    return seqs, nodes, toks


def _fill_target(gen, st, c):
    """Target side of the step: logits (or hidden states and LM head) whose preference follows one path of the tree."""
    dev = st.device
    seqs, nodes, toks = (torch.tensor(x, device=dev) for x in
                         _planted(gen, st.token, st.parent, st.depth, st.n_nodes, c["plant"], c["V"]))
    if c["accept"] == "hidden":
        st.enable_lm_head(c["d_model"])
        st.hidden.normal_(generator=gen)
        st.lm_head.normal_(0.0, 0.02, generator=gen)
        w = st.lm_head[toks].float()
        st.hidden[seqs * c["B"] + nodes] = (8.0 * w / w.norm(dim=1, keepdim=True)).bfloat16()
    else:
        st.logits.normal_(0.0, 2.0, generator=gen)
        lead = 8.0 if c["accept"] == "sample" else 1.0        # a confident target: its token carries nearly all the mass
        st.logits[seqs, nodes, toks] = st.logits[seqs, nodes].amax(dim=1) + lead
    if c["accept"] == "sample":
        st.u_accept.uniform_(generator=gen)
        st.u_sample.uniform_(generator=gen)
    st.accept_mode = c["accept"]


def _step_buffers(c, dev):
    """The step object of a case (for an accept case: its tree and target side, with no cache to speak of)."""
    lens = _lens(c) if "L" in c else [1] * c["batch"]
    kw = dict(batch=c["batch"], layers=c.get("layers", 1), Hq=c.get("Hq", 8), Hkv=c.get("Hkv", 2), D=c.get("D", 64), B=c["B"],
              N=c.get("N", 1), W=c.get("W", 1), V=c.get("V", 1), max_seq_len=max(lens), device=dev, tail=bool(c.get("tail")))
    if c.get("paged"):
        reserve = max(c["N"] + 1, c["B"]) if c["tail"] else c["N"] + 1
        need = [(n + reserve + 15) // 16 for n in lens]
        # (a caller's table has room for every position the bound on the lengths allows)
        kw.update(page_size=16, num_pages=sum(need) + 3, max_pages=(max(lens) + max(reserve, c["B"]) + 15) // 16)
    return VerifyStep(**kw), lens


def _graph(fn):
    fn()                                         # first call of the shapes: outside the capture
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        fn()
    return g


def prepare(case, seed):
    c, dev = case, torch.device("cuda", torch.cuda.current_device())
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed)
    if c["kind"] == "build":
        return _prepare_build(c, gen, dev)
    st, lens = _step_buffers(c, dev)
    state = {"case": c, "st": st, "graph": None}
    if "L" in c:
        order = torch.randperm(len(lens), generator=gen, device=dev)
        st.seq_len0.copy_(torch.tensor(lens, dtype=torch.int32, device=dev)[order])
        st.seq_len.copy_(st.seq_len0)
        for t in (st.q, st.tree_k, st.tree_v, st.k_cache, st.v_cache):
            t.normal_(generator=gen)
        if st.paged:          # pages dealt out in random order; entries behind a sequence's own pages are never used
            pages = torch.randperm(st.num_pages, generator=gen, device=dev).to(torch.int32)
            reserve = max(c["N"] + 1, c["B"]) if c["tail"] else c["N"] + 1
            need = (st.seq_len0 + reserve + 15) // 16
            first = torch.cumsum(need, 0) - need
            slot = first[:, None] + torch.arange(st.max_pages, device=dev)[None, :]
            st.page_table.copy_(pages[slot.clamp(max=st.num_pages - 1)])
        if st.tail:
            st.place_tree()
    if c["kind"] == "attn":   # a chain: node v sees nodes 0 .. v
        v = torch.arange(c["B"], dtype=torch.int64, device=dev)
        st.anc_mask.copy_(((2 << v) - 1).to(torch.int32)[None, :, None].expand_as(st.anc_mask))
        st.n_nodes.fill_(c["B"])
        return state
    st.draft_logits = c.get("draft") == "logits"
    st.score_mode, st.score_alpha = c.get("score", "accum_logp"), 0.5
    st.logp.copy_(_draft_rows(gen, c["batch"], c["N"], c["V"], st.draft_logits, dev))
    st.root_token.copy_(torch.randint(0, c["V"], (c["batch"],), generator=gen, device=dev))
    st.tree_build()
    _fill_target(gen, st, c)
    if c.get("graph"):
        state["graph"] = _graph(st.run)
    return state


def _prepare_build(c, gen, dev):
    batch, N, V, W, B = (c[k] for k in ("batch", "N", "V", "W", "B"))
    raw = c["draft"] == "logits"
    i32 = dict(dtype=torch.int32, device=dev)
    f32 = dict(dtype=torch.float32, device=dev)
    scored = c["score"] != "accum_logp"
    need = (jet.jet_tree_build_logits_workspace_bytes if raw else jet.jet_tree_build_scored_workspace_bytes if scored
            else jet.jet_tree_build_workspace_bytes)(batch, N, V, W)
    out = dict(parent=torch.empty((batch, B), **i32), depth=torch.empty((batch, B), **i32),
               token=torch.empty((batch, B), **i32), score=torch.empty((batch, B), **f32),
               anc_mask=torch.empty((batch, B, (B + 31) // 32), **i32), n_nodes=torch.empty(batch, **i32))
    if scored:
        out["depth_entropy"] = torch.empty((batch, N), **f32)
    if raw:
        out["depth_lse"] = torch.empty((batch, N), **f32)
    return {"case": c, "rows": _draft_rows(gen, batch, N, V, raw, dev),
            "root": torch.randint(0, V, (batch,), generator=gen, device=dev).to(torch.int32),
            "ws": torch.empty(max(need, 256), dtype=torch.uint8, device=dev), "out": out}


# ------------------------------------------------------------------------------------------------ one pass
def run(state):
    c = state["case"]
    if c["kind"] == "build":
        return _run_build(c, state)
    st = state["st"]
    if c["kind"] == "attn":
        for layer in range(st.layers):
            st.verify_attn(layer)
        return {"out": st.out}
    if c["kind"] == "accept":
        if c["accept"] == "hidden":
            st.tree_accept_hidden()
        elif c["accept"] == "sample":
            st.tree_accept_sample()
        else:
            st.tree_accept()
    elif state["graph"] is not None:
        state["graph"].replay()
    else:
        st.run()
    r = dict(accept_len=st.accept_len, path=st.path, out_tokens=st.out_tokens)
    r["alpha" if c["accept"] == "sample" else "tgt"] = st.alpha if c["accept"] == "sample" else st.tgt
    if c["kind"] == "step":
        r.update(parent=st.parent, depth=st.depth, token=st.token, score=st.score, anc_mask=st.anc_mask, n_nodes=st.n_nodes,
                 out=st.out, seq_len=st.seq_len, k_cache=st.k_cache, v_cache=st.v_cache)
        if c["draft"] == "logits":
            r["depth_lse"] = st.depth_lse
        if c["score"] != "accum_logp":
            r["depth_entropy"] = st.depth_entropy
    return r


def _run_build(c, s):
    o, dims = s["out"], tuple(c[k] for k in ("batch", "N", "V", "W", "B"))
    tree = (o["parent"], o["depth"], o["token"], o["score"], o["anc_mask"], o["n_nodes"])
    if c["draft"] == "logits":
        jet.jet_tree_build_logits(s["rows"], s["root"], *dims, SCORE_MODES[c["score"]], 0.5, *tree, o.get("depth_entropy"),
                                  o["depth_lse"], s["ws"])
    elif c["score"] == "accum_logp":
        jet.jet_tree_build(s["rows"], s["root"], *dims, *tree, s["ws"])
    else:
        jet.jet_tree_build_scored(s["rows"], s["root"], *dims, SCORE_MODES[c["score"]], 0.5, *tree, o["depth_entropy"], s["ws"])
    return o
