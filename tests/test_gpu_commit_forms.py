"""Commit of the accepted path at the edges of its forms: one CTA per sequence up to 64 rows and a second launch beyond, more
sequences than CTAs, rows of one to 33 16-byte columns, the in-place form's sixteen rows in flight; byte-exact against the
oracle.  And a long path of one sequence is not left to a few SMs."""
import numpy as np
import pytest
import torch

import jet_harness as H
import paper_2606_18394_b200 as jet
from oracle import kv_compact_ref, kv_compact_tail_ref
from test_gpu_kv_compact import _rand_bits, _random_paths

pytestmark = pytest.mark.gpu

SHAPES = [(1, 3, 64, 8, 128, 31), (1, 3, 64, 8, 128, 32), (36, 1, 64, 8, 128, 8), (3, 2, 512, 4, 64, 64), (5, 40, 16, 1, 8, 8),
          (7, 3, 40, 3, 88, 10), (40, 150, 6, 1, 8, 4), (40, 300, 6, 1, 8, 4), (40, 450, 6, 1, 8, 4), (2, 5, 80, 2, 64, 17)]


def _table(rng, batch, need, page):
    pages = rng.permutation(sum(need) + 2)
    table = np.zeros((batch, max(need)), np.int32)
    at = 0
    for b, n in enumerate(need):
        table[b, :n] = pages[at:at + n]
        at += n
    return table, len(pages)


def _case(shape, paged, room):
    layers, batch, B, Hkv, D, N = shape
    rng = np.random.default_rng(layers * 1000 + batch * 10 + N)
    accept = rng.integers(0, min(N, B - 1) + 1, size=batch)
    accept[0] = min(N, B - 1)
    accept[-1] = min(16, N, B - 1) if batch > 1 else accept[0]
    path = _random_paths(rng, batch, B, N, accept)
    seq = rng.integers(0, 21, size=batch).astype(np.int32)
    table, pages = _table(rng, batch, [(int(n) + room + 15) // 16 for n in seq], 16) if paged else (None, 0)
    dims = (layers, pages, 16, Hkv, D) if paged else (layers, batch, 21 + room, Hkv, D)
    return rng, accept, path, seq, table, _rand_bits(rng, dims), _rand_bits(rng, dims)


@pytest.mark.parametrize("paged", [False, True])
@pytest.mark.parametrize("shape", SHAPES)
def test_copy(shape, paged):
    layers, batch, B, Hkv, D, N = shape
    rng, accept, path, seq, table, kc, vc = _case(shape, paged, N + 1)
    tk, tv = _rand_bits(rng, (layers, batch, B, Hkv, D)), _rand_bits(rng, (layers, batch, B, Hkv, D))
    rk, rv, rs = kv_compact_ref(tk, tv, kc, vc, table, path, accept, seq)
    gk, gv, gs = H.run_kv_compact(tk, tv, kc, vc, table, path, accept, seq, N)
    assert np.array_equal(gs, rs)
    assert np.array_equal(gk, rk) and np.array_equal(gv, rv)


@pytest.mark.parametrize("paged", [False, True])
@pytest.mark.parametrize("shape", SHAPES)
def test_in_place(shape, paged):
    rng, accept, path, seq, table, kc, vc = _case(shape, paged, max(shape[2], shape[5] + 1))
    rk, rv, rs = kv_compact_tail_ref(kc, vc, table, path, accept, seq)
    gk, gv, gs = H.run_kv_compact_tail(kc, vc, table, path, accept, seq, shape[2])
    assert np.array_equal(gs, rs)
    assert np.array_equal(gk.reshape(kc.shape), rk) and np.array_equal(gv.reshape(vc.shape), rv)


@pytest.mark.parametrize("layers,batch,D", [(2, 1, 64), (9, 1, 64), (6, 40, 64), (3, 150, 8)])
def test_commits_in_a_row(layers, batch, D):
    """Each commit takes the length that the one before it left, with no kernel between them: a copy that saw a length too early
    or too late, or a commit that began before the last one's copies ended, leaves other rows."""
    B, N, commits, dev = 16, 8, 24, "cuda:0"
    rng = np.random.default_rng(layers + batch)
    paths, accepts = [], []
    for _ in range(commits):
        accepts.append(rng.integers(0, N + 1, size=batch))
        paths.append(_random_paths(rng, batch, B, N, accepts[-1]))
    rows = commits * (N + 1)
    tk, tv = _rand_bits(rng, (layers, batch, B, 1, D)), _rand_bits(rng, (layers, batch, B, 1, D))
    rk, rv = _rand_bits(rng, (layers, batch, rows, 1, D)), _rand_bits(rng, (layers, batch, rows, 1, D))
    rs = np.zeros(batch, np.int32)
    on_gpu = lambda x: torch.from_numpy(np.ascontiguousarray(x).view(np.int16)).to(dev)
    gtk, gtv, gk, gv = on_gpu(tk), on_gpu(tv), on_gpu(rk), on_gpu(rv)
    seq = torch.zeros(batch, dtype=torch.int32, device=dev)
    gp = [torch.from_numpy(np.asarray(p, np.int32)).to(dev) for p in paths]
    ga = [torch.from_numpy(np.asarray(a, np.int32)).to(dev) for a in accepts]
    torch.cuda.synchronize()

    def run():
        for p, a in zip(gp, ga):
            jet.jet_kv_compact(gtk, gtv, gk, gv, gk.stride(0), gk.stride(1), None, 0, 0, p, a, seq, layers, batch, B, 1, D, N)

    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        run()
    graph.replay()
    for p, a in zip(paths, accepts):
        rk, rv, rs = kv_compact_ref(tk, tv, rk, rv, None, p, a, rs)
    assert np.array_equal(seq.cpu().numpy(), rs)
    for got, want in ((gk, rk), (gv, rv)):
        assert np.array_equal(got.cpu().numpy(), np.ascontiguousarray(want).view(np.int16))
    with_graph = gk.clone(), gv.clone()
    gk.zero_(), gv.zero_(), seq.zero_()
    run()                                            # and issued one by one
    assert np.array_equal(seq.cpu().numpy(), rs)
    for b in range(batch):
        n = int(rs[b])
        assert torch.equal(gk[:, b, :n], with_graph[0][:, b, :n]) and torch.equal(gv[:, b, :n], with_graph[1][:, b, :n])


def _time(layers, N, a):
    B, Hkv, D, dev = 256, 8, 128, "cuda:0"
    i32 = dict(dtype=torch.int32, device=dev)
    tree = torch.zeros((2, layers, 1, B, Hkv, D), dtype=torch.bfloat16, device=dev)
    cache = torch.zeros((2, layers, 1, 600, Hkv, D), dtype=torch.bfloat16, device=dev)
    path, accept, seq = torch.full((1, N + 1), -1, **i32), torch.full((1,), a, **i32), torch.zeros(1, **i32)
    path[0, :a + 1] = torch.arange(a + 1, **i32)
    start_len = torch.zeros_like(seq)

    def commits():
        for _ in range(10):
            seq.copy_(start_len)
            jet.jet_kv_compact(tree[0], tree[1], cache[0], cache[1], cache[0].stride(0), 600 * Hkv * D, None, 0, 0, path, accept, seq,
                               layers, 1, B, Hkv, D, N)

    commits()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):                    # (issued call by call the host would be timed)
        commits()
    times = []
    for _ in range(12):
        start, end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        start.record()
        graph.replay()
        end.record()
        torch.cuda.synchronize()
        times.append(start.elapsed_time(end))
    return min(times)


def test_a_long_path_uses_the_whole_gpu():
    """19 MB moved: 8 times the time of a single row's commit while a cluster of eight CTAs did it, twice now."""
    assert _time(36, 64, 64) < 4 * _time(1, 64, 0)
