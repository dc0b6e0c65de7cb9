"""Allocations that fail, each in turn: gp_graph_set_options and
gp_batch_set_options then leave the graph and the batch as they were (chunk
tables, work areas and options, and so the results),
and a hot set or the triangle counts' directed lists that found no memory are
built by the next call."""
import ctypes

import numpy as np
import pytest

import graphgen as gg

pytestmark = pytest.mark.gpu


CALLBACKS = []  # kept: what they allocated is released through them, whenever that is


@pytest.fixture()
def scarce():
    """gp, and a context in which the allocation of the given number fails."""
    import contextlib

    import torch

    import paper_2010_16012_gb300 as gp

    lib = gp.load()
    left = [-1]

    @gp.ALLOC_FN
    def alloc(nbytes, stream, ctx):
        left[0] -= 1
        return None if left[0] == -1 else torch.cuda.caching_allocator_alloc(nbytes)

    @gp.FREE_FN
    def free(p, nbytes, stream, ctx):
        torch.cuda.synchronize()
        torch.cuda.caching_allocator_delete(p)

    CALLBACKS.extend((alloc, free))

    @contextlib.contextmanager
    def failing(k):
        left[0] = k
        try:
            yield
        finally:
            left[0] = -1

    assert lib.gp_set_allocator(alloc, free, None) == gp.OK
    yield gp, failing
    assert lib.gp_set_allocator(gp.ALLOC_FN(), gp.FREE_FN(), ctypes.c_void_p()) == gp.OK


def results(gp, G, w):
    import torch

    x, _ = gp.pagerank(G, gp.PULL, iters=5)
    gw, gs, _ = gp.pagerank_backward(G, x, torch.ones_like(x), iters=5)
    level, parent, _ = gp.bfs(G, 1)
    dist, pred, _ = gp.sssp(G, 1, 0.5)
    fe, _ = gp.pagerank_fe(G, gp.PULL, eps=-1.0, iters=5)
    G.set_weights(*w)  # the sums of new weights use the chunk tables too
    y, _ = gp.pagerank(G, gp.PULL, iters=5)
    return [t.cpu().numpy() for t in (x, gw, gs, level, dist, pred, fe, y)]


def test_options_without_memory(scarce):
    import torch

    gp, failing = scarce
    g = gg.rmat(12, 16, seed=3, symmetrize=False)
    rng = np.random.default_rng(0)
    w = rng.uniform(0.1, 1.0, g.m).astype(np.float32)
    src = np.repeat(np.arange(g.n), np.diff(g.csr_off))
    order = np.lexsort((src, g.csr_idx))
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    G = gp.Graph(g.n, t(g.csr_off), t(g.csr_idx), t(g.csc_off), t(g.csc_idx), t(w), t(w[order]), normalize=True,
                 validate=True)
    both = t(w), t(w[order])
    want = results(gp, G, both)
    old, new = gp.options_dict(G.options()), dict(pull_light_max=8, push_light_max=4, chunk_edges=64)
    k = 0
    while True:
        try:
            with failing(k):
                G.set_options(**new)
            break
        except gp.GpError as e:
            assert e.status == gp.ERR_OOM
        assert gp.options_dict(G.options()) == old
        for a, b in zip(want, results(gp, G, both)):
            assert np.array_equal(a, b)
        k += 1
    assert k >= 10 and G.options().chunk_edges == 64
    for a, b in zip(want, results(gp, G, both)):  # the same but for the order of sums
        if a.dtype == np.int32:
            assert np.array_equal(a, b)
        else:
            assert np.allclose(a, b, rtol=1e-4, atol=1e-6 * np.abs(a[np.isfinite(a)]).max())
    G.free()


def test_hot_set_without_memory(scarce):
    gp, failing = scarce
    g = gg.rmat(12, 16, seed=3)
    graphs = [gp.Graph.from_graphgen(g) for _ in range(2)]
    for G in graphs:
        gp.pagerank(G, gp.PULL, iters=2)
    want, _ = gp.pagerank(graphs[0], gp.PUSH, iters=5)
    held = graphs[0].info()["device_bytes"]
    k = 0
    while True:
        try:
            with failing(k):
                gp.pagerank(graphs[1], gp.PUSH, iters=5)
            break
        except gp.GpError as e:
            assert e.status == gp.ERR_OOM
        k += 1
    assert k >= 8
    x, _ = gp.pagerank(graphs[1], gp.PUSH, iters=5)
    assert graphs[1].info()["device_bytes"] == held
    assert np.allclose(x.cpu().numpy(), want.cpu().numpy(), rtol=1e-5)
    for G in graphs:
        G.free()


def test_directed_lists_without_memory(scarce):
    gp, failing = scarce
    g = gg.rmat(12, 16, seed=3)
    G = gp.Graph.from_graphgen(g)
    want, total, _ = gp.triangles(G)
    held = G.info()["device_bytes"]
    k, last = 0, None
    while last != held:  # (the first call in which nothing fails leaves the lists)
        H = gp.Graph.from_graphgen(g)
        try:
            with failing(k):
                tc, t, _ = gp.triangles(H)
            assert t == total and (tc == want).all()
        except gp.GpError as e:
            assert e.status == gp.ERR_OOM
        last = H.info()["device_bytes"]
        tc, t, _ = gp.triangles(H)  # with memory again
        assert t == total and (tc == want).all() and H.info()["device_bytes"] == held
        H.free()
        k += 1
    assert k > 3  # the offsets, the lists and a temporary list, each without memory once
    G.free()


def test_batch_options_without_memory(scarce):
    gp, failing = scarce
    graphs = [gp.Graph.from_graphgen(gg.rmat(s, 16, seed=s)) for s in (10, 11)]
    B = gp.Batch(graphs, k_ppr=32)
    rng = np.random.default_rng(2)
    seeds, sources = rng.integers(0, 1024, (2, 32)), rng.integers(0, 1024, (2, 9))

    def results():
        outs, done, _ = B.ppr(seeds, iters=40, tol=1e-6)
        return [t.cpu().numpy() for t in outs] + [done] + [t.cpu().numpy() for t in B.msbfs(sources)[0]]

    want, old, k = results(), B.options(), 0
    while True:
        try:
            with failing(k):
                B.set_options(big_in_degree=8, chunk_edges=64, l2_budget_mb=1)
            break
        except gp.GpError as e:
            assert e.status == gp.ERR_OOM
        assert B.options() == old
        for a, b in zip(want, results()):
            assert np.array_equal(a, b)
        k += 1
    assert k > 4  # the five lists
    for a, b in zip(want, results()):  # the same but for the order of sums
        assert np.array_equal(a, b) if a.shape[1] == 64 else np.allclose(a, b, rtol=1e-4, atol=1e-6)
    B.free()
    for G in graphs:
        G.free()
