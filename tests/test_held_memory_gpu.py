"""gp_graph_info's device_bytes is the library-owned device memory that the handle
holds: it follows every entry point's workspaces as the library's pool does.
Bound: the pool counts whole allocations, each at most 512 bytes more than asked
for, and at most 300 of them."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_every_workspace_is_counted():
    import torch

    import paper_2010_16012_gb300 as gp

    rng = np.random.default_rng(1)
    n = 60013
    a, b = rng.integers(0, n, 12 * n), rng.integers(0, n, 12 * n)
    a, b = np.concatenate([a, np.zeros(3000, dtype=np.int64)]), np.concatenate([b, np.arange(1, 3001)])
    key = np.unique(np.concatenate([a * n + b, b * n + a])[np.concatenate([a != b, a != b])])
    src, dst = key // n, key % n
    off = torch.from_numpy(np.concatenate([[0], np.cumsum(np.bincount(src, minlength=n))])).cuda()
    idx = torch.from_numpy(dst).int().cuda()
    used = lambda: (torch.cuda.synchronize(), gp.pool_usage()[1])[1]  # noqa: E731
    before = used()
    G = gp.Graph(n, off, idx, symmetric=True)
    x, _ = gp.pagerank(G, gp.PULL, iters=3)
    calls = [lambda: gp.pagerank(G, gp.PUSH, iters=3), lambda: gp.bfs(G, 0), lambda: gp.bfs_multi(G, [0, 1, 2]),
             lambda: gp.sssp(G, 0, 2.0), lambda: gp.pagerank_fe(G, iters=5), lambda: gp.triangles(G),
             lambda: gp.bc(G, np.arange(16, dtype=np.int32)),
             lambda: gp.pagerank_backward(G, x, torch.ones_like(x), iters=3, want_weights=False)]
    for i, call in enumerate([lambda: None] + calls):
        call()
        held = G.info()["device_bytes"]
        assert abs(used() - before - held) <= 300 * 512, (i, held, used() - before)
    G.free()
    assert abs(used() - before) <= 300 * 512
