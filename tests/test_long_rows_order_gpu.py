"""The pull sweep's residual is a fixed sum: the same bits for every upload of
one graph, with many rows long enough to be summed by a warp each, in one launch
for all sweeps and in launches of their own."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,ef", [(30011, 8), (400009, 24)])
def test_residual_bits_do_not_depend_on_the_upload(n, ef):
    import torch

    import paper_2010_16012_gb300 as gp

    rng = np.random.default_rng(3)
    hubs = rng.permutation(n)[:90]
    src = np.concatenate([rng.integers(0, n, ef * n)] + [rng.permutation(n)[:4700 + 40 * i] for i in range(90)])
    dst = np.concatenate([rng.integers(0, n, ef * n)] + [np.full(4700 + 40 * i, h) for i, h in enumerate(hubs)])
    key = np.unique(src.astype(np.int64) * n + dst)
    src, dst = key // n, key % n
    order = np.argsort(dst, kind="stable")
    dev = lambda a, dt: torch.from_numpy(np.ascontiguousarray(a)).to(dt).cuda()  # noqa: E731
    off = lambda x: dev(np.concatenate([[0], np.cumsum(np.bincount(x, minlength=n))]), torch.int64)  # noqa: E731
    arrays = off(src), dev(dst, torch.int32), off(dst), dev(src[order], torch.int32)
    x0 = dev(rng.random(n), torch.float32)
    seen = set()
    for _ in range(25):
        G = gp.Graph(n, *arrays)
        x, st = gp.pagerank(G, gp.PULL, iters=1, x0=x0)
        seen.add(st["residual"])
        G.free()
    assert len(seen) == 1, sorted(seen)
