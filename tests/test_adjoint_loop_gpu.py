"""The adjoint's pull sweeps where rows change hands: degrees at the light limit,
at a chunk's end and over more than 16 chunks (added by a warp), on a graph
whose sweeps run in one launch and on one that takes a launch per step; stopped
by count and by tolerance.  Against the same sweeps in FP64.  Bound on lambda: a
row's FP32 sum of k products of size at most max|lambda| * P errs by at most
(k + 4) * 2^-24 of sum(P) * max|lambda| <= max|lambda| a sweep, carried on by
the factor d: divided by 1 - d."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gp():
    import torch

    import paper_2010_16012_gb300 as gp

    assert torch.cuda.is_available()
    gp.load()
    return gp


@pytest.mark.parametrize("bulk", [0, 9_000_000])
@pytest.mark.parametrize("weighted", [False, True])
@pytest.mark.parametrize("light,chunk", [(32, 256), (0, 32)])
def test_rows(gp, light, chunk, weighted, bulk):
    import torch

    rng = np.random.default_rng(7)
    deg = [0, 1, 31, 32, 33, 255, 256, 257, 16 * 256, 16 * 256 + 1, 9000, 0, 3]
    if bulk:
        if (light, chunk) != (32, 256):
            pytest.skip("one shape of the large graph is enough")
        deg = deg + rng.integers(0, 37, bulk // 18).tolist() + deg
    deg = np.array(deg + [0] * max(0, 9100 - len(deg)))
    n = deg.size
    src = np.repeat(np.arange(n), deg)
    dst = rng.integers(0, n, src.size)
    order = np.argsort(dst, kind="stable")
    w = rng.uniform(0.5, 1.0, src.size).astype(np.float32) if weighted else None
    dev = lambda a, dt: torch.from_numpy(np.ascontiguousarray(a)).to(dt).cuda()  # noqa: E731
    off = lambda x: dev(np.concatenate([[0], np.cumsum(np.bincount(x, minlength=n))]), torch.int64)  # noqa: E731
    ws = [dev(w, torch.float32), dev(w[order], torch.float32)] if weighted else [None, None]
    G = gp.Graph(n, off(src), dev(dst, torch.int32), off(dst), dev(src[order], torch.int32), *ws, normalize=weighted)
    G.set_options(push_light_max=light, chunk_edges=chunk)
    wt = w.astype(np.float64) if weighted else np.ones(src.size)
    p = wt / np.bincount(src, weights=wt, minlength=n)[src]
    g = rng.standard_normal(n).astype(np.float32)
    x = torch.full((n,), 1.0 / n, device="cuda")
    d = float(np.float32(0.85))
    for iters, tol in ((1, 0.0), (4, 0.0), (400, 1e-3)):
        _, gs, st = gp.pagerank_backward(G, x, dev(g, torch.float32), gp.PULL, 0.85, iters, tol, want_weights=False)
        lam = g.astype(np.float64)
        for _ in range(st["iters_done"]):
            lam = g + d * np.bincount(src, weights=p * lam[dst], minlength=n)
        assert st["iters_done"] == iters if tol == 0.0 else st["converged"] and st["iters_done"] < 400
        bound = (deg.max() + 4) * 2.0 ** -24 / (1 - d) * np.abs(lam).max()
        assert np.abs(gs.cpu().numpy() - (1 - d) * lam).max() <= (1 - d) * bound + 1e-7


@pytest.mark.parametrize("tol", [0.0, 1e-3])
def test_drawn_units_repeat(gp, tol):
    """More groups of rows and chunks than warps, drawn in no fixed order: the same
    bits, sweeps and residual each time (no rounding may depend on who adds)."""
    import torch

    rng = np.random.default_rng(3)
    n = 300_000
    deg = rng.integers(0, 9, n)
    deg[rng.integers(0, n, 2000)] = rng.integers(33, 900, 2000)
    src = np.repeat(np.arange(n), deg)
    dst = rng.integers(0, n, src.size)
    order = np.argsort(dst, kind="stable")
    dev = lambda a, dt: torch.from_numpy(np.ascontiguousarray(a)).to(dt).cuda()  # noqa: E731
    off = lambda x: dev(np.concatenate([[0], np.cumsum(np.bincount(x, minlength=n))]), torch.int64)  # noqa: E731
    G = gp.Graph(n, off(src), dev(dst, torch.int32), off(dst), dev(src[order], torch.int32))
    g = dev(rng.standard_normal(n), torch.float32)
    x = torch.full((n,), 1.0 / n, device="cuda")
    runs = [gp.pagerank_backward(G, x, g, gp.PULL, 0.85, 12 if tol == 0.0 else 400, tol, want_weights=False)
            for _ in range(3)]
    for _, gs, st in runs[1:]:
        assert torch.equal(gs, runs[0][1])
        assert (st["iters_done"], st["residual"]) == (runs[0][2]["iters_done"], runs[0][2]["residual"])
