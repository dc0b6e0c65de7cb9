"""Batched PageRank's last columns, swept on the rows that they reach: seeds in
small components (pairs, a triangle, a path, vertices alone) beside a large one,
sets that edges leave (a chain that the column still runs along), a long in-list
inside the set, few and many columns left, stops by tolerance and by the cap at
odd and even sweeps.  Against the power iteration in FP64 at each column's own
sweep count; tolerance of the method's contract (max-abs 1e-6, L1 1e-5)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

MAX_ABS, L1 = 1e-6, 1e-5


@pytest.fixture(scope="module")
def gp():
    import torch

    import paper_2010_16012_gb300 as gp

    assert torch.cuda.is_available()
    gp.load()
    return gp


def edges(kind):
    """Vertices 0..1999 a large component, then the small sets; returns n, src, dst and seeds in the small sets."""
    rng = np.random.default_rng(4)
    s, d = rng.integers(0, 2000, 12000), rng.integers(0, 2000, 12000)
    ring = np.arange(2000)
    s, d = np.concatenate([s, ring]), np.concatenate([d, (ring + 1) % 2000])
    small = [(2000 + 2 * i, 2001 + 2 * i) for i in range(5)]          # pairs
    small += [(2010, 2011), (2011, 2012), (2010, 2012)]               # a triangle
    small += [(2013 + i, 2014 + i) for i in range(5)]                 # a path
    a, b = np.array(small).T
    n = 2600
    s, d = np.concatenate([s, a]), np.concatenate([d, b])
    s, d = np.concatenate([s, d]), np.concatenate([d, s])
    if kind == "leaves":  # a pair whose mass runs along a one-way chain to the end
        c = np.arange(2100, 2590)
        s, d = np.concatenate([s, [2000], c]), np.concatenate([d, [2100], c + 1])
    if kind == "long":    # a pair into a vertex that many of the large component lead to as well
        c = rng.permutation(2000)[:300]
        s, d = np.concatenate([s, [2000, 2001], c]), np.concatenate([d, [2599] * 302])
    key = np.unique((s * n + d)[s != d])
    return n, key // n, key % n, [2000, 2001, 2002, 2005, 2006, 2010, 2013, 2015, 2598, 2020]


@pytest.mark.parametrize("iters", [500, 30, 31])
@pytest.mark.parametrize("nslow", [2, 7, 10])
@pytest.mark.parametrize("kind", ["closed", "leaves", "long"])
def test_last_columns(gp, kind, nslow, iters):
    import torch
    from scipy.sparse import csr_matrix

    n, src, dst, slow = edges(kind)
    order = np.argsort(dst, kind="stable")
    dev = lambda a, dt: torch.from_numpy(np.ascontiguousarray(a)).to(dt).cuda()  # noqa: E731
    off = lambda x: dev(np.concatenate([[0], np.cumsum(np.bincount(x, minlength=n))]), torch.int64)  # noqa: E731
    G = gp.Graph(n, off(src), dev(dst, torch.int32), off(dst), dev(src[order], torch.int32))
    k = 32
    seeds = np.random.default_rng(nslow).integers(0, 2000, (1, k))
    seeds[0, 3:3 + nslow] = slow[:nslow]
    B = gp.Batch([G], k_ppr=k)
    P = csr_matrix((1.0 / np.bincount(src, minlength=n)[src], (dst, src)), shape=(n, n))
    for _ in range(2):  # a second call starts from the first one's work areas
        outs, done, st = B.ppr(seeds, iters=iters, tol=1e-6)
        assert done.max() <= iters
        assert st["packed"] > 0 or kind == "long"  # (there the mass drains and all columns may stop together)
        X = outs[0].cpu().numpy().astype(np.float64)
        for j in range(k):
            e = np.zeros(n)
            e[seeds[0, j]] = 1.0
            x, r = e, 0.0
            for _ in range(int(done[0, j])):
                y = 0.15 * e + 0.85 * (P @ x)
                r, x = np.abs(y - x).sum(), y
            err = np.abs(X[:, j] - x)
            assert err.max() <= MAX_ABS and err.sum() <= L1, (j, int(done[0, j]), float(err.max()))
            assert r < 1e-6 + 8e-7 or done[0, j] == iters, (j, r)
    B.free()
