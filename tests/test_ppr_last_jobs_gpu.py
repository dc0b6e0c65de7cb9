"""Batched PageRank where one graph's slices leave several slow last columns,
which then share a job: seeds in pairs (whose alternating mode decays as d^k
only), in different components, so that what one column reaches says nothing of
the others; closed sets, a set that the column still runs along (a long path),
one after the other in either order.  Slices of 64 columns leave two of them,
slices of 32 four.  Every column against the power iteration in FP64 at its own
sweep count: the result, and its L1 change below the tolerance.  Bounds: a sweep
rounds an entry four times at most (sum, compensation, product, base; the scales
1/2 and 1 are exact), each by 2^-24 of it, the entries of a column sum to one and
a sweep takes errors on with the factor d in the L1 norm, so the iterate is within
4 * 2^-24 / (1 - d) and the change of two of them within twice that.  At d = 0.99
that is 4.8e-5, so the tolerance there is 1e-4."""
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


def components(n, last):
    """Rings and paths of n vertices (the rest alone): edges, and the first vertices of each kind."""
    src, dst, at = [], [], 0
    first = {}

    def ring(kind, size, closed=True):
        nonlocal at
        v = np.arange(at, at + size)
        src.extend(v[:-1]), dst.extend(v[1:])
        if closed and size > 2:
            src.append(v[-1]), dst.append(v[0])
        first.setdefault(kind, []).append(at + (0 if closed else size // 2))
        at += size

    for i in range(8):
        for kind, size in (("3", 3), ("5", 5), ("7", 7), ("7", 7), ("9", 9), ("9", 9)):
            ring(kind, size)
    for kind in last:
        if kind == "pair":
            ring("last", 2)
        elif kind == "six":
            ring("last", 6)
        else:
            ring("last", 420, closed=False)
    assert at <= n
    s, d = np.array(src + dst), np.array(dst + src)
    order = np.lexsort((d, s))
    return s[order], d[order], first


@pytest.mark.parametrize("damping,tol", [(0.85, 1e-6), (0.99, 1e-4)])
@pytest.mark.parametrize("last", [("pair", "pair"), ("pair", "path"), ("path", "pair"), ("six", "pair"),
                                  ("pair", "pair", "pair", "pair"), ("pair", "six", "path", "pair")])
def test_several_last_columns(gp, last, damping, tol):
    import torch
    from scipy.sparse import csr_matrix

    # two iterates of 64 columns fit 1 MiB up to n = 2048: slices of 64 below, of 32 above
    n, width = (1900, 64) if len(last) == 2 else (2600, 32)
    src, dst, first = components(n, last)
    K, nslices = 256, 256 // width
    seeds = np.empty(K, dtype=np.int64)
    for i in range(nslices):
        s = [first["3"][i]] * (width - 16) + [first["5"][i]] * 12 + first["7"][2 * i:2 * i + 2]
        s += [first["9"][2 * i], first["9"][2 * i + 1] if i % 2 == 0 else first["last"][i // 2]]
        seeds[i * width:(i + 1) * width] = s
    off = np.concatenate([[0], np.cumsum(np.bincount(src, minlength=n))])
    G = gp.Graph(n, torch.from_numpy(off).cuda(), torch.from_numpy(dst).int().cuda(), symmetric=True, validate=True)
    B = gp.Batch([G], k_ppr=K)
    B.set_options(l2_budget_mb=1)
    deg = np.maximum(np.bincount(src, minlength=n), 1)
    P = csr_matrix((1.0 / deg[src], (dst, src)), shape=(n, n))
    E = np.zeros((n, K))
    E[seeds, np.arange(K)] = 1.0
    d = float(np.float32(damping))
    bound = 4 * 2.0 ** -24 / (1 - d)
    for _ in range(2):  # a second call starts from the first one's work areas
        outs, done, st = B.ppr(seeds, damping, iters=3000, tol=tol)
        assert st["jobs"] == nslices and st["packed"] == 16 * nslices
        done = done[0]
        assert 0 < done.min() and done.max() < 3000
        got = outs[0].cpu().numpy().astype(np.float64)
        x, ref, change = E, np.zeros_like(E), np.full(K, np.inf)
        for k in range(1, int(done.max()) + 1):
            y = (1.0 - d) * E + d * (P @ x)
            at = done == k
            ref[:, at] = y[:, at]
            change[at] = np.abs(y - x)[:, at].sum(axis=0)
            x = y
        err = np.abs(got - ref)
        bad = np.nonzero((err.sum(axis=0) > bound) | (change > tol + 2 * bound))[0]
        assert bad.size == 0, [(int(j), int(done[j]), float(err[:, j].sum()), float(change[j])) for j in bad]
    B.free()
