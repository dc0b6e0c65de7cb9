"""Triangle counts by the directed lists at the places where they can go wrong:
lists at and around the warp/block limit (32 out-neighbours), tables at and
around their doublings, one and no out-neighbour, self-loops; and the inputs
that take the listing instead (a duplicate edge, an unsorted list), against the
listing itself.  Whole numbers: equal."""
import math

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


def upload(gp, n, rows):
    import torch

    off = np.concatenate([[0], np.cumsum([len(r) for r in rows])])
    idx = np.concatenate([np.asarray(r, dtype=np.int64) for r in rows])
    return gp.Graph(n, torch.from_numpy(off).cuda(), torch.from_numpy(idx).int().cuda(), symmetric=True)


def clique_rows(n, k, loops=False):
    """A clique on the last k of n vertices; the others hang on vertex n - 1."""
    rows = [[n - 1] for _ in range(n - k)]
    rows += [[u for u in range(n - k, n) if loops or u != v] for v in range(n - k, n)]
    rows[n - 1] = sorted(set(rows[n - 1]) | set(range(n - k)))
    return rows


def listing(n, rows):
    """The NodeIterator as the general kernels run it: every edge slot (v, w), the shorter list's elements found in the longer."""
    tc, probes = np.zeros(n, dtype=np.int64), 0
    for v in range(n):
        for w in rows[v]:
            if w == v:
                continue
            a, b = (rows[v], rows[w]) if len(rows[v]) <= len(rows[w]) else (rows[w], rows[v])
            probes += len(a)
            tc[v] += sum(x not in (v, w) and x in set(b) for x in a)
    return tc // 2, probes


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("k", [2, 3, 32, 33, 34, 64, 65, 66, 129, 257, 600, 2100])
def test_cliques(gp, k, mode):
    n = k + 5
    G = upload(gp, n, clique_rows(n, k))
    for _ in range(2):  # the lists are built by the first call
        tc, total, st = gp.triangles(G, mode)
        ref = np.zeros(n, dtype=np.int64)
        ref[n - k:] = math.comb(k - 1, 2)
        assert np.array_equal(tc.cpu().numpy(), ref) and total == st["triangles"] == math.comb(k, 3)
        deg = np.array([1] * 5 + [k - 1] * (k - 1) + [k + 4])
        assert st["probes"] == (k - 1) * (k - 2) * (k - 1) + 2 * (k - 1) * (k - 1) + 2 * 5 * 1, deg


@pytest.mark.parametrize("mode", [0, 1])
def test_self_loops_and_random(gp, mode):
    rng = np.random.default_rng(3)
    n = 150
    adj = np.triu(rng.random((n, n)) < 0.4, 1)
    adj = adj | adj.T
    adj[np.arange(0, n, 3), np.arange(0, n, 3)] = True
    adj[7, :] = adj[:, 7] = False
    rows = [np.nonzero(adj[v])[0].tolist() for v in range(n)]
    ref, probes = listing(n, rows)
    tc, total, st = gp.triangles(upload(gp, n, rows), mode)
    assert np.array_equal(tc.cpu().numpy(), ref) and total == ref.sum() // 3 and st["probes"] == probes


@pytest.mark.parametrize("mode", [0, 1])
def test_outside_the_contract(gp, mode):
    """A duplicate edge (both ways) and a list out of order: the listing's answer, as ever."""
    rows = clique_rows(9, 6)
    rows[4] = sorted(rows[4] + [6])
    rows[6] = sorted(rows[6] + [4])
    ref, probes = listing(9, rows)
    tc, total, st = gp.triangles(upload(gp, 9, rows), mode)
    if mode == 1:  # push credits w1 instead of v: the same sums on a simple graph only
        assert np.array_equal(tc.cpu().numpy(), ref)
    assert st["probes"] == probes
    rows = clique_rows(9, 6)
    rows[0] = []
    rows[8] = [r for r in rows[8] if r != 0]
    rows[5] = rows[5][::-1]
    tc, total, st = gp.triangles(upload(gp, 9, rows), mode)  # searched as if sorted: ends, in bounds
    assert 0 <= total <= math.comb(6, 3)


@pytest.mark.parametrize("mode", [0, 1])
def test_one_way_edges(gp, mode):
    """A graph called symmetric whose edge 8 -> 3 has no reverse (and 2 -> 6 none, so that the lists' lengths
    agree): the listing's answer, on the first call and after."""
    rows = clique_rows(9, 6)
    rows[8] = [r for r in rows[8] if r != 3]
    rows[2] = sorted(rows[2] + [6])
    ref, probes = listing(9, rows)
    G = upload(gp, 9, rows)
    for _ in range(2):
        tc, total, st = gp.triangles(G, mode)
        if mode == 1:
            assert np.array_equal(tc.cpu().numpy(), ref)
        assert st["probes"] == probes


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("n", [(1 << 19) - 1, 1 << 19, (1 << 19) + 1])
def test_bitmap_and_table(gp, n, mode):
    """A clique at each end of the ids of a graph at, below and above the vertices whose bitmap fits in shared
    memory (the hash table from there on), joined by one edge."""
    import torch

    k = 90
    a = np.concatenate([np.arange(k), np.arange(n - k, n)])
    u, v = np.triu_indices(k, 1)
    src = np.concatenate([a[u], a[k + u], [a[0]]])
    dst = np.concatenate([a[v], a[k + v], [a[-1]]])
    src, dst = np.concatenate([src, dst]), np.concatenate([dst, src])
    order = np.lexsort((dst, src))
    off = np.concatenate([[0], np.cumsum(np.bincount(src, minlength=n))])
    G = gp.Graph(n, torch.from_numpy(off).cuda(), torch.from_numpy(dst[order]).int().cuda(), symmetric=True)
    tc, total, _ = gp.triangles(G, mode)
    ref = np.zeros(n, dtype=np.int64)
    ref[a] = math.comb(k - 1, 2)
    assert total == 2 * math.comb(k, 3) and np.array_equal(tc.cpu().numpy(), ref)


@pytest.mark.parametrize("mode", [0, 1])
def test_one_way_edge_into_the_last_vertex(gp, mode):
    """An edge without its reverse into the last vertex, whose in-list is empty and lies at the end of all of them
    (and another one-way edge, so that the lists' lengths agree): nothing counted for it has a place to go."""
    k = 6
    n = k + 3
    rows = [[] for _ in range(n)]
    for v in range(2, k + 2):
        rows[v] = [u for u in range(2, k + 2) if u != v]
    rows[0] = [4, n - 1]        # one way to n - 1
    rows[4] = [0] + rows[4]
    rows[2] = [1] + rows[2]     # one way to 1
    rows[n - 1] = [2, 3]
    rows[2].append(n - 1)
    rows[3].append(n - 1)
    ref, probes = listing(n, rows)
    G = upload(gp, n, rows)
    for _ in range(2):
        tc, total, st = gp.triangles(G, mode)
        if mode == 1:
            assert np.array_equal(tc.cpu().numpy(), ref)
        assert st["probes"] == probes
