"""Betweenness of several sources at a time (groups of blocks that draw sources):
fewer sources than groups, as many, more, repeated ones, a group that meets a
bad source while others work, and the clean call after it.  Against the oracle,
relative 1e-9 (the method's contract)."""
import numpy as np
import pytest

import graphgen as gg
import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gp():
    import torch

    import paper_2010_16012_gb300 as gp

    assert torch.cuda.is_available()
    gp.load()
    return gp


def close(x, ref):
    return np.all(np.abs(x.cpu().numpy() - ref) <= 1e-9 * np.maximum(np.abs(ref), 1e-3 * np.abs(ref).max()))


@pytest.mark.parametrize("g", [lambda: gg.rmat(11, 8, seed=3), lambda: gg.rmat(10, 8, seed=4, symmetrize=False),
                               lambda: gg.path(300), lambda: gg.star(1500)])
def test_counts_of_sources(gp, g):
    import torch

    g = g()
    G = gp.Graph.from_graphgen(g)
    O = oracle.OracleGraph.from_graph(g)
    rng = np.random.default_rng(1)
    for k in (1, 2, 15, 16, 17, 40, 3):
        src = rng.integers(0, g.n, k).astype(np.int32)
        src[k // 2] = src[0]
        x, st = gp.bc(G, src)
        ref = O.bc(src)
        assert close(x, ref), k
        assert st["sources"] == k and st["reached"] >= k
    bad = rng.integers(0, g.n, 20).astype(np.int32)
    bad[7] = g.n
    with pytest.raises(gp.GpError):
        gp.bc(G, torch.from_numpy(bad).cuda())
    x, _ = gp.bc(G, src)
    assert close(x, ref)
