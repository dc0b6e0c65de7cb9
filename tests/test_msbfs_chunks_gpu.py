"""Batched BFS where lists are cut in chunks and graphs share one range of
units: hubs in one direction only, graphs of fewer vertices than a unit beside
larger ones, fewer searches than columns, outputs in device memory that holds
something else and in host memory.  Levels against the oracle's: equal, -1 where
nothing is reached and in unused columns."""
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


def out_star(k, inward):
    """A hub of k edges to (or from) leaves, and a path through the leaves; directed."""
    hub, leaf = np.zeros(k, dtype=np.int64), np.arange(1, k + 1)
    a, b = (leaf, hub) if inward else (hub, leaf)
    return gg.from_edges(k + 1, np.concatenate([a, leaf[:-1]]), np.concatenate([b, leaf[1:]]))


GRAPHS = [lambda: out_star(700, False), lambda: gg.path(5), lambda: out_star(3000, True),
          lambda: gg.rmat(9, 8, seed=4, symmetrize=False), lambda: gg.star(129), lambda: gg.rmat(11, 16, seed=2),
          lambda: gg.empty(33)]


@pytest.mark.parametrize("nsrc", [1, 33, 64])
@pytest.mark.parametrize("opts", [{}, dict(big_in_degree=0, chunk_edges=32), dict(big_in_degree=100000),
                                  dict(msbfs_alpha=1e9, msbfs_beta=1e-9), dict(msbfs_alpha=1e-9)])
def test_levels(gp, nsrc, opts):
    import torch

    gs = [g() for g in GRAPHS]
    B = gp.Batch([gp.Graph.from_graphgen(g) for g in gs], k_ppr=32)
    B.set_options(**opts)
    rng = np.random.default_rng(nsrc)
    src = np.stack([rng.integers(0, g.n, nsrc) for g in gs])
    src[:, 0] = 0
    outs = [torch.full((g.n, 64), 77, dtype=torch.int32, device="cuda") if i != 3 else
            np.full((g.n, 64), 77, dtype=np.int32) for i, g in enumerate(gs)]
    for _ in range(2):
        B.msbfs(src, outs=outs)
        for i, g in enumerate(gs):
            O = oracle.OracleGraph.from_graph(g)
            got = outs[i] if i == 3 else outs[i].cpu().numpy()
            assert (got[:, nsrc:] == -1).all()
            for j in range(nsrc):
                assert np.array_equal(got[:, j], O.bfs(int(src[i, j]))[0]), (i, j)
