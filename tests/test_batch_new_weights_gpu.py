"""Batched PageRank on graphs whose weights were replaced after the batch was
made: the same as gp_pagerank with the seed's personalization on the graph as it
is now.  Bound: the method's contract (max-abs 1e-6)."""
import numpy as np
import pytest

import graphgen as gg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("normalize", [True, False])
def test_batch_follows_the_graph(normalize):
    import torch

    import paper_2010_16012_gb300 as gp

    g = gg.rmat(10, 8, seed=5, symmetrize=False)
    rng = np.random.default_rng(1)
    src = np.repeat(np.arange(g.n), np.diff(g.csr_off))
    order = np.lexsort((src, g.csr_idx))
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731

    def weights():
        w = rng.uniform(0.05, 1.0, g.m)
        if not normalize:
            w /= np.bincount(src, weights=w, minlength=g.n)[src]
        w = w.astype(np.float32)
        return t(w), t(w[order])

    old = weights()
    arrays = t(g.csr_off), t(g.csr_idx), t(g.csc_off), t(g.csc_idx)
    G = gp.Graph(g.n, *arrays, *old, normalize=normalize, validate=True)
    H = gp.Graph(g.n, *arrays, *old, normalize=normalize)
    B = gp.Batch([H, G], k_ppr=32)
    seeds = rng.integers(0, g.n, (2, 32))
    for new in (None, weights(), weights()):
        if new is not None:
            G.set_weights(*new)
        outs, done, _ = B.ppr(seeds, iters=200, tol=1e-7)
        for graph, x, sd in ((H, outs[0], seeds[0]), (G, outs[1], seeds[1])):
            for j in range(0, 32, 7):
                s = torch.zeros(g.n, device="cuda")
                s[int(sd[j])] = 1.0
                ref, _ = gp.pagerank(graph, gp.PULL, iters=200, tol=1e-7, personalization=s, x0=s)
                assert (x[:, j] - ref).abs().max() <= 1e-6
    B.free()
