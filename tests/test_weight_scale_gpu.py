"""Normalised uploads and gp_graph_set_weights: the per-source weight sums at
the edges of the light limit and of the chunks (and a hub over many chunks),
seen through one PageRank sweep, which is linear in them.  Bound: one FP32
rounding each of the scale, the contribution, the product and the scaled base
per term, and of the sum of at most 3 terms per head."""
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


@pytest.mark.parametrize("light,chunk", [(32, 256), (0, 32), (1 << 20, 256)])
def test_weight_sums(gp, light, chunk):
    import torch

    out_deg = [0, 1, 2, 31, 32, 33, 255, 256, 257, 511, 512, 513, 0, 5000, 1]
    n = max(out_deg)
    rng = np.random.default_rng(5)
    deg = np.zeros(n, dtype=np.int64)
    deg[:len(out_deg)] = out_deg
    src = np.repeat(np.arange(n), deg)
    dst = np.concatenate([np.sort(rng.permutation(n)[:k]) for k in deg]).astype(np.int64)
    order = np.lexsort((src, dst))
    off = lambda x: torch.from_numpy(np.concatenate([[0], np.cumsum(np.bincount(x, minlength=n))])).cuda()  # noqa: E731
    dev = lambda a, dt: torch.from_numpy(np.ascontiguousarray(a)).to(dt).cuda()  # noqa: E731
    most = int(np.bincount(dst, minlength=n).max())
    arrays = off(src), dev(dst, torch.int32), off(dst), dev(src[order], torch.int32)
    for upload in (True, False):  # the weights given at upload, and set afterwards
        w = rng.uniform(0.01, 1.0, dst.size).astype(np.float32)
        w0 = w if upload else np.ones_like(w)
        G = gp.Graph(n, *arrays, dev(w0, torch.float32), dev(w0[order], torch.float32), normalize=True, validate=True)
        G.set_options(push_light_max=light, chunk_edges=chunk)
        if upload:  # the options rebuild the chunks; the sums do not change
            pass
        else:
            G.set_weights(dev(w, torch.float32), dev(w[order], torch.float32))
        x, _ = gp.pagerank(G, gp.PULL, 0.85, 1)
        w64 = w.astype(np.float64)
        p = w64 / np.bincount(src, weights=w64, minlength=n)[src]
        d = float(np.float32(0.85))
        gathered = d / n * np.bincount(dst, weights=p, minlength=n)
        ref = (1 - d) / n + gathered
        assert np.all(np.abs(x.cpu().numpy() - ref) <= 2.0 ** -24 * (4 + most) * (gathered + 1.0 / n))
