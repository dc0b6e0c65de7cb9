"""Shortest paths after gp_graph_set_weights: the check of the weights is of the
present ones; and zero-weight edges out of vertex 0 as the source, whose head's
key (distance 0, predecessor 0) is the least there is."""
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


def path(gp, w):
    """0 -> 1 -> 2 -> 3 with weights w."""
    import torch

    dev = lambda a, dt: torch.tensor(a, dtype=dt, device="cuda")  # noqa: E731
    return gp.Graph(4, dev([0, 1, 2, 3, 3], torch.int64), dev([1, 2, 3], torch.int32),
                    dev([0, 0, 1, 2, 3], torch.int64), dev([0, 1, 2], torch.int32),
                    dev(w, torch.float32), dev(w, torch.float32))


@pytest.mark.parametrize("bad", [-1.0, float("nan")])
@pytest.mark.parametrize("start_bad", [False, True])
def test_weights_checked_anew(gp, bad, start_bad):
    import torch

    good, wrong = [1.0, 2.0, 3.0], [1.0, bad, 3.0]
    G = path(gp, wrong if start_bad else good)
    for i in range(4):
        ok = (i % 2 == 0) != start_bad
        if i:
            w = torch.tensor(good if ok else wrong, device="cuda")
            G.set_weights(w, w.clone())
        if ok:
            dist, pred, _ = gp.sssp(G, 0, 1.5)
            assert dist.tolist() == [0.0, 1.0, 3.0, 6.0] and pred.tolist() == [0, 0, 1, 2]
        else:
            with pytest.raises(gp.GpError) as e:
                gp.sssp(G, 0, 1.5)
            assert e.value.status == -1


@pytest.mark.parametrize("mode", [0, 1, 2])
@pytest.mark.parametrize("fan", [3, 700])
def test_zero_weight_from_vertex_zero(gp, mode, fan):
    """0 -> every v at weight 0, and v -> v + 1 at weight 0 (and back to 0): all distances 0, predecessor 0."""
    import torch

    n = fan + 1
    src = np.concatenate([np.zeros(fan, dtype=np.int64), np.arange(1, n), np.arange(1, n - 1)])
    dst = np.concatenate([np.arange(1, n), np.zeros(fan, dtype=np.int64), np.arange(2, n)])
    order = np.lexsort((dst, src))
    src, dst = src[order], dst[order]
    csc = np.lexsort((src, dst))
    dev = lambda a, dt: torch.from_numpy(np.ascontiguousarray(a)).to(dt).cuda()  # noqa: E731
    off = lambda x: dev(np.concatenate([[0], np.cumsum(np.bincount(x, minlength=n))]), torch.int64)  # noqa: E731
    w = torch.zeros(src.size, device="cuda")
    G = gp.Graph(n, off(src), dev(dst, torch.int32), off(dst), dev(src[csc], torch.int32), w, w.clone())
    dist, pred, st = gp.sssp(G, 0, 1.0, mode)
    assert not dist.any() and not pred.any() and st["reached"] == n
