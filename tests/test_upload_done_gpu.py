"""The upload of a normalised graph returns with the sources' scale computed: a
program that uploads on one stream calls on others without waiting.  The sums
over 256M weights take the GPU longer than the host takes to ask."""
import pytest

pytestmark = pytest.mark.gpu


def test_nothing_in_flight_after_the_upload():
    import torch

    import paper_2010_16012_gb300 as gp

    n, deg = 1 << 22, 64
    off = torch.arange(n + 1, device="cuda") * deg
    idx = torch.randint(0, n, (n * deg,), dtype=torch.int32, device="cuda")
    w = torch.rand(n * deg, device="cuda")
    up = torch.cuda.Stream()
    torch.cuda.synchronize()
    for _ in range(3):
        G = gp.Graph(n, off, idx, off, idx, w, w, normalize=True, stream=up)
        assert up.query()
        G.free()
