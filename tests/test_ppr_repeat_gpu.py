"""A batched PageRank column's sweep count does not depend on the order in which
the warps take their work: the sweep's L1 change is the same in every run to far
below FP32 rounding, so with a tolerance just above it the column stops there in
every run, and just below it in none.  The change (of the device's iterates) is
found by bisection on the tolerance; the margin of 1e-9 is between the FP32
rounding of one sum (6e-8) and that of the compensated sums (n terms of 2^-48
each, 1e-9 for 3e5 vertices at the very most)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,k,budget", [(300007, 32, 96), (150001, 128, 192)])
def test_stops_at_the_same_sweep(n, k, budget):
    import torch

    import paper_2010_16012_gb300 as gp

    gen = torch.Generator(device="cuda").manual_seed(11)
    s, d = (torch.randint(0, n, (6 * n,), generator=gen, device="cuda") for _ in range(2))
    key = torch.unique(torch.cat([s * n + d, d * n + s])[torch.cat([s, s]) != torch.cat([d, d])])
    row, col = key // n, (key % n).int()
    off = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    off[1:] = torch.cumsum(torch.bincount(row, minlength=n), 0)
    G = gp.Graph(n, off, col, symmetric=True)
    B = gp.Batch([G], k_ppr=k)
    B.set_options(l2_budget_mb=budget, ppr_start=0)
    seeds = torch.randint(0, n, (1, k), generator=gen, device="cuda").cpu().numpy()
    sweep = 9
    # the change of sweep 9, by the FP64 iteration of column 0
    inv = 1.0 / torch.bincount(row, minlength=n).clamp(min=1).double()
    x = torch.full((n,), 1.0 / n, dtype=torch.float64, device="cuda")
    e = torch.zeros_like(x)
    e[int(seeds[0, 0])] = 1.0
    damp = float(np.float32(0.85))
    for _ in range(sweep):
        y = (1 - damp) * e + damp * torch.zeros_like(x).index_add_(0, col.long(), (x * inv)[row])
        change, x = float((y - x).abs().sum()), y

    def stops(tol):
        return B.ppr(seeds, iters=sweep + 1, tol=tol)[1][0, 0] <= sweep

    lo, hi = change * (1 - 1e-4), change * (1 + 1e-4)
    assert stops(hi) and not stops(lo)
    for _ in range(20):  # to 2e-10 of the change
        mid = 0.5 * (lo + hi)
        lo, hi = (lo, mid) if stops(mid) else (mid, hi)
    above, below = hi * (1 + 1e-9), lo * (1 - 1e-9)
    assert all(stops(above) for _ in range(25))
    assert not any(stops(below) for _ in range(25))
    B.free()
