"""The pull sweep's edge tiles (256 edges each, whatever the degrees) at the
places where they can go wrong: rows that end on, one before and one after a
tile's edge, rows over several and over more than sixteen tiles, vertices
without in-edges between them, one-edge rows, a last tile of one edge, index and
weight arrays that do not start on a 32-byte boundary.  Against the same sweeps
in FP64; tolerance of the method's contract (max-abs 1e-6, L1 1e-5)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

MAX_ABS, L1 = 1e-6, 1e-5
T = 256


@pytest.fixture(scope="module")
def gp():
    import torch

    import paper_2010_16012_gb300 as gp

    assert torch.cuda.is_available()
    gp.load()
    return gp


DEGREES = {
    "one edge": [1],
    "one tile": [T],
    "tile and one": [T, 1],
    "short of a tile": [T - 1],
    "over the edge": [T - 1, 2, T - 1, 1],
    "aligned rows": [T, 0, T, 2 * T, 0, 0, T],
    "one-edge rows": [1] * (3 * T + 1),
    "lanes": [8] * 40 + [7, 9, 0, 1] * 30,
    "sixteen tiles and more": [3, 16 * T, 5, 17 * T, 0, 18 * T + 1, 1, 40 * T - 9],
    "none": [0, 0, 0],
    "holes": [0, 0, 5, 0, 300, 0, 0, 1, 0],
}


def make(degrees, seed):
    """CSC with the given in-degrees over at least 64 vertices, its CSR and weights (some sources repeat)."""
    rng = np.random.default_rng(seed)
    n = max(64, len(degrees))
    deg = np.zeros(n, dtype=np.int64)
    deg[:len(degrees)] = degrees
    heads = np.repeat(np.arange(n), deg)
    tails = np.sort(rng.integers(0, n, heads.size) * (rng.random(heads.size) < 0.8))
    rng.shuffle(tails)
    csc_off = np.concatenate([[0], np.cumsum(deg)])
    order = np.argsort(tails, kind="stable")
    csr_off = np.concatenate([[0], np.cumsum(np.bincount(tails, minlength=n))])
    total = np.bincount(tails, minlength=n)[tails].astype(np.float64)
    w = rng.uniform(0.2, 1.0, heads.size) / np.maximum(total, 1)
    return n, csr_off, heads[order], w[order], csc_off, tails, w


def sweeps(n, csr_off, csc_off, tails, w, iters, d=float(np.float32(0.85))):
    heads = np.repeat(np.arange(n), np.diff(csc_off))
    scale = w if w is not None else 1.0 / np.maximum(np.diff(csr_off), 1)[tails]
    x = np.full(n, 1.0 / n)
    for _ in range(iters):
        x = (1 - d) / n + d * np.bincount(heads, weights=scale * x[tails], minlength=n)
    return x


@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("weighted", [False, True])
@pytest.mark.parametrize("slots", [0, 5])
@pytest.mark.parametrize("name", list(DEGREES))
def test_tiles(gp, name, slots, weighted, shift):
    import torch

    n, csr_off, csr_idx, csr_w, csc_off, csc_idx, csc_w = make(DEGREES[name], seed=len(name))

    def dev(a, dt):  # a view that starts `shift` elements into its storage
        return torch.cat([torch.zeros(shift, dtype=dt), torch.from_numpy(np.ascontiguousarray(a)).to(dt)]).cuda()[shift:]

    w = [dev(csr_w, torch.float32), dev(csc_w, torch.float32)] if weighted else [None, None]
    G = gp.Graph(n, dev(csr_off, torch.int64), dev(csr_idx, torch.int32), dev(csc_off, torch.int64),
                 dev(csc_idx, torch.int32), *w, validate=True)
    G.set_options(pull_hot_slots=slots)
    wx = csc_w.astype(np.float32).astype(np.float64) if weighted else None
    for iters in (1, 2, 3, 8):
        ref = sweeps(n, csr_off, csc_off, csc_idx, wx, iters)
        x, st = gp.pagerank(G, gp.PULL, 0.85, iters)
        err = np.abs(x.cpu().numpy().astype(np.float64) - ref)
        assert st["iters_done"] == iters
        assert err.max() <= MAX_ABS and err.sum() <= L1, (name, iters, float(err.max()), float(err.sum()))


@pytest.mark.parametrize("weighted,slots,shift", [(False, 20480, 0), (True, 20480, 1), (False, 0, 1)])
@pytest.mark.parametrize("bulk", [1_200_000, 8_600_000])
def test_tiles_of_larger_graphs(gp, bulk, weighted, slots, shift):
    """The same rows in graphs that the one-launch loop holds a tile to a warp no
    longer (1.2M edges) and that run a launch per step (8.6M edges, above 32768
    tiles): before and after a bulk of other rows, and a last tile cut short."""
    import torch

    rng = np.random.default_rng(bulk)
    edges = [d for name in DEGREES for d in DEGREES[name]]
    fill = rng.integers(0, 33, bulk // 16).tolist()
    n, csr_off, csr_idx, csr_w, csc_off, csc_idx, csc_w = make(edges + fill + edges, seed=3)

    def dev(a, dt):
        return torch.cat([torch.zeros(shift, dtype=dt), torch.from_numpy(np.ascontiguousarray(a)).to(dt)]).cuda()[shift:]

    w = [dev(csr_w, torch.float32), dev(csc_w, torch.float32)] if weighted else [None, None]
    G = gp.Graph(n, dev(csr_off, torch.int64), dev(csr_idx, torch.int32), dev(csc_off, torch.int64),
                 dev(csc_idx, torch.int32), *w)
    G.set_options(pull_hot_slots=slots)
    wx = csc_w.astype(np.float32).astype(np.float64) if weighted else None
    for iters in (1, 2, 5):
        ref = sweeps(n, csr_off, csc_off, csc_idx, wx, iters)
        x, st = gp.pagerank(G, gp.PULL, 0.85, iters)
        err = np.abs(x.cpu().numpy().astype(np.float64) - ref)
        assert st["iters_done"] == iters
        assert err.max() <= MAX_ABS and err.sum() <= L1, (iters, float(err.max()), float(err.sum()))
    ref = sweeps(n, csr_off, csc_off, csc_idx, wx, 200)
    x, st = gp.pagerank(G, gp.PULL, 0.85, 200, 1e-6)  # stopped by the residual, within its bound of the fixed point
    err = np.abs(x.cpu().numpy().astype(np.float64) - ref)
    assert st["converged"] and st["residual"] < 1e-6 and st["iters_done"] < 200 and err.sum() <= 1e-6 / 0.15 + L1


@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("weighted", [False, True])
@pytest.mark.parametrize("slots", [0, 5])
@pytest.mark.parametrize("name", list(DEGREES))
def test_push_tiles(gp, name, slots, weighted, shift):
    """The same lists as out-edges: the push sweep's tiles, heads that several of a tile's sources share among them."""
    import torch

    n, csc_off, csc_idx, csc_w, csr_off, csr_idx, csr_w = make(DEGREES[name], seed=len(name))
    out = np.maximum(np.bincount(np.repeat(np.arange(n), np.diff(csr_off)), minlength=n), 1)
    csr_w = csr_w / out[np.repeat(np.arange(n), np.diff(csr_off))]  # scaled down: what leaves a source stays below 1
    csc_w = csr_w[np.argsort(csr_idx, kind="stable")]

    def dev(a, dt):
        return torch.cat([torch.zeros(shift, dtype=dt), torch.from_numpy(np.ascontiguousarray(a)).to(dt)]).cuda()[shift:]

    w = [dev(csr_w, torch.float32), dev(csc_w, torch.float32)] if weighted else [None, None]
    G = gp.Graph(n, dev(csr_off, torch.int64), dev(csr_idx, torch.int32), dev(csc_off, torch.int64),
                 dev(csc_idx, torch.int32), *w, validate=True)
    G.set_options(push_hot_slots=slots, push_fp64_accum=1)
    wx = csc_w.astype(np.float32).astype(np.float64) if weighted else None
    for iters in (1, 3):
        ref = sweeps(n, csr_off, csc_off, csc_idx, wx, iters)
        x, st = gp.pagerank(G, gp.PUSH, 0.85, iters)
        err = np.abs(x.cpu().numpy().astype(np.float64) - ref)
        assert st["push_updates_l2"] + st["push_updates_shared"] + st["push_updates_merged"] == csr_idx.size * iters
        assert err.max() <= MAX_ABS and err.sum() <= L1, (name, iters, float(err.max()), float(err.sum()))


@pytest.mark.parametrize("mode", ["PUSH", "PULL"])
def test_hot_set_sizes_in_turn(gp, mode):
    """A large hot set, a small one and the large one again, on one graph and with another graph's in between: every
    size's shared memory is to be had each time.  Equal to the run without a hot set within the orders' rounding."""
    import torch

    rng = np.random.default_rng(1)
    n = 60_000
    deg = rng.integers(0, 300, n)  # over 32768 tiles: a launch per step
    src = np.repeat(np.arange(n), deg)
    dst = rng.integers(0, n, src.size)
    order = np.argsort(dst, kind="stable")
    off = lambda x: torch.from_numpy(np.concatenate([[0], np.cumsum(np.bincount(x, minlength=n))])).cuda()  # noqa: E731
    arrays = off(src), torch.from_numpy(dst).int().cuda(), off(dst), torch.from_numpy(src[order]).int().cuda()
    A, B = gp.Graph(n, *arrays), gp.Graph(n, *arrays)
    key = mode.lower() + "_hot_slots"
    ref = None
    for G, slots in ((A, 0), (A, 40960), (A, 8192), (A, 40960), (B, 4096), (A, 40960), (B, 4096)):
        G.set_options(**{key: slots})
        x, _ = gp.pagerank(G, getattr(gp, mode), 0.85, 3)
        x = x.cpu().numpy().astype(np.float64)
        ref = x if ref is None else ref
        assert np.abs(x - ref).max() <= MAX_ABS and np.abs(x - ref).sum() <= L1, (slots,)
