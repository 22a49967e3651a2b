"""Rows past the block class, beside few and beside many other entries: by the
hub kernels in the first case, by the block kernel in the second."""
import numpy as np
import pytest
import torch

import inputs as I
import oracle as O

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


def hubs_among(length, others, seed):
    """Two rows of `length` entries and about `others` entries of random pairs."""
    rng = np.random.default_rng(seed)
    n = 140_000
    u = [rng.integers(0, n, others // 2)] + [np.full(length, n + k) for k in range(2)]
    v = [rng.integers(0, n, others // 2)] + [rng.choice(n, length, replace=False) for _ in range(2)]
    u, v = np.concatenate(u), np.concatenate(v)
    keep = u != v
    return I.csr_from_pairs(n + 2, u[keep], v[keep], perm=rng.permutation(n + 2), name="hubs-among")


@pytest.mark.parametrize("weighted", [False, True])
# hidden by 512 times the longest row's entries, up to 131,072 by 128 times
@pytest.mark.parametrize("length, others, slot, idle", [
    (131_100, 0, "sweep_hub", "sweep_block"), (131_100, 17_000_000, "sweep_hub", "sweep_block"),
    (131_100, 68_000_000, "sweep_block", "sweep_hub"),
    (32_769, 0, "sweep_hub", "sweep_block"), (40_000, 1_000_000, "sweep_hub", "sweep_block"),
    (40_000, 5_300_000, "sweep_block", "sweep_hub")])
def test_route_and_labels(gpu_lib, length, others, slot, idle, weighted):
    g = hubs_among(length, others, seed=others + length)
    d = np.diff(g.offsets)
    rest = 512 if length > 131_072 else 128
    assert (d >= length).sum() == 2 and (g.nnz < rest * d.max()) == (slot == "sweep_hub")
    if weighted:
        g = I.Graph(g.offsets, g.cols, I.symmetric_weights(g, 4, 9))
    off, col = torch.from_numpy(g.offsets).to(DEV), torch.from_numpy(g.cols).to(DEV)
    w = torch.from_numpy(g.weights).to(DEV) if weighted else None
    c = gpu_lib.Context(0)
    c.set_profiling(True)
    got, st = c.lpa(off, col, w, tolerance=0.0, max_iters=3, stats=True)
    want, t, dn = O.lpa_sync(g, 0.0, 3)
    assert st["iterations"] == t and st["changed"] == dn[:t].tolist()
    assert np.array_equal(got.cpu().numpy(), want)
    launches = {p["name"]: p["launches"] for p in c.profile()}
    assert launches[slot] > 0 and launches[idle] == 0


# in place, up to 768 times
@pytest.mark.parametrize("others, slot", [(5_300_000, "sweep_hub"), (32_000_000, "sweep_block")])
def test_route_in_place(gpu_lib, others, slot):
    g = hubs_among(40_000, others, seed=others)
    assert (g.nnz < 768 * np.diff(g.offsets).max()) == (slot == "sweep_hub")
    off, col = torch.from_numpy(g.offsets).to(DEV), torch.from_numpy(g.cols).to(DEV)
    c = gpu_lib.Context(0)
    c.set_profiling(True)
    got, st = c.lpa(off, col, mode=1, tolerance=0.0, max_iters=40, stats=True)
    lab = got.cpu().numpy()
    if st["changed"][-1] == 0:   # settled: every vertex holds its Eq. 2 label
        assert (O.sync_sweep(g, lab)[0] == lab).all()
    launches = {p["name"]: p["launches"] for p in c.profile()}
    assert ((lab >= 0) & (lab < g.n)).all() and launches[slot] > 0
