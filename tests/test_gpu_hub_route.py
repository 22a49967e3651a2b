"""Rows past the block class, beside few and beside many other entries: by the
hub kernels in the first case, by the block kernel in the second."""
import numpy as np
import pytest
import torch

import inputs as I
import oracle as O

pytestmark = pytest.mark.gpu

DEV = "cuda:0"
LENGTH = 131_100   # of the class above 131,072


def hubs_among(others, seed):
    """Two rows of LENGTH entries and about `others` entries of random pairs."""
    rng = np.random.default_rng(seed)
    n = 140_000
    u = [rng.integers(0, n, others // 2)] + [np.full(LENGTH, n + k) for k in range(2)]
    v = [rng.integers(0, n, others // 2)] + [rng.choice(n, LENGTH, replace=False) for _ in range(2)]
    u, v = np.concatenate(u), np.concatenate(v)
    keep = u != v
    return I.csr_from_pairs(n + 2, u[keep], v[keep], perm=rng.permutation(n + 2), name="hubs-among")


@pytest.mark.parametrize("weighted", [False, True])
@pytest.mark.parametrize("others, slot, idle", [(0, "sweep_hub", "sweep_block"), (1_000_000, "sweep_hub", "sweep_block"),
                                                (17_000_000, "sweep_block", "sweep_hub")])
def test_route_and_labels(gpu_lib, others, slot, idle, weighted):
    g = hubs_among(others, seed=others + 1)
    d = np.diff(g.offsets)
    assert (d >= LENGTH).sum() == 2 and (g.nnz < 128 * d.max()) == (slot == "sweep_hub")
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
