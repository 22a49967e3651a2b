"""The split over rows of every length its hooks treat alike, both in one launch
and by the separate kernels, with stray members in every community."""
import numpy as np
import pytest
import torch

import inputs as I
import oracle as O

from test_gpu_sketch import hub_graph

pytestmark = pytest.mark.gpu

DEV = "cuda:0"
GRAPHS = {"hubs": lambda: hub_graph(8), "sbm": lambda: I.sbm_planted(6000, 200, 14.0, 4.0, seed=2),
          "lattice": lambda: I.lattice_chains(60, 70, n_chains=500, seed=3)}


@pytest.mark.parametrize("name", sorted(GRAPHS))
def test_split_with_strays(gpu_lib, name):
    g = GRAPHS[name]()
    off, col = torch.from_numpy(g.offsets).to(DEV), torch.from_numpy(g.cols).to(DEV)
    rng = np.random.default_rng(6)
    one = gpu_lib.Context(0)
    several = gpu_lib.Context(0)
    several.set_hub_cluster(1 << 29)   # any setting of the caller keeps the separate kernels
    blocks = (np.arange(g.n) // 200 * 200).astype(np.int32)
    for lab in (rng.integers(0, 2, g.n), rng.integers(0, 40, g.n), np.zeros(g.n),
                np.where(rng.random(g.n) < 0.05, blocks[rng.integers(0, g.n, g.n)], blocks), np.full(g.n, -7)):
        lab = lab.astype(np.int32)
        want = O.split_bfs(g, lab)
        pieces = int((want == np.arange(g.n)).sum())
        for c in (one, several):
            got, k = c.split(off, col, torch.from_numpy(lab).to(DEV))
            assert np.array_equal(got.cpu().numpy(), want) and k == pieces
            got, k = c.split(off, col, torch.from_numpy(lab).to(DEV), renumber=True)
            assert k == pieces and np.array_equal(got.cpu().numpy(), np.unique(want, return_inverse=True)[1])


@pytest.mark.parametrize("n", [622_591, 622_593, 933_889, 1_245_184, 1_245_185, 1_400_003])
def test_split_of_long_paths(gpu_lib, n):
    """Communities of 2000 vertices on a path with cuts: runs of vertices a warp
    links, their last one ragged, and more runs than warps."""
    rng = np.random.default_rng(n)
    linked = rng.random(n - 1) < 0.995
    deg = np.zeros(n, np.int64)
    deg[:-1] += linked
    deg[1:] += linked
    off = np.concatenate(([0], np.cumsum(deg)))
    u = np.flatnonzero(linked)
    row, col = np.concatenate((u, u + 1)), np.concatenate((u + 1, u))
    col = col[np.lexsort((col, row))].astype(np.int32)
    lab = (np.arange(n) // 2000).astype(np.int32)
    first = np.concatenate(([True], ~linked | (lab[1:] != lab[:-1])))
    want = np.maximum.accumulate(np.where(first, np.arange(n), 0))
    got, k = gpu_lib.split(*(torch.from_numpy(x).to(DEV) for x in (off, col, lab)))
    assert k == first.sum() and np.array_equal(got.cpu().numpy(), want)
