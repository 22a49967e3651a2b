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
