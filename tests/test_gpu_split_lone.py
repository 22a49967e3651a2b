"""The split where communities hold vertices that no edge links: a lone vertex
keeps its label without its row being read."""
import numpy as np
import pytest
import torch

import inputs as I
import oracle as O

from test_gpu_sketch import hub_graph

pytestmark = pytest.mark.gpu

DEV = "cuda:0"
GRAPHS = {"hubs": lambda: hub_graph(12), "rmat14": lambda: I.rmat(14, 16, seed=6), "star": lambda: I.from_edges(5000, [(0, k) for k in range(1, 5000)])}


def contexts(gpu_lib):
    one, several = gpu_lib.Context(0), gpu_lib.Context(0)
    several.set_hub_cluster(1 << 29)   # any setting of the caller keeps the separate kernels
    return one, several


@pytest.mark.parametrize("name", sorted(GRAPHS))
def test_lone_vertices(gpu_lib, name):
    g = GRAPHS[name]()
    off, col = torch.from_numpy(g.offsets).to(DEV), torch.from_numpy(g.cols).to(DEV)
    ids, rng = np.arange(g.n), np.random.default_rng(2)
    for lab in (ids, ids // 2 * 2, rng.permutation(g.n), np.where(rng.random(g.n) < 0.5, ids, 0),
                np.where(rng.random(g.n) < 0.9, ids + g.n, ids // 8)):   # labels past n share slots
        lab = lab.astype(np.int32)
        want = O.split_bfs(g, lab)
        for c in contexts(gpu_lib):
            got, k = c.split(off, col, torch.from_numpy(lab).to(DEV))
            assert np.array_equal(got.cpu().numpy(), want) and k == (want == ids).sum()


def test_lone_vertices_read_no_more_than_the_sample(gpu_lib):
    """Every entry after a row's first eight is out of range, so that reading
    one would fail the call."""
    degree = np.tile([3, 9, 40, 700], 1000)
    degree[17] = 9000
    n = degree.size
    off = np.concatenate(([0], np.cumsum(degree))).astype(np.int64)
    at = np.arange(off[-1]) - np.repeat(off[:-1], degree)
    col = np.where(at < 8, (np.repeat(np.arange(n), degree) + 1 + at) % n, n).astype(np.int32)
    off, col = torch.from_numpy(off).to(DEV), torch.from_numpy(col).to(DEV)
    ids = torch.arange(n, dtype=torch.int32, device=DEV)
    for c in contexts(gpu_lib):
        got, k = c.split(off, col, ids)
        assert k == n and torch.equal(got, ids)
        with pytest.raises(gpu_lib.GslError):
            c.split(off, col, torch.div(ids, 200, rounding_mode="floor").to(torch.int32) % 3)
