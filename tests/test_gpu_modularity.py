"""Modularity's per-block community table: one community, few, and more than
it holds, on graphs whose vertex count is no multiple of a warp."""
import numpy as np
import pytest
import torch

import inputs as I
import oracle as O

pytestmark = pytest.mark.gpu

DEV = "cuda:0"
GRAPHS = {"rmat13": lambda: I.rmat(13, 16, seed=3), "sbm": lambda: I.sbm_planted(3030, 30, 12.0, 2.0, seed=4),
          "path33": lambda: I.path(33)}


@pytest.mark.parametrize("weighted", [False, True])
@pytest.mark.parametrize("name", sorted(GRAPHS))
def test_community_counts(gpu_lib, name, weighted):
    g = GRAPHS[name]()
    if weighted:
        g = I.Graph(g.offsets, g.cols, I.symmetric_weights(g, 5, 1000))
    c = gpu_lib.Context(0)
    off, col = torch.from_numpy(g.offsets).to(DEV), torch.from_numpy(g.cols).to(DEV)
    w = torch.from_numpy(g.weights).to(DEV) if weighted else None
    rng = np.random.default_rng(2)
    for k in (1, 5, min(g.n, 300), g.n):
        lab = rng.integers(0, k, g.n).astype(np.int32)
        want = O.modularity(g, lab)
        got = c.modularity(off, col, torch.from_numpy(lab).to(DEV), w)
        # the sums are integers on both sides; forming Q rounds a few times, and Q may cancel to near 0
        assert abs(got - want) <= 1e-12, k
    one = np.full(g.n, g.n - 1, dtype=np.int32)
    one[g.n // 2] = g.n
    with pytest.raises(gpu_lib.GslError):
        c.modularity(off, col, torch.from_numpy(one).to(DEV), w)
