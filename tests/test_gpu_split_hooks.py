"""The split's offers by the separate kernels: rows around the borders between
a lane, half a warp, a listed warp and a block, dense and heavy ids side by
side, and communities whose sampled entries link nothing."""
import numpy as np
import pytest
import torch

import inputs as I
import oracle as O

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


def rows_of(lengths, pool, seed):
    """One vertex per length, side by side after a pool of sparse ones."""
    rng = np.random.default_rng(seed)
    u = [np.arange(pool - 1)] + [np.full(d, pool + k) for k, d in enumerate(lengths)]
    v = [np.arange(1, pool)] + [rng.choice(pool, d, replace=False) for d in lengths]
    return I.csr_from_pairs(pool + len(lengths), np.concatenate(u), np.concatenate(v), name="rows")


BORDERS = [d + 2 for d in (0, 1, 7, 8, 9, 15, 16, 17, 31, 32, 33, 63, 64, 65, 127, 2047, 2048, 2049, 4100)]
GRAPHS = {"borders": lambda: rows_of(BORDERS * 3, 5000, 1),
          "tiles of 64 steps": lambda: rows_of([66] * 32 + [64] * 32 + [66] * 31 + [68] * 33, 4001, 2),
          "heavy ids": lambda: rows_of([300] * 500, 3000, 3),
          "dense": lambda: I.sbm_planted(900, 300, 200.0, 30.0, seed=4)}


@pytest.mark.parametrize("name", sorted(GRAPHS))
def test_offers(gpu_lib, name):
    g = GRAPHS[name]()
    off, col = torch.from_numpy(g.offsets).to(DEV), torch.from_numpy(g.cols).to(DEV)
    c = gpu_lib.Context(0)
    c.set_hub_cluster(1 << 29)   # any setting of the caller keeps the separate kernels
    ids, rng = np.arange(g.n), np.random.default_rng(5)
    for lab in (ids % 2, ids % 7, rng.integers(0, 3, g.n), rng.integers(0, 100, g.n), ids // 50, g.n - ids // 300):
        lab = lab.astype(np.int32)
        want = O.split_bfs(g, lab)
        for _ in range(3):   # the order of the unions differs from call to call
            got, k = c.split(off, col, torch.from_numpy(lab).to(DEV))
            assert np.array_equal(got.cpu().numpy(), want) and k == (want == ids).sum()
