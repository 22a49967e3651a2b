"""Rows around the borders of the counting kernels (a warp, 128 and 256
threads per row, labels in registers or in the scratch list), against the
oracle: labels all distinct, few, and one dominating."""
import numpy as np
import pytest
import torch

import inputs as I
import oracle as O

pytestmark = pytest.mark.gpu

DEV = "cuda:0"
BORDERS = (33, 63, 64, 65, 127, 128, 129, 255, 256, 257, 511, 512, 513, 1023, 1024, 1025, 2047, 2048, 2049, 4095, 4096,
           4097, 9000, 20011)


def hub_graph(seed=3, pool=21000):
    """One vertex of every border degree among a pool of sparse ones, ids shuffled."""
    rng = np.random.default_rng(seed)
    n = pool + len(BORDERS)
    u = [np.arange(pool - 1)]
    v = [np.arange(1, pool)]
    for k, d in enumerate(BORDERS):
        v.append(rng.choice(pool, d, replace=False))
        u.append(np.full(d, pool + k))
    return I.csr_from_pairs(n, np.concatenate(u), np.concatenate(v), perm=rng.permutation(n), name="border-hubs")


@pytest.fixture(scope="module")
def graph():
    return hub_graph()


@pytest.mark.parametrize("weighted", [False, True])
@pytest.mark.parametrize("tuning", [None, (64, 128), (1024, 1 << 20)])
def test_border_rows(gpu_lib, graph, weighted, tuning):
    g = graph
    assert set(BORDERS) <= set(np.diff(g.offsets).tolist())
    if weighted:
        g = I.Graph(g.offsets, g.cols, I.symmetric_weights(g, 4, 50))
    c = gpu_lib.Context(0)
    if tuning:
        c.set_tuning(*tuning)
    off, col = torch.from_numpy(g.offsets).to(DEV), torch.from_numpy(g.cols).to(DEV)
    w = torch.from_numpy(g.weights).to(DEV) if weighted else None
    rng = np.random.default_rng(5)
    flat = rng.permutation(g.n).astype(np.int32)                        # every label distinct
    few = rng.integers(0, 7, g.n).astype(np.int32)
    heavy = np.where(rng.random(g.n) < 0.4, 11, flat).astype(np.int32)  # one label of 40 %, no majority
    for prev in (flat, few, heavy):
        got = c.lpa(off, col, w, labels_init=torch.from_numpy(prev).to(DEV), tolerance=0.0, max_iters=1)
        assert np.array_equal(got.cpu().numpy(), O.sync_sweep(g, prev)[0])
    got, st = c.lpa(off, col, w, tolerance=0.0, max_iters=5, stats=True)
    want, t, dn = O.lpa_sync(g, 0.0, 5)
    assert st["iterations"] == t and st["changed"] == dn[:t].tolist()
    assert np.array_equal(got.cpu().numpy(), want)
