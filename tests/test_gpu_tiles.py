"""Rows of 1..33 entries at the borders of the short-row kernels (one lane, 8,
16 and 32 lanes per row, the first longer class), against the oracle."""
import numpy as np
import pytest
import torch

import inputs as I
import oracle as O

pytestmark = pytest.mark.gpu

DEV = "cuda:0"
BORDERS = (1, 2, 3, 4, 5, 8, 9, 16, 17, 31, 32, 33)


def border_graph(n, weighted, seed):
    """A vertex of every border degree several times over, joined to a pool of
    n ordinary vertices in shuffled order, with self-loops on some."""
    rng = np.random.default_rng(seed)
    edges, v = [], n
    for _ in range(7):
        for d in rng.permutation(BORDERS):
            edges += [(int(u), v) for u in rng.choice(n, d, replace=False)]
            v += 1
    edges += [(k, k) for k in range(0, v, 11)]
    perm = rng.permutation(v)
    edges = [(int(perm[a]), int(perm[b])) for a, b in edges]
    w = rng.integers(1, 4, len(edges)) if weighted else None
    return I.from_edges(v, edges, weights=w, name=f"borders-{n}")


@pytest.mark.parametrize("weighted", [False, True])
@pytest.mark.parametrize("n", [33, 64, 1000])
def test_border_degrees(gpu_lib, n, weighted):
    g = border_graph(n, weighted, seed=n)
    assert set(BORDERS) - {33} <= set(np.diff(g.offsets).tolist())
    c = gpu_lib.Context(0)
    off, col = torch.from_numpy(g.offsets).to(DEV), torch.from_numpy(g.cols).to(DEV)
    w = torch.from_numpy(g.weights).to(DEV) if weighted else None
    rng = np.random.default_rng(1)
    for k in (2, 9, g.n):
        prev = rng.integers(0, k, g.n).astype(np.int32)
        got = c.lpa(off, col, w, labels_init=torch.from_numpy(prev).to(DEV), tolerance=0.0, max_iters=1)
        assert np.array_equal(got.cpu().numpy(), O.sync_sweep(g, prev)[0]), k
    got, st = c.lpa(off, col, w, tolerance=0.0, max_iters=7, stats=True)
    want, t, dn = O.lpa_sync(g, 0.0, 7)
    assert st["iterations"] == t and st["changed"] == dn[:t].tolist()
    assert np.array_equal(got.cpu().numpy(), want)


def test_batch_replay_with_other_degrees_in_the_same_buffers(gpu_lib):
    """A captured batched loop launches the classes its graph had: the same
    buffers holding another graph of the same size must not reuse it."""
    ring = I.from_edges(40, [(k, (k + 1) % 40) for k in range(40)])          # degree 2 everywhere
    hub = I.from_edges(40, [(0, k) for k in range(1, 40)] + [(1, 2)])        # degrees 39, 2 and 1
    assert ring.nnz == hub.nnz
    off, col = torch.from_numpy(ring.offsets).to(DEV), torch.from_numpy(ring.cols).to(DEV)
    c = gpu_lib.Context(0)
    for g in (ring, hub, ring):
        off.copy_(torch.from_numpy(g.offsets))
        col.copy_(torch.from_numpy(g.cols))
        labels, sweeps = c.gsllpa_batch(off, col, [0, g.n])
        want, t, _ = O.gsl_lpa(g, 0.05, 20)
        assert np.array_equal(labels.cpu().numpy(), want) and sweeps.tolist() == [t]
