"""Modularity over rows that the blocks share in pieces: lengths at the borders
of a piece, alone in their graph and beside many other entries."""
import numpy as np
import pytest
import torch

import inputs as I
import oracle as O

from test_gpu_filter_long import LENGTHS, long_rows

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


def among_many():
    rng = np.random.default_rng(8)
    n, extra = 152_000, 19_500_000   # the longest row is less than 1/256 of the entries
    u = [rng.integers(0, n, extra)] + [np.full(d, n + k) for k, d in enumerate(LENGTHS)]
    v = [rng.integers(0, n, extra)] + [rng.choice(n, d, replace=False) for d in LENGTHS]
    u, v = np.concatenate(u), np.concatenate(v)
    return I.csr_from_pairs(n + len(LENGTHS), u[u != v], v[u != v], name="among-many")


GRAPHS = {"alone": (lambda: long_rows(5), True), "among many": (among_many, False)}


@pytest.mark.parametrize("weighted", [False, True])
@pytest.mark.parametrize("name", sorted(GRAPHS))
def test_long_rows(gpu_lib, name, weighted):
    make, pieces = GRAPHS[name]
    g = make()
    d = np.diff(g.offsets)
    assert (d > 65536).sum() >= 6 and (g.nnz < 256 * d.max()) == pieces
    if weighted:
        g = I.Graph(g.offsets, g.cols, I.symmetric_weights(g, 5, 1000))
    c = gpu_lib.Context(0)
    off, col = torch.from_numpy(g.offsets).to(DEV), torch.from_numpy(g.cols).to(DEV)
    w = torch.from_numpy(g.weights).to(DEV) if weighted else None
    rng = np.random.default_rng(2)
    for k in (1, 5, g.n):
        lab = rng.integers(0, k, g.n).astype(np.int32)
        # the sums are integers on both sides; forming Q rounds a few times, and Q may cancel to near 0
        assert abs(c.modularity(off, col, torch.from_numpy(lab).to(DEV), w) - O.modularity(g, lab)) <= 1e-12, k
