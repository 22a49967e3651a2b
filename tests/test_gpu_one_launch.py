"""The one-launch path of small graphs, against the oracle: few rows that hold
many entries, and what it leaves to the class kernels."""
import numpy as np
import pytest
import torch

import inputs as I
import oracle as O

from test_gpu_split_hooks import rows_of

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


def launched(gpu_lib, call):
    before = gpu_lib.kernel_launches()
    out = call()
    return out, gpu_lib.kernel_launches() - before


@pytest.mark.parametrize("weighted", [False, True])
@pytest.mark.parametrize("n", [64, 129, 500, 1200])
def test_few_dense_rows(gpu_lib, n, weighted):
    g = I.random_graph(n, 0.97, seed=n)
    if weighted:
        g = I.Graph(g.offsets, g.cols, I.symmetric_weights(g, 4, 30))
    off, col = torch.from_numpy(g.offsets).to(DEV), torch.from_numpy(g.cols).to(DEV)
    w = torch.from_numpy(g.weights).to(DEV) if weighted else None
    c = gpu_lib.Context(0)
    rng = np.random.default_rng(3)
    for labels in (2, 5, n):
        prev = rng.integers(0, labels, n).astype(np.int32)
        got, launches = launched(gpu_lib, lambda: c.lpa(off, col, w, labels_init=torch.from_numpy(prev).to(DEV),
                                                        tolerance=0.0, max_iters=1))
        assert launches == 1 and np.array_equal(got.cpu().numpy(), O.sync_sweep(g, prev)[0])
    (got, st), launches = launched(gpu_lib, lambda: c.gsllpa(off, col, w, tolerance=0.0, max_iters=9, stats=True))
    want, t, dn = O.gsl_lpa(g, 0.0, 9)
    assert launches == 1 and st["iterations"] == t and st["changed"] == dn[:t].tolist()
    assert np.array_equal(got.cpu().numpy(), want)


# rows of more than 4096 entries with 3 * 2^19 entries in all are the most it takes
@pytest.mark.parametrize("rows, one", [([8000] * 196 + [4864], True), ([8000] * 196 + [4865], False),
                                       ([4097] * 383, True), ([4097] * 384, False), ([32768] * 3, True),
                                       ([32769] + [5000] * 3, False)])
def test_many_huge_rows(gpu_lib, rows, one):
    g = rows_of(rows, 33_000, len(rows))
    off, col = torch.from_numpy(g.offsets).to(DEV), torch.from_numpy(g.cols).to(DEV)
    c = gpu_lib.Context(0)
    (got, st), launches = launched(gpu_lib, lambda: c.gsllpa(off, col, tolerance=0.0, max_iters=4, stats=True))
    want, t, dn = O.gsl_lpa(g, 0.0, 4)
    assert (launches == 1) == one and st["iterations"] == t and st["changed"] == dn[:t].tolist()
    assert np.array_equal(got.cpu().numpy(), want)
    lab = (np.arange(g.n) % 3).astype(np.int32)
    (got, k), launches = launched(gpu_lib, lambda: c.split(off, col, torch.from_numpy(lab).to(DEV)))
    want = O.split_bfs(g, lab)
    assert (launches == 1) == one and np.array_equal(got.cpu().numpy(), want)


def ring(n):
    u = np.arange(n)
    return I.csr_from_pairs(n, u, (u + 1) % n, name="ring")


def circulant(n, half, extra=0):
    u = np.repeat(np.arange(n), half)
    v = (u + np.tile(np.arange(1, half + 1), n)) % n
    more = np.arange(extra)
    return I.csr_from_pairs(n, np.concatenate((u, more)), np.concatenate((v, more + n // 2)), name="circulant")


# 2^19 vertices, 2^23 entries and 64 sweeps are the most it takes
@pytest.mark.parametrize("graph, sweeps, one", [
    (lambda: ring(1 << 19), 5, True), (lambda: ring((1 << 19) + 1), 5, False),
    (lambda: circulant(1 << 17, 32), 3, True), (lambda: circulant(1 << 17, 32, extra=1), 3, False),
    (lambda: ring(1000), 64, True), (lambda: ring(1000), 65, False)])
def test_limits(gpu_lib, graph, sweeps, one):
    g = graph()
    off, col = torch.from_numpy(g.offsets).to(DEV), torch.from_numpy(g.cols).to(DEV)
    c = gpu_lib.Context(0)
    (got, st), launches = launched(gpu_lib, lambda: c.gsllpa(off, col, tolerance=0.0, max_iters=sweeps, stats=True))
    want, t, dn = O.gsl_lpa(g, 0.0, sweeps)
    assert (launches == 1) == one and st["iterations"] == t and st["changed"] == dn[:len(st["changed"])].tolist()
    assert np.array_equal(got.cpu().numpy(), want)


def test_split_of_long_rows_side_by_side(gpu_lib):
    """Rows around the border between a warp and a block, and up to the longest
    the launch takes, in communities that their sampled entries leave apart."""
    g = rows_of([255, 256, 257, 258] * 40 + [300, 4096, 4097, 20_000, 32_768], 33_000, 9)
    off, col = torch.from_numpy(g.offsets).to(DEV), torch.from_numpy(g.cols).to(DEV)
    c = gpu_lib.Context(0)
    ids, rng = np.arange(g.n), np.random.default_rng(5)
    for lab in (ids, ids % 2, rng.integers(0, 40, g.n), rng.integers(0, 2000, g.n), ids // 700, np.zeros(g.n)):
        lab = lab.astype(np.int32)
        want = O.split_bfs(g, lab)
        for _ in range(3):   # the order of the unions differs from call to call
            (got, k), launches = launched(gpu_lib, lambda: c.split(off, col, torch.from_numpy(lab).to(DEV)))
            assert launches == 1 and np.array_equal(got.cpu().numpy(), want) and k == (want == ids).sum()
