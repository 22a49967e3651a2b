"""The separate kernels of the degree classes on small graphs, which calls with
default settings run in one launch: short rows at the borders of the lane and
tile kernels, counting rows, the majority filter's two tests, and the parity
graphs, each against the oracle."""
import numpy as np
import pytest
import torch

import inputs as I
import oracle as O

from test_gpu_sketch import BORDERS as LONG_BORDERS
from test_gpu_sketch import hub_graph
from test_gpu_tiles import BORDERS as SHORT_BORDERS
from test_gpu_tiles import border_graph

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


def class_context(gpu_lib, majority=1):
    c = gpu_lib.Context(0)
    c.set_majority(majority)
    c.set_hub_cluster(1 << 29)   # any setting of the caller keeps the separate kernels
    return c


def on_device(g, w):
    return (torch.from_numpy(g.offsets).to(DEV), torch.from_numpy(g.cols).to(DEV),
            None if w is None else torch.from_numpy(w).to(DEV))


@pytest.mark.parametrize("weighted", [False, True])
@pytest.mark.parametrize("n", [33, 64, 1000])
def test_short_rows(gpu_lib, n, weighted):
    g = border_graph(n, weighted, seed=n)
    off, col, w = on_device(g, g.weights if weighted else None)
    c = class_context(gpu_lib)
    rng = np.random.default_rng(1)
    for k in (2, 9, g.n):
        prev = rng.integers(0, k, g.n).astype(np.int32)
        start, want = torch.from_numpy(prev).to(DEV), prev
        for sweeps in (1, 2):   # the first sweep has kernels of its own
            want = O.sync_sweep(g, want)[0]
            got = c.lpa(off, col, w, labels_init=start, tolerance=0.0, max_iters=sweeps)
            assert np.array_equal(got.cpu().numpy(), want), (k, sweeps)
    c.set_profiling(True)
    got, st = c.lpa(off, col, w, tolerance=0.0, max_iters=7, stats=True)
    want, t, dn = O.lpa_sync(g, 0.0, 7)
    assert st["iterations"] == t and st["changed"] == dn[:t].tolist()
    assert np.array_equal(got.cpu().numpy(), want)
    launched = {p["name"] for p in c.profile() if p["launches"] > 0}
    assert {"sweep_deg1_4", "sweep_deg5_8", "sweep_deg9_16", "sweep_deg17_32"} <= launched
    assert max(SHORT_BORDERS) <= 33


@pytest.mark.parametrize("weighted", [False, True])
def test_long_rows(gpu_lib, weighted):
    g = hub_graph()
    if weighted:
        g = I.Graph(g.offsets, g.cols, I.symmetric_weights(g, 4, 50))
    off, col, w = on_device(g, g.weights if weighted else None)
    c = class_context(gpu_lib)
    rng = np.random.default_rng(5)
    flat = rng.permutation(g.n).astype(np.int32)
    few = rng.integers(0, 7, g.n).astype(np.int32)
    heavy = np.where(rng.random(g.n) < 0.4, 11, flat).astype(np.int32)
    for prev in (flat, few, heavy):
        start, want = torch.from_numpy(prev).to(DEV), prev
        for sweeps in (1, 2):
            want = O.sync_sweep(g, want)[0]
            got = c.lpa(off, col, w, labels_init=start, tolerance=0.0, max_iters=sweeps)
            assert np.array_equal(got.cpu().numpy(), want), sweeps
    c.set_profiling(True)
    got, st = c.lpa(off, col, w, tolerance=0.0, max_iters=5, stats=True)
    want, t, dn = O.lpa_sync(g, 0.0, 5)
    assert st["changed"] == dn[:t].tolist() and np.array_equal(got.cpu().numpy(), want)
    launched = {p["name"] for p in c.profile() if p["launches"] > 0}
    assert {"sweep_warp_small", "sweep_warp_large", "sweep_block"} <= launched and max(LONG_BORDERS) > 4096


@pytest.mark.parametrize("weighted", [False, True])
@pytest.mark.parametrize("share", [0.2, 0.52, 0.7, 0.97])
@pytest.mark.parametrize("name", ["hubs", "rmat15"])
def test_filter_by_default(gpu_lib, name, share, weighted):
    g = hub_graph(5) if name == "hubs" else I.rmat(15, 24, seed=3)
    if weighted:
        g = I.Graph(g.offsets, g.cols, I.symmetric_weights(g, 4, 9))
    off, col, w = on_device(g, g.weights if weighted else None)
    rng = np.random.default_rng(int(100 * share))
    prev = np.where(rng.random(g.n) < share, g.n // 2, rng.integers(0, g.n, g.n)).astype(np.int32)
    start = torch.from_numpy(prev).to(DEV)
    lab, changed = prev, []
    for sweeps in (1, 2, 3, 4, 5):
        nxt = O.sync_sweep(g, lab)[0]
        changed.append(int((nxt != lab).sum()))
        lab = nxt
        got, st = class_context(gpu_lib).lpa(off, col, w, labels_init=start, tolerance=0.0, max_iters=sweeps, stats=True)
        assert st["changed"] == changed and np.array_equal(got.cpu().numpy(), lab), sweeps
        if changed[-1] == 0:
            break


PARITY = {"cliques": lambda: I.two_cliques_bridge(5), "path": lambda: I.path(9), "lattice": lambda: I.lattice_chains(30, 40, n_chains=50, seed=2),
          "random": lambda: I.random_graph(500, 0.006, seed=4), "rmat13": lambda: I.rmat(13, 16, seed=1),
          "sbm": lambda: I.sbm_planted(3000, 300, 60.0, 6.0, seed=5)}


@pytest.mark.parametrize("weighted", [False, True])
@pytest.mark.parametrize("name", sorted(PARITY))
def test_whole_calls(gpu_lib, name, weighted):
    g = PARITY[name]()
    if weighted:
        g = I.Graph(g.offsets, g.cols, I.symmetric_weights(g, 5, 40))
    off, col, w = on_device(g, g.weights if weighted else None)
    c = class_context(gpu_lib)
    before = gpu_lib.kernel_launches()
    got, st = c.gsllpa(off, col, w, stats=True)
    assert gpu_lib.kernel_launches() - before > 1
    want, t, dn = O.gsl_lpa(g, 0.05, 20)
    assert st["iterations"] == t and st["changed"] == dn.tolist()
    assert np.array_equal(got.cpu().numpy(), want)
