"""The autotuner times what the call will run: the one-launch path of small
graphs is a candidate, and settings that run the same kernels are timed once."""
import numpy as np
import pytest
import torch

import inputs as I
import oracle as O

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


def dev(g):
    return torch.from_numpy(g.offsets).to(DEV), torch.from_numpy(g.cols).to(DEV)


def launches_of(gpu_lib, call):
    before = gpu_lib.kernel_launches()
    call()
    return gpu_lib.kernel_launches() - before


def circulant(n, d):
    u = np.repeat(np.arange(n), d // 2)
    return I.csr_from_pairs(n, u, (u + np.tile(np.arange(1, d // 2 + 1), n)) % n, name="circulant")


@pytest.mark.parametrize("name", ["rmat15", "sbm"])
def test_small_graphs_keep_the_one_launch_path(gpu_lib, name):
    g = I.rmat(15, 16, seed=4) if name == "rmat15" else I.sbm_planted(4000, 200, 20.0, 2.0, seed=3)
    off, col = dev(g)
    want = O.gsl_lpa(g, 0.05, 20)[0]
    c = gpu_lib.Context(0)
    for setting in (None, lambda: c.set_majority(0), lambda: c.set_tuning(128, 4096)):
        if setting:
            setting()
            assert launches_of(gpu_lib, lambda: c.gsllpa(off, col)) > 1
        r = c.autotune(off, col, sweeps=6)
        assert r["best_ms"] <= r["entry_ms"] or setting
        assert launches_of(gpu_lib, lambda: c.gsllpa(off, col)) == 1   # several times faster than the class kernels
        assert np.array_equal(c.gsllpa(off, col).cpu().numpy(), want)
    c.set_retry_bounds(1 << 20, 0)   # lowered bounds act on the class kernels
    c.autotune(off, col, sweeps=6)
    assert launches_of(gpu_lib, lambda: c.gsllpa(off, col)) > 1
    c.set_retry_bounds(0, 0)
    assert np.array_equal(c.gsllpa(off, col).cpu().numpy(), want)


def test_tuning_on_a_large_graph_leaves_small_ones(gpu_lib):
    big, small = I.rmat(19, 16, seed=2), I.sbm_planted(4000, 200, 20.0, 2.0, seed=3)   # past 2^23 entries; small
    assert big.nnz > 1 << 23
    c = gpu_lib.Context(0)
    off, col = dev(small)
    c.autotune(*dev(big), sweeps=3)
    assert launches_of(gpu_lib, lambda: c.gsllpa(off, col)) == 1
    c.autotune_batch(off, col, [0, small.n])
    assert launches_of(gpu_lib, lambda: c.gsllpa(off, col)) == 1
    assert np.array_equal(c.gsllpa(off, col).cpu().numpy(), O.gsl_lpa(small, 0.05, 20)[0])


# two-phase mode 2 x majority 3 (rows above 32 only) x binnings; block shapes
# only with rows for the hub kernels; 1 for the one-launch path
@pytest.mark.parametrize("degree, settings", [(16, 2), (60, 6), (200, 2 * 6), (2000, 6)])
def test_candidates(gpu_lib, degree, settings):
    g = circulant(2 * degree + 1, degree)
    off, col = dev(g)
    c = gpu_lib.Context(0)
    assert c.autotune(off, col, sweeps=1)["candidates"] == settings + 1
    _, r = c.autotune_batch(off, col, [0, g.n], max_iters=2)
    assert r["candidates"] == settings // 2
