"""Float weights whose fixed-point form needs 64-bit row sums: every float64
partial sum is still exact, so the labels equal the oracle's bit for bit."""
import numpy as np
import pytest
import torch

import inputs as I
import oracle as O

from test_gpu_sketch import hub_graph
from test_gpu_tiles import border_graph

pytestmark = pytest.mark.gpu

DEV = "cuda:0"
GRAPHS = {"borders": lambda: border_graph(300, False, 2), "hubs": lambda: hub_graph(9),
          "rmat14": lambda: I.rmat(14, 16, seed=2), "sbm": lambda: I.sbm_planted(3000, 300, 60.0, 6.0, seed=5)}


def full_mantissa(g, seed):
    """Symmetric weights in [0.25, 1): multiples of 2^-26, row totals below 2^17."""
    src = np.repeat(np.arange(g.n), np.diff(g.offsets))
    key = np.minimum(src, g.cols).astype(np.int64) * g.n + np.maximum(src, g.cols)
    uniq, inv = np.unique(key, return_inverse=True)
    rng = np.random.default_rng(seed)
    return rng.uniform(0.25, 1.0, uniq.shape[0]).astype(np.float32)[inv]


@pytest.mark.parametrize("tuning", [None, (64, 128)])
@pytest.mark.parametrize("name", sorted(GRAPHS))
def test_wide_sums_equal_the_oracle(gpu_lib, name, tuning):
    g = GRAPHS[name]()
    wf = full_mantissa(g, 7)
    off, col = torch.from_numpy(g.offsets).to(DEV), torch.from_numpy(g.cols).to(DEV)
    w = torch.from_numpy(wf).to(DEV)
    rng = np.random.default_rng(3)
    for fixed in (1, 0):
        c = gpu_lib.Context(0)
        c.set_f32_fixed(fixed)
        if tuning:
            c.set_tuning(*tuning)
        for k in (5, g.n):
            prev = rng.integers(0, k, g.n).astype(np.int32)
            got = c.lpa_f32(off, col, w, labels_init=torch.from_numpy(prev).to(DEV), tolerance=0.0, max_iters=1)
            assert np.array_equal(got.cpu().numpy(), O.sync_sweep_f32(g, wf, prev)[0]), (fixed, k)
        got, st = c.lpa_f32(off, col, w, tolerance=0.0, max_iters=6, stats=True)
        want, t, dn = O.lpa_sync_f32(g, wf, 0.0, 6)
        assert st["iterations"] == t and st["changed"] == dn[:t].tolist()
        assert np.array_equal(got.cpu().numpy(), want), fixed
        lab = c.gsllpa_f32(off, col, w, mode=1).cpu().numpy()
        assert (lab <= np.arange(g.n)).all() and O.disconnected(g, lab)[0] == 0
