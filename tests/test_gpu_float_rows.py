"""The float64 kernels with more long rows than blocks, of uneven lengths."""
import numpy as np
import pytest
import torch

import oracle as O

from fixtures import float_weights
from test_gpu_split_hooks import rows_of

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.mark.parametrize("majority", [1, 2])
def test_uneven_long_rows(gpu_lib, majority):
    g = rows_of([300] * 400 + [1025] * 1400 + [6000] * 20 + [1100, 20_000, 1100], 21_000, 6)
    w = float_weights(g, 3)   # multiples of 1/8: sums exact in any order
    off, col, wf = (torch.from_numpy(x).to(DEV) for x in (g.offsets, g.cols, w))
    c = gpu_lib.Context(0)
    c.set_f32_fixed(0)
    c.set_majority(majority)
    got, st = c.lpa_f32(off, col, wf, tolerance=0.0, max_iters=5, stats=True)
    want, t, dn = O.lpa_sync_f32(g, w, 0.0, 5)
    assert st["iterations"] == t and st["changed"] == dn[:t].tolist()
    assert np.array_equal(got.cpu().numpy(), want)
    lab = c.gsllpa_f32(off, col, wf, mode=1, max_iters=6).cpu().numpy()
    assert (lab <= np.arange(g.n)).all() and O.disconnected(g, lab)[0] == 0
