"""Rows of one warp with 64-bit sums, counted in shared counters that several
labels and lanes share: the counters are read only after every lane's adds."""
import numpy as np
import pytest
import torch

import inputs as I
import oracle as O

from test_gpu_wide import full_mantissa

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.mark.parametrize("degree", [40.0, 64.0, 100.0, 128.0, 200.0])
def test_warp_rows_with_close_sums(gpu_lib, degree):
    g = I.random_graph(1500, degree / 1500, seed=int(degree))
    d = np.diff(g.offsets)
    assert (d > 32).mean() > 0.8 and (d <= 256).all()   # one warp per row
    wf = full_mantissa(g, 3)   # full mantissas: 64-bit sums
    off, col, w = (torch.from_numpy(x).to(DEV) for x in (g.offsets, g.cols, wf))
    c = gpu_lib.Context(0)
    rng = np.random.default_rng(4)
    for labels in (2, 3, 17, 300, g.n):   # from hot counters to all labels distinct
        prev = rng.integers(0, labels, g.n).astype(np.int32)
        start, want = torch.from_numpy(prev).to(DEV), prev
        for sweeps in (1, 2):   # the first sweep has kernels of its own
            want = O.sync_sweep_f32(g, wf, want)[0]
            got = c.lpa_f32(off, col, w, labels_init=start, tolerance=0.0, max_iters=sweeps)
            assert np.array_equal(got.cpu().numpy(), want), (labels, sweeps)
