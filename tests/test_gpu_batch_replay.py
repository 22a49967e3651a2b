"""The captured batched loop is not replayed once a buffer it reads has moved."""
import numpy as np
import pytest
import torch

import oracle as O

from test_gpu_batch import mixed_graphs, pack

pytestmark = pytest.mark.gpu


def test_rejected_call_with_more_graphs_between_replays(gpu_lib):
    """A rejected batch of more graphs grows the per-graph arrays that the loop
    captured by the call before it reads."""
    graphs = mixed_graphs(3, seed=4)
    off, col, _, vptr = pack(graphs)
    off, col = torch.from_numpy(off).cuda(), torch.from_numpy(col).cuda()
    want = [O.gsl_lpa(g, 0.05, 20) for g in graphs]
    bad = off.clone()
    bad[-1] += 1   # the last offset is not the number of entries
    c = gpu_lib.Context(0)
    for more in (1 << 8, 1 << 12, 1 << 16):
        for rejected in (False, True):
            if rejected:
                with pytest.raises(gpu_lib.GslError) as e:
                    c.gsllpa_batch(bad, col, np.concatenate((vptr, np.full(more, vptr[-1]))))
                assert e.value.code == 1
            got, iters = c.gsllpa_batch(off, col, vptr)
            got = got.cpu().numpy()
            for k, (lab, sweeps, _) in enumerate(want):
                assert np.array_equal(got[vptr[k]:vptr[k + 1]], lab) and int(iters[k]) == sweeps
