"""A call that the class kernels can run in the context's present memory is
not refused because the one-launch path's label lists do not fit."""
import numpy as np
import torch
import pytest

import inputs as I
import oracle as O

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


def test_no_room_for_label_lists(gpu_lib):
    g = I.sbm_planted(3000, 150, 20.0, 2.0, seed=7)
    off, col = torch.from_numpy(g.offsets).to(DEV), torch.from_numpy(g.cols).to(DEV)
    out = torch.empty(g.n, dtype=torch.int32, device=DEV)
    want = O.gsl_lpa(g, 0.05, 20)[0]
    c = gpu_lib.Context(0)
    c.set_hub_cluster(1 << 29)   # the class kernels: their scratch and code are in place after this
    c.gsllpa(off, col, out=out)
    c.set_hub_cluster(1 << 30)   # the default again
    filler = []
    try:
        for chunk in (1 << 30, 1 << 26, 1 << 22, 1 << 21):
            while torch.cuda.mem_get_info()[0] > chunk + (6 << 20):
                free = torch.cuda.mem_get_info()[0] - (6 << 20)
                filler.append(torch.empty(free // chunk * chunk, dtype=torch.uint8, device=DEV))
        assert torch.cuda.mem_get_info()[0] < 12 << 20
        out.zero_()
        c.gsllpa(off, col, out=out)
    finally:
        filler.clear()
        torch.cuda.empty_cache()
    assert np.array_equal(out.cpu().numpy(), want)
    before = gpu_lib.kernel_launches()
    c.gsllpa(off, col, out=out)
    assert gpu_lib.kernel_launches() == before + 1   # with memory back, one launch
    assert np.array_equal(out.cpu().numpy(), want)
