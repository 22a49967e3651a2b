"""Several threads with a context and a stream each, on graphs that are large
enough together for the separate kernels and small enough alone for the
one-launch path: every call gives the oracle's labels, whichever it took."""
import threading

import numpy as np
import pytest
import torch

import inputs as I
import oracle as O

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.mark.parametrize("threads", [2, 7])
def test_threads_on_mid_size_graphs(gpu_lib, threads):
    graphs = [I.sbm_planted(120_000 + 200 * k, 200, 12.0, 3.0, seed=k) for k in range(threads)]
    want = [O.gsl_lpa(g, 0.05, 20) for g in graphs]
    errors = []

    def work(k):
        try:
            c, s = gpu_lib.Context(0), torch.cuda.Stream()
            with torch.cuda.stream(s):
                off, col = torch.from_numpy(graphs[k].offsets).to(DEV), torch.from_numpy(graphs[k].cols).to(DEV)
                for _ in range(6):
                    got, st = c.gsllpa(off, col, stream=s, stats=True)
                    assert np.array_equal(got.cpu().numpy(), want[k][0])
                    assert st["iterations"] == want[k][1] and st["changed"] == want[k][2].tolist()
        except BaseException as e:  # noqa: BLE001 -- reported by the test's own thread
            errors.append(e)

    pool = [threading.Thread(target=work, args=(k,)) for k in range(threads)]
    for t in pool:
        t.start()
    for t in pool:
        t.join()
    assert not errors, errors[0]
    off, col = torch.from_numpy(graphs[0].offsets).to(DEV), torch.from_numpy(graphs[0].cols).to(DEV)
    before = gpu_lib.kernel_launches()
    gpu_lib.gsllpa(off, col)
    assert gpu_lib.kernel_launches() == before + 1   # alone again: one launch
