"""The majority filter's two tests (own label, one label dominating the whole
graph) over every row class, against the oracle sweep by sweep."""
import numpy as np
import pytest
import torch

import inputs as I
import oracle as O

from test_gpu_sketch import hub_graph

pytestmark = pytest.mark.gpu

DEV = "cuda:0"
GRAPHS = {"hubs": lambda: hub_graph(5), "rmat15": lambda: I.rmat(15, 24, seed=3)}


@pytest.mark.parametrize("weights", ["none", "int32", "float32"])
@pytest.mark.parametrize("share", [0.2, 0.52, 0.7, 0.97])
@pytest.mark.parametrize("name", sorted(GRAPHS))
def test_dominating_label(gpu_lib, name, share, weights):
    g = GRAPHS[name]()
    rng = np.random.default_rng(int(100 * share))
    prev = np.where(rng.random(g.n) < share, g.n // 2, rng.integers(0, g.n, g.n)).astype(np.int32)
    off, col = torch.from_numpy(g.offsets).to(DEV), torch.from_numpy(g.cols).to(DEV)
    start = torch.from_numpy(prev).to(DEV)
    wi = I.symmetric_weights(g, 4, 9)
    wf = ((1 << 20) + wi.astype(np.float64) * 77777).astype(np.float32) / np.float32(1 << 22)   # 64-bit sums, exact
    for majority in (1, 2):
        c = gpu_lib.Context(0)
        c.set_majority(majority)
        for iters in (2, 3, 4):
            if weights == "float32":
                w = torch.from_numpy(wf).to(DEV)
                got, st = c.lpa_f32(off, col, w, labels_init=start, tolerance=0.0, max_iters=iters, stats=True)
            else:
                w = torch.from_numpy(wi).to(DEV) if weights == "int32" else None
                got, st = c.lpa(off, col, w, labels_init=start, tolerance=0.0, max_iters=iters, stats=True)
            lab, changed = prev, []
            h = I.Graph(g.offsets, g.cols, wi if weights == "int32" else None)
            for _ in range(st["iterations"]):
                nxt = O.sync_sweep_f32(g, wf, lab)[0] if weights == "float32" else O.sync_sweep(h, lab)[0]
                changed.append(int((nxt != lab).sum()))
                lab = nxt
            assert st["changed"] == changed
            assert np.array_equal(got.cpu().numpy(), lab), (majority, iters)
