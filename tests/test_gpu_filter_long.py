"""The majority filter over rows that it reads in pieces, against the oracle
sweep by sweep: lengths at the borders of a piece, rows settled early, late
and not at all."""
import numpy as np
import pytest
import torch

import inputs as I
import oracle as O

pytestmark = pytest.mark.gpu

DEV = "cuda:0"
LONG, PIECE = 65536, 8192
LENGTHS = (LONG, LONG + 1, LONG + PIECE, LONG + PIECE + 1, 131072, 131073, 150001)


def long_rows(seed, pool=152_000):
    """One vertex of each length among a pool of sparse ones, ids shuffled."""
    rng = np.random.default_rng(seed)
    n = pool + len(LENGTHS)
    u, v = [np.arange(pool - 1)], [np.arange(1, pool)]
    for k, d in enumerate(LENGTHS):
        v.append(rng.choice(pool, d, replace=False))
        u.append(np.full(d, pool + k))
    return I.csr_from_pairs(n, np.concatenate(u), np.concatenate(v), perm=rng.permutation(n), name="long-rows")


@pytest.fixture(scope="module")
def graph():
    g = long_rows(3)
    assert set(LENGTHS) <= set(np.diff(g.offsets).tolist())
    return g


@pytest.mark.parametrize("weights", ["none", "int32", "float32"])
@pytest.mark.parametrize("share", [0.3, 0.502, 0.8])
def test_long_rows_sweep_by_sweep(gpu_lib, graph, share, weights):
    g = graph
    rng = np.random.default_rng(int(1000 * share))
    prev = np.where(rng.random(g.n) < share, g.n // 3, rng.integers(0, g.n, g.n)).astype(np.int32)
    off, col = torch.from_numpy(g.offsets).to(DEV), torch.from_numpy(g.cols).to(DEV)
    start = torch.from_numpy(prev).to(DEV)
    wi = I.symmetric_weights(g, 4, 9)
    wf = ((1 << 20) + wi.astype(np.float64) * 77777).astype(np.float32) / np.float32(1 << 22)   # 64-bit sums, exact
    h = I.Graph(g.offsets, g.cols, wi if weights == "int32" else None)
    w = {"none": None, "int32": torch.from_numpy(wi).to(DEV), "float32": torch.from_numpy(wf).to(DEV)}[weights]
    c = gpu_lib.Context(0)
    c.set_majority(2)
    call = c.lpa_f32 if weights == "float32" else c.lpa
    lab, changed = prev, []
    for sweeps in (1, 2, 3, 4):
        nxt = O.sync_sweep_f32(g, wf, lab)[0] if weights == "float32" else O.sync_sweep(h, lab)[0]
        changed.append(int((nxt != lab).sum()))
        lab = nxt
        got, st = call(off, col, w, labels_init=start, tolerance=0.0, max_iters=sweeps, stats=True)
        assert st["changed"] == changed[:st["iterations"]]
        assert np.array_equal(got.cpu().numpy(), lab), sweeps
        if changed[-1] == 0:
            break


@pytest.mark.parametrize("weighted", [False, True])
def test_long_rows_in_place_and_batched(gpu_lib, graph, weighted):
    g = I.Graph(graph.offsets, graph.cols, I.symmetric_weights(graph, 4, 9)) if weighted else graph
    off, col = torch.from_numpy(g.offsets).to(DEV), torch.from_numpy(g.cols).to(DEV)
    w = torch.from_numpy(g.weights).to(DEV) if weighted else None
    c = gpu_lib.Context(0)
    c.set_majority(2)
    want, t, _ = O.gsl_lpa(g, 0.0, 6)
    for _ in range(2):   # captured, then replayed
        got, iters = c.gsllpa_batch(off, col, [0, g.n], w, tolerance=0.0, max_iters=6)
        assert np.array_equal(got.cpu().numpy(), want) and iters.tolist() == [t]
    lab, st = c.lpa(off, col, w, mode=1, tolerance=0.0, max_iters=60, stats=True)
    lab = lab.cpu().numpy()
    if st["changed"][-1] == 0:   # settled: every vertex holds its Eq. 2 label
        assert (O.sync_sweep(g, lab)[0] == lab).all()
    assert ((lab >= 0) & (lab < g.n)).all()
