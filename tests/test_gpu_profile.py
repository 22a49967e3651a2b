"""The profiler's books: kernels launched, and the bytes of the majority
filter's two tests and of the rows the block kernel takes over."""
import numpy as np
import pytest
import torch

import inputs as I

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


def profiled(gpu_lib, g, call, settings=()):
    off, col = torch.from_numpy(g.offsets).to(DEV), torch.from_numpy(g.cols).to(DEV)
    c = gpu_lib.Context(0)
    for name, args in settings:
        getattr(c, name)(*args)
    call(c, off, col)
    c.set_profiling(True)
    before = gpu_lib.kernel_launches()
    out = call(c, off, col)
    launches = gpu_lib.kernel_launches() - before
    return out, launches, {p["name"]: p for p in c.profile()}


GRAPHS = {"rmat14": lambda: I.rmat(14, 24, seed=3), "path": lambda: I.path(500),
          "sbm": lambda: I.sbm_planted(3000, 300, 60.0, 6.0, seed=5)}


@pytest.mark.parametrize("what", ["modularity", "gsllpa", "split"])
@pytest.mark.parametrize("name", sorted(GRAPHS))
def test_slots_count_every_kernel(gpu_lib, name, what):
    g = GRAPHS[name]()
    lab = torch.arange(g.n, dtype=torch.int32, device=DEV) % 7
    call = {"modularity": lambda c, off, col: c.modularity(off, col, lab),
            "gsllpa": lambda c, off, col: c.gsllpa(off, col, tolerance=0.0, max_iters=6),
            "split": lambda c, off, col: c.split(off, col, lab, renumber=True)}[what]
    _, launches, prof = profiled(gpu_lib, g, call)
    assert sum(p["kernels"] for p in prof.values()) == launches > 0


def test_filter_bytes(gpu_lib):
    """Of two sweeps the filter runs in the second: on labels of which one
    dominates the graph, and on blocks whose vertices mostly keep their own."""
    rng = np.random.default_rng(1)
    skewed, blocks = I.rmat(14, 24, seed=3), I.sbm_planted(3000, 600, 400.0, 40.0, seed=2)
    for g, common, share, bits in ((skewed, np.full(skewed.n, 3), 0.9, True),
                                   (blocks, np.arange(blocks.n) // 600 * 600, 0.8, False)):
        prev = np.where(rng.random(g.n) < share, common, rng.integers(0, g.n, g.n)).astype(np.int32)
        start = torch.from_numpy(prev).to(DEV)
        _, _, prof = profiled(gpu_lib, g, lambda c, off, col: c.lpa(off, col, labels_init=start, tolerance=0.0, max_iters=2),
                              [("set_majority", (2,))])
        p = prof["majority_filter"]
        assert p["entries"] > 0
        assert p["bytes"] == 20.0 * p["vertices"] + (4.125 * p["entries"] + 4.125 * g.n if bits else 8.0 * p["entries"])


def test_block_kernel_books_the_hubs_it_sweeps(gpu_lib):
    from test_gpu_hub_route import hubs_among
    g = hubs_among(131_100, 68_000_000, 5)   # two rows of class 9, hidden by the rest
    _, _, prof = profiled(gpu_lib, g, lambda c, off, col: c.lpa(off, col, tolerance=0.0, max_iters=2))
    assert prof["sweep_hub"]["entries"] == 0 and prof["sweep_block"]["entries"] >= 2 * 131_100
