"""Performance cases of the GSL-LPA library: what its users have it do.

Each case names a graph family, its sizes and the entry point it goes
through.  Graphs are made on the GPU from the seed alone (torch, no files);
families, densities and size ranges are those of the library's benchmark:
planted partitions (SBM), R-MAT with permuted ids (web / social shape), a
4-neighbour lattice with deleted edges, shortcuts and chains (road / k-mer
shape), batches of planted partitions, and a mixed stream of requests.

Asynchronous sweeps are not among the cases: their labels depend on the
schedule, so two runs on the same input differ.
"""
import math

import numpy as np
import torch

import paper_2403_01261_gb300 as gsl

TOLERANCE, MAX_ITERS = 0.05, 20


def listed():
    return [
        # the smallest ordinary call: the 10,000-vertex planted partition; launches and latency
        dict(name="sbm_10k", call="gsllpa", family="sbm", n=10_000, blocks=50, degree=18.0, ratio=8.0, weights="none"),
        # one mid-size community graph with an odd vertex count
        dict(name="sbm_300k", call="gsllpa", family="sbm", n=300_007, blocks=150, degree=24.0, ratio=6.0,
             weights="none"),
        # a request-sized skewed graph whose vertex count is not a power of two
        dict(name="rmat_1m", call="gsllpa", family="rmat", n=1_000_003, edge_factor=16, weights="none"),
        # the headline: R-MAT scale 25, edge factor 24
        dict(name="rmat_33m", call="gsllpa", family="rmat", n=1 << 25, edge_factor=24, weights="none"),
        # road / k-mer shape at full size: low degree, many sweeps
        dict(name="lattice_60m", call="gsllpa", family="lattice", side=6000, chains=2_000_000, weights="none"),
        # small-integer edge weights
        dict(name="rmat_4m_int32", call="gsllpa", family="rmat", n=1 << 22, edge_factor=24, weights="int32"),
        # the paper's precision: float32 weights, float64 sums
        dict(name="rmat_2m_float32", call="gsllpa", family="rmat", n=2_000_003, edge_factor=16, weights="float32"),
        # many uneven graphs in one call
        dict(name="batch_256", call="batch", family="sbm", graphs=256, n_lo=1_000, n_hi=200_000),
        # the split alone, renumbered, on communities with stray members
        dict(name="split_sbm_4m", call="split", family="sbm", n=4_000_037, blocks=2000, degree=24.0, ratio=6.0,
             renumber=True),
        # scoring a partition dominated by one community, as sweeps leave on a skewed graph
        dict(name="modularity_rmat_8m", call="modularity", family="rmat", n=1 << 23, edge_factor=24, weights="none"),
        # a graph in pinned host memory, labels back to the host
        dict(name="host_rmat_4m", call="host", family="rmat", n=1 << 22, edge_factor=24),
        # a burst of mixed requests through the server, 70 % planted partitions, 30 % R-MAT
        dict(name="served_40", call="served", requests=40, n_lo=1_000, n_hi=1 << 20),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_sbm(rng, n_lo, n_hi):
    n = _log_int(rng, n_lo, n_hi)
    return dict(family="sbm", n=n, blocks=rng.randint(5, 200), degree=round(rng.uniform(8.0, 40.0), 3),
                ratio=round(rng.uniform(3.0, 12.0), 3))


def _draw_rmat(rng, n_lo, n_hi):
    return dict(family="rmat", n=_log_int(rng, n_lo, n_hi), edge_factor=rng.randint(8, 24))


def draw(rng):
    call = rng.choice(["gsllpa"] * 6 + ["batch", "split", "split", "modularity", "modularity", "host", "served"])
    if call == "batch":
        return dict(call="batch", family="sbm", graphs=_log_int(rng, 8, 256), n_lo=1_000, n_hi=200_000)
    if call == "served":
        return dict(call="served", requests=rng.randint(8, 40), n_lo=1_000, n_hi=1 << rng.randint(16, 20))
    if call == "host":
        return dict(_draw_rmat(rng, 100_000, 1 << 22), call="host")
    family = rng.choice(["sbm", "rmat"] if call != "gsllpa" else ["sbm", "sbm", "rmat", "rmat", "rmat", "lattice"])
    if family == "lattice":
        side = _log_int(rng, 100, 5000)
        case = dict(family="lattice", side=side, chains=side * side // rng.randint(10, 30))
    elif family == "sbm":
        case = _draw_sbm(rng, 1_000, 1 << 22)
    else:
        case = _draw_rmat(rng, 1_000, 1 << (23 if call == "modularity" else 24))
    case["call"] = call
    if call == "split":
        case["renumber"] = rng.random() < 0.5
    else:
        case["weights"] = rng.choice(["none", "none", "int32", "float32"])
        largest = {"none": 1 << 24, "int32": 1 << 22, "float32": 1 << 21}[case["weights"]]
        if case.get("n", 0) > largest:
            case["n"] = _log_int(rng, 1_000, largest)
        if family == "lattice" and case["weights"] != "none" and case["side"] > 2000:
            case["side"], case["chains"] = 2000 + case["side"] % 97, case["chains"] // 7
    return case


# ------------------------------------------------------------------ graphs
def _device():
    return torch.device("cuda", torch.cuda.current_device())


def _csr(n, u, v):
    """Symmetric, deduplicated, loop-free CSR of the pairs (u[i], v[i]): rows sorted."""
    keep = u != v
    if not bool(keep.all()):
        u, v = u[keep], v[keep]
    keys = torch.unique(torch.cat((u * n + v, v * n + u)))
    starts = torch.arange(n + 1, dtype=torch.int64, device=keys.device) * n
    offsets = torch.searchsorted(keys, starts)
    cols = torch.empty(keys.numel(), dtype=torch.int32, device=keys.device)
    for a in range(0, keys.numel(), 1 << 28):
        b = min(a + (1 << 28), keys.numel())
        cols[a:b] = keys[a:b] % n
    return offsets, cols


def _below(gen, size, hi):
    """Uniform integers in [0, hi); hi a number or a tensor of `size` bounds."""
    return (torch.rand(size, dtype=torch.float64, device=gen.device, generator=gen) * hi).to(torch.int64)


def _rmat(gen, n, edge_factor):
    """R-MAT (0.57, 0.19, 0.19, 0.05) of the scale that holds n, ids permuted;
    of the permuted vertices the first n stay."""
    scale = max(1, (n - 1).bit_length())
    full = 1 << scale
    perm = torch.randperm(full, device=gen.device, generator=gen)
    us, vs = [], []
    total, step = edge_factor * full, 1 << 26
    for a in range(0, total, step):
        m = min(step, total - a)
        u = torch.zeros(m, dtype=torch.int32, device=gen.device)
        v = torch.zeros(m, dtype=torch.int32, device=gen.device)
        for _ in range(scale):
            r = torch.rand(m, device=gen.device, generator=gen)
            down = r >= 0.76
            u.mul_(2).add_(down)
            v.mul_(2).add_(((r >= 0.57) & ~down) | (r >= 0.95))
        u, v = perm[u.long()], perm[v.long()]
        if n < full:
            keep = (u < n) & (v < n)
            u, v = u[keep], v[keep]
        us.append(u)
        vs.append(v)
    return _csr(n, torch.cat(us), torch.cat(vs))


def _planted(gen, graphs):
    """Planted partitions packed side by side: graphs are (n, blocks, degree,
    ratio), blocks contiguous.  Returns offsets, cols, vptr and each vertex's
    block start."""
    dev = gen.device
    n = torch.tensor([g[0] for g in graphs], dtype=torch.int64, device=dev)
    nb = torch.tensor([min(g[1], g[0]) for g in graphs], dtype=torch.int64, device=dev)
    base = torch.cumsum(n, 0) - n
    us, vs = [], []
    for inside in (True, False):
        share = [g[3] / (g[3] + 1.0) if inside else 1.0 / (g[3] + 1.0) for g in graphs]
        m = torch.tensor([int(g[0] * g[2] * s / 2.0) for g, s in zip(graphs, share)], dtype=torch.int64, device=dev)
        k = torch.repeat_interleave(torch.arange(len(graphs), device=dev), m)
        nk, bk = n[k], base[k]
        u = _below(gen, k.numel(), nk)
        if inside:
            nbk = nb[k]
            b = ((u + 1) * nbk - 1) // nk          # the block [b n / nb, (b + 1) n / nb) that holds u
            lo = b * nk // nbk
            hi = (b + 1) * nk // nbk
            v = lo + _below(gen, k.numel(), hi - lo)
        else:
            v = _below(gen, k.numel(), nk)
        us.append(u + bk)
        vs.append(v + bk)
    total = int(n.sum())
    offsets, cols = _csr(total, torch.cat(us), torch.cat(vs))
    k = torch.repeat_interleave(torch.arange(len(graphs), device=dev), n)
    local = torch.arange(total, device=dev) - base[k]
    block = ((local + 1) * nb[k] - 1) // n[k]
    starts = base[k] + block * n[k] // nb[k]
    vptr = np.concatenate(([0], np.cumsum([g[0] for g in graphs]))).astype(np.int64)
    return offsets, cols, vptr, starts


def _lattice(gen, side, chains):
    """side x side 4-neighbour lattice, a quarter of its edges deleted, 0.5 %
    long shortcuts, and `chains` paths of 4..20 vertices after it."""
    dev = gen.device
    ids = torch.arange(side * side, dtype=torch.int64, device=dev).view(side, side)
    u = torch.cat((ids[:, :-1].reshape(-1), ids[:-1].reshape(-1)))
    v = torch.cat((ids[:, 1:].reshape(-1), ids[1:].reshape(-1)))
    keep = torch.rand(u.numel(), device=dev, generator=gen) >= 0.25
    u, v = u[keep], v[keep]
    extra = int(0.005 * u.numel())
    lens = 4 + torch.arange(chains, dtype=torch.int64, device=dev) * 7 % 17
    ends = torch.cumsum(lens, 0)
    m = int(ends[-1]) if chains else 0
    chain = torch.arange(m, dtype=torch.int64, device=dev)
    last = torch.zeros(m, dtype=torch.bool, device=dev)
    if chains:
        last[ends - 1] = True
    a = chain[~last] + side * side
    u = torch.cat((u, _below(gen, extra, side * side), a))
    v = torch.cat((v, _below(gen, extra, side * side), a + 1))
    return _csr(side * side + m, u, v)


def _weights(offsets, cols, seed, kind):
    """Symmetric edge weights from a hash of the edge's ends: int32 in 1..32,
    or float32 in (0.05, 1.05) with full mantissas."""
    n = offsets.numel() - 1
    out = torch.empty(cols.numel(), dtype=torch.int32 if kind == "int32" else torch.float32, device=cols.device)
    rows = torch.repeat_interleave(torch.arange(n, device=cols.device, dtype=torch.int32), offsets.diff())
    for a in range(0, cols.numel(), 1 << 27):
        i, j = rows[a:a + (1 << 27)].long(), cols[a:a + (1 << 27)].long()
        z = torch.minimum(i, j) * 0x1E3779B97F4A7C15 + torch.maximum(i, j) * 0x51B54A32D192ED03 + seed
        z = (z ^ ((z >> 30) & 0x3FFFFFFFF)) * 0x3F58476D1CE4E5B9
        z = z ^ ((z >> 27) & 0x1FFFFFFFFF)
        if kind == "int32":
            out[a:a + (1 << 27)] = 1 + ((z >> 20) & 31)
        else:
            out[a:a + (1 << 27)] = 0.05 + ((z >> 20) & 0xFFFFFF).float() / (1 << 24)
    return out


def _sbm_law(r, n):
    """Blocks, degree and intra:inter ratio of a planted partition of the benchmark's law."""
    return (n, 5 + int(r.integers(0, 196)), 8.0 + 32.0 * r.random(), 3.0 + 9.0 * r.random())


def _log_uniform(r, lo, hi):
    return int(round(math.exp(math.log(lo) + (math.log(hi) - math.log(lo)) * r.random())))


def _batch_graphs(case):
    # sizes from the case alone (stratified over the range, so that work() knows them): the seed draws the edges
    r = np.random.default_rng(case["graphs"])
    lo, hi, g = math.log(case["n_lo"]), math.log(case["n_hi"]), case["graphs"]
    sizes = [int(round(math.exp(lo + (hi - lo) * (k + r.random()) / g))) for k in range(g)]
    return [_sbm_law(r, sizes[k]) for k in r.permutation(g)]


def _served_requests(case):
    r = np.random.default_rng(case["requests"] * 64 + case["n_hi"].bit_length())
    reqs = []
    for k in range(case["requests"]):
        n = _log_uniform(r, case["n_lo"], case["n_hi"])
        if k % 10 in (2, 5, 8):
            reqs.append(("rmat", 1 << min(22, max(10, int(round(math.log2(n)))))))
        else:
            reqs.append(("sbm",) + _sbm_law(r, n))
    return reqs


def _partition(gen, case, offsets, starts):
    """Labels to split or score: the planted blocks with 3 % of the vertices
    moved to another one, or one community of nearly all linked vertices."""
    n = offsets.numel() - 1
    ids = torch.arange(n, device=offsets.device)
    roll = torch.rand(n, device=offsets.device, generator=gen)
    if case["family"] == "sbm":
        other = starts[_below(gen, n, n)]
        return torch.where(roll < 0.03, other, starts).to(torch.int32)
    big = (offsets.diff() > 0) & (roll < 0.98)
    first = int(torch.argmax(big.to(torch.uint8)))
    return torch.where(big, torch.full_like(ids, first), ids).to(torch.int32)


def _graph(case, gen):
    starts = None
    if case["family"] == "rmat":
        offsets, cols = _rmat(gen, case["n"], case["edge_factor"])
    elif case["family"] == "lattice":
        offsets, cols = _lattice(gen, case["side"], case["chains"])
    else:
        offsets, cols, _, starts = _planted(gen, [(case["n"], case["blocks"], case["degree"], case["ratio"])])
    return offsets, cols, starts


def _inputs(case, seed):
    gen = torch.Generator(device=_device())
    gen.manual_seed(seed)
    if case["call"] == "batch":
        offsets, cols, vptr, _ = _planted(gen, _batch_graphs(case))
        return dict(offsets=offsets, cols=cols, vptr=vptr)
    offsets, cols, starts = _graph(case, gen)
    s = dict(offsets=offsets, cols=cols, weights=None, labels=None)
    if case.get("weights", "none") != "none":
        s["weights"] = _weights(offsets, cols, seed, case["weights"])
    if case["call"] in ("split", "modularity"):
        s["labels"] = _partition(gen, case, offsets, starts)
    return s


_server = None


def _the_server():
    """One server for the process, as a serving program keeps it."""
    global _server
    if _server is None:
        _server = gsl.Server(slots=3, slot_vertices=1 << 23, slot_entries=1 << 27, tolerance=TOLERANCE,
                             max_iters=MAX_ITERS)
    return _server


def prepare(case, seed):
    if case["call"] == "served":
        gen = torch.Generator(device=_device())
        gen.manual_seed(seed)
        graphs = []
        for q in _served_requests(case):
            offsets, cols = _rmat(gen, q[1], 16) if q[0] == "rmat" else _planted(gen, [q[1:]])[:2]
            pinned = [torch.empty(t.numel(), dtype=t.dtype, pin_memory=True).copy_(t) for t in (offsets, cols)]
            graphs.append(pinned)
        return dict(case=case, graphs=graphs, server=_the_server())
    s = _inputs(case, seed)
    s["case"] = case
    if case["call"] == "host":
        for k in ("offsets", "cols"):
            s[k] = torch.empty(s[k].numel(), dtype=s[k].dtype, pin_memory=True).copy_(s[k])
        s["out"] = torch.empty(s["offsets"].numel() - 1, dtype=torch.int32, pin_memory=True)
    torch.cuda.empty_cache()   # what generating the graph took goes back before the library asks for memory
    return s


def run(state):
    case = state["case"]
    call = case["call"]
    if call == "served":
        server = state["server"]
        ids = [server.submit(o.numpy(), c.numpy()) for o, c in state["graphs"]]
        return {"labels": [server.wait(i) for i in ids]}
    off, col = state["offsets"], state["cols"]
    if call == "batch":
        labels, sweeps = _ctx().gsllpa_batch(off, col, state["vptr"], tolerance=TOLERANCE, max_iters=MAX_ITERS)
        return {"labels": labels, "sweeps": sweeps}
    if call == "split":
        labels, pieces = gsl.split(off, col, state["labels"], renumber=case["renumber"])
        return {"labels": labels, "pieces": pieces}
    if call == "modularity":
        if case["weights"] == "float32":
            return {"q": _ctx().modularity_f32(off, col, state["labels"], state["weights"])}
        return {"q": gsl.modularity(off, col, state["labels"], state["weights"])}
    if call == "host":
        labels, st = gsl.gsllpa_host(off, col, tolerance=TOLERANCE, max_iters=MAX_ITERS, out=state["out"], stats=True)
    elif case["weights"] == "float32":
        labels, st = _ctx().gsllpa_f32(off, col, state["weights"], tolerance=TOLERANCE, max_iters=MAX_ITERS,
                                       stats=True)
    else:
        labels, st = gsl.gsllpa(off, col, state["weights"], tolerance=TOLERANCE, max_iters=MAX_ITERS, stats=True)
    changed = np.zeros(MAX_ITERS, dtype=np.int64)
    changed[:st["iterations"]] = st["changed"]
    return {"labels": labels, "sweeps": st["iterations"], "communities": st["communities"], "changed": changed}


_context = None


def _ctx():
    """The context a program keeps for the calls that have no module-level form."""
    global _context
    if _context is None:
        _context = gsl.Context(torch.cuda.current_device())
    return _context


def _entries(family, **k):
    """Expected vertices and CSR entries of a graph."""
    if family == "sbm":
        return k["n"], k["n"] * k["degree"]
    if family == "lattice":
        side = k["side"]
        return side * side + 12.0 * k["chains"], 3.02 * side * side + 22.0 * k["chains"]
    scale = max(1, (k["n"] - 1).bit_length())
    kept = 1.0 - 0.9 * 2.0 ** (-0.18 * scale)   # what deduplication leaves
    return k["n"], 2.0 * k["edge_factor"] * (1 << scale) * kept * (k["n"] / (1 << scale)) ** 2


def work(case):
    """Offsets, columns, weights and labels read once, labels written once;
    one addition per entry."""
    if case["call"] == "batch":
        n, e = map(sum, zip(*(_entries("sbm", n=g[0], degree=g[2]) for g in _batch_graphs(case))))
    elif case["call"] == "served":
        n, e = map(sum, zip(*(_entries("rmat", n=q[1], edge_factor=16) if q[0] == "rmat" else
                              _entries("sbm", n=q[1], degree=q[3]) for q in _served_requests(case))))
    else:
        n, e = _entries(**case)
    b = 8.0 * n + 4.0 * e + (4.0 * e if case.get("weights", "none") != "none" else 0.0) + 4.0 * n
    if case["call"] == "split":
        b += 4.0 * n
    return {"bytes": b, "flops": e}


def exact(case, seed):
    """Modularity in 64 bits from its definition; labels and counts are whole numbers."""
    if case["call"] != "modularity":
        return None
    s = _inputs(case, seed)
    off, col, lab = s["offsets"], s["cols"], s["labels"].long()
    n = lab.numel()
    degree = torch.zeros(n, dtype=torch.float64, device=lab.device)
    within = torch.zeros((), dtype=torch.float64, device=lab.device)
    rows = torch.repeat_interleave(torch.arange(n, device=lab.device, dtype=torch.int32), off.diff())
    for a in range(0, col.numel(), 1 << 27):
        i, j = rows[a:a + (1 << 27)].long(), col[a:a + (1 << 27)].long()
        w = torch.ones_like(i, dtype=torch.float64) if s["weights"] is None else s["weights"][a:a + (1 << 27)].double()
        degree.index_add_(0, i, w)
        within += (w * (lab[i] == lab[j])).sum()
    total = degree.sum()
    community = torch.zeros_like(degree).index_add_(0, lab, degree)
    return {"q": float(within / total - (community / total).square().sum())}
