"""The work a user of this library has it do, as measurable cases.

A case is one call (or the sequence of calls that belongs together) through
the package's public functions on a synthetic graph: a sampler batch, a run of
Alg. 1 in all-nodes or top-k mode, a batch of graphs, a burst of served jobs,
the load of a graph, or a load with the run that follows it.  The graph
families and their sizes are those of the repository's benchmark: Erdos-Renyi
of mean degree 8, Chung-Lu with exponent 2.5 and mean degree 16, Barabasi-
Albert with 4 to 16 edges per node, and directed R-MAT with edge factor 16.
The graphs are drawn on the GPU with torch, from the seed alone.
"""

from __future__ import annotations

import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_1604_08553_gb300 import kadabra

DEVICE = "cuda"
DELTA = 0.1


# ---------------------------------------------------------------- cases
def listed():
    return [
        # the smallest job: a run on a graph of two thousand nodes, whose time
        # is launches, stop tests and the latency of single samples
        dict(name="er_2k_run", call="run", family="er", n=2000, lam=0.01, k=0, interval=1000),
        # an ordinary job with every default of kadabra_run: a few hundred
        # thousand nodes, a stop test after every thousand samples
        dict(name="ba_300k_run", call="run", family="ba", n=299993, attach=7, lam=0.01, k=0, interval=1000),
        # the benchmark's run: a power-law graph that fits in the L2
        dict(name="chung_lu_1m_run", call="run", family="chung_lu", n=1000000, lam=0.005, k=0, interval=65536),
        # its sampler alone, as a program calls it that keeps its own schedule
        dict(name="chung_lu_1m_sample", call="sample", family="chung_lu", n=1000000, samples=65536),
        # the same job from the host and back: upload, checks, run, results
        dict(name="chung_lu_1m_load_run", call="load_run", family="chung_lu", n=1000000, lam=0.005, k=0,
             interval=65536),
        # a graph without hubs, the slowest kind of served job: searches of
        # thousands of nodes per side
        dict(name="er_3m_run", call="run", family="er", n=3400000, lam=0.01, k=0, interval=0),
        # a directed graph beyond the L2
        dict(name="rmat_22_sample", call="sample", family="rmat", scale=22, samples=65536),
        # top-k mode on the largest graph the benchmark has
        dict(name="rmat_24_topk_run", call="run", family="rmat", scale=24, lam=0.0025, k=10, interval=65536),
        # that graph's load from device memory: CSR checks and the VD bound
        dict(name="rmat_24_load", call="load", family="rmat", scale=24),
        # many graphs of uneven sizes run together
        dict(name="ba_64_batch", call="batch", family="ba", graphs=64, n_lo=10000, n_hi=2000000, lam=0.01),
        # a burst of mixed jobs (both modes, three families) sent to the server
        dict(name="serve_24_jobs", call="serve", graphs=6, n_lo=2000, n_hi=1000000, jobs=24),
        # the stop test alone, for counts that were added up elsewhere
        dict(name="stop_test_1m", call="check", n=1000003),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["run", "run", "run", "sample", "sample", "load", "load_run", "batch", "serve", "check"])
    if call == "check":
        return dict(call=call, n=_log_uniform(rng, 1000, 4000000))
    if call == "batch":
        return dict(call=call, family="ba", graphs=rng.randint(2, 48), n_lo=10000,
                    n_hi=_log_uniform(rng, 20000, 1500000), lam=rng.choice([0.02, 0.01]))
    if call == "serve":
        return dict(call=call, graphs=rng.randint(2, 6), n_lo=2000, n_hi=_log_uniform(rng, 5000, 800000),
                    jobs=rng.randint(4, 20))
    family = rng.choice(["er", "chung_lu", "ba", "rmat"])
    case = dict(call=call, family=family)
    if family == "rmat":
        case["scale"] = rng.randint(14, 22)
    else:
        case["n"] = _log_uniform(rng, 2000, 2000000)
        if family == "ba":
            case["attach"] = rng.randint(4, 16)
    if call == "sample":
        case["samples"] = _log_uniform(rng, 500, 65536)
    elif call != "load":
        case["lam"] = rng.choice([0.02, 0.01, 0.005])
        case["k"] = rng.choice([0, 0, 10, 50])
        case["interval"] = rng.choice([1000, 0, 4096, 65536])
    return case


# ---------------------------------------------------------------- graphs
def _generator(seed):
    return torch.Generator(device=DEVICE).manual_seed(seed)


def _csr(n, src, dst):
    """Sorted, duplicate-free rows without self-loops, from arcs (src, dst)."""
    keep = src != dst
    key = torch.unique_consecutive(torch.sort(src[keep] * n + dst[keep]).values)
    bounds = torch.arange(n + 1, device=DEVICE, dtype=torch.int64) * n
    return torch.searchsorted(key, bounds).to(torch.int32), (key % n).to(torch.int32)


def _connect(n, a, b, g):
    """The edges (a, b) with one more for every component but the largest,
    from its lowest node to a random node of the largest (components by
    minimum labels over neighbours, with pointer jumping)."""
    src, dst = torch.cat([a, b]), torch.cat([b, a])
    label = torch.arange(n, device=DEVICE)
    while True:
        new = label.scatter_reduce(0, src, label[dst], "amin")
        new = new[new]
        if torch.equal(new, label):
            break
        label = new
    size = torch.bincount(label, minlength=n)
    main = size.argmax()
    inside = torch.nonzero(label == main)[:, 0]
    size[main] = 0
    lone = torch.nonzero(size)[:, 0]
    far = inside[torch.randint(0, inside.numel(), (lone.numel(),), generator=g, device=DEVICE)]
    return n, torch.cat([a, lone]), torch.cat([b, far])


def _undirected(n, a, b):
    rp, ci = _csr(n, torch.cat([a, b]), torch.cat([b, a]))
    return SimpleNamespace(n=n, directed=False, row_ptr=rp, col=ci, rrow_ptr=None, rcol=None)


def _erdos_renyi(n, g):
    """Mean degree 8, connected."""
    e = torch.randint(0, n, (2, 4 * n), generator=g, device=DEVICE)
    return _undirected(*_connect(n, e[0], e[1], g))


def _chung_lu(n, g):
    """Expected degrees ~ (i + 1)^(-2/3) (exponent 2.5), mean 16, at most
    n/100, drawn as endpoint pairs; connected."""
    w = torch.arange(1, n + 1, device=DEVICE, dtype=torch.float64) ** (-2.0 / 3.0)
    w = torch.clamp(w * (16.0 * n / w.sum()), max=max(16.0, n / 100))
    cum = torch.cumsum(w, 0)
    x = torch.rand((2, 8 * n), generator=g, device=DEVICE, dtype=torch.float64) * cum[-1]
    e = torch.clamp(torch.searchsorted(cum, x, right=True), max=n - 1)
    return _undirected(*_connect(n, e[0], e[1], g))


def _barabasi_albert(n, attach, g):
    """Linear form of preferential attachment: every new edge's far end is a
    uniform choice among all earlier edge ends, chains of choices resolved by
    pointer jumping."""
    m = n * attach
    first = 2 * torch.arange(m, device=DEVICE)
    far = (torch.rand(m, generator=g, device=DEVICE, dtype=torch.float64) * (first + 1)).to(torch.int64)
    ptr = torch.stack([first, torch.minimum(far, first)], 1).reshape(-1)
    while True:
        nxt = ptr[ptr]
        if torch.equal(nxt, ptr):
            break
        ptr = nxt
    return _undirected(n, ptr[0::2] // (2 * attach), ptr[1::2] // (2 * attach))


def _rmat(scale, g):
    """(a, b, c, d) = (.57, .19, .19, .05), directed, every id kept."""
    n, m = 1 << scale, 16 << scale
    src = torch.zeros(m, device=DEVICE, dtype=torch.int32)
    dst = torch.zeros(m, device=DEVICE, dtype=torch.int32)
    for _ in range(scale):
        r = torch.rand(m, generator=g, device=DEVICE)
        low = r >= 0.76
        src.mul_(2).add_(low)
        dst.mul_(2).add_(torch.where(low, r >= 0.95, r >= 0.57))
    src, dst = src.to(torch.int64), dst.to(torch.int64)
    rp, ci = _csr(n, src, dst)
    rrp, rci = _csr(n, dst, src)
    return SimpleNamespace(n=n, directed=True, row_ptr=rp, col=ci, rrow_ptr=rrp, rcol=rci)


def _graph(case, seed):
    g = _generator(seed)
    if case["family"] == "er":
        return _erdos_renyi(case["n"], g)
    if case["family"] == "chung_lu":
        return _chung_lu(case["n"], g)
    if case["family"] == "ba":
        return _barabasi_albert(case["n"], case["attach"], g)
    return _rmat(case["scale"], g)


def _host(t):
    """A pinned host copy as an int32 numpy array."""
    return None if t is None else t.cpu().pin_memory().numpy()


def _host_graph(x):
    return SimpleNamespace(n=x.n, directed=x.directed, row_ptr=_host(x.row_ptr), col=_host(x.col),
                           rrow_ptr=_host(x.rrow_ptr), rcol=_host(x.rcol))


def _load(x):
    return kadabra.kadabra_load_csr_device(x.n, x.row_ptr, x.col, x.directed, x.rrow_ptr, x.rcol)


def _pool(case):
    """Graph sizes of the batched and served cases, log-uniform, and their
    attachments; one graph at each end of the range."""
    rng = np.random.default_rng(case["n_hi"] + case["graphs"])
    ns = np.exp(rng.uniform(math.log(case["n_lo"]), math.log(case["n_hi"]), case["graphs"])).astype(np.int64)
    ns[0], ns[-1] = case["n_hi"], case["n_lo"]
    return rng, [int(n) for n in ns], [int(m) for m in rng.integers(4, 17, case["graphs"])]


# ---------------------------------------------------------------- state
def prepare(case, seed):
    call = case["call"]
    state = SimpleNamespace(case=case, seed=seed, stream=torch.cuda.current_stream().cuda_stream)
    if call == "check":
        state.check = _check_inputs(case, seed)
    elif call == "batch":
        _, ns, ms = _pool(case)
        graphs = [_barabasi_albert(n, m, _generator(seed + 1 + i)) for i, (n, m) in enumerate(zip(ns, ms))]
        graphs = [SimpleNamespace(n=x.n, directed=False, row_ptr=x.row_ptr.cpu().numpy(), col=x.col.cpu().numpy())
                  for x in graphs]
        state.batch = kadabra.Batch(graphs)
        state.counts = torch.zeros(sum(ns), dtype=torch.int32, device=DEVICE)
        state.btilde = torch.zeros(sum(ns), dtype=torch.float64, device=DEVICE)
        state.parts = list(state.counts.split(ns)), list(state.btilde.split(ns))
    elif call == "serve":
        rng, ns, ms = _pool(case)
        state.graphs = []
        for i, (n, m) in enumerate(zip(ns, ms)):
            kind = dict(family=("er", "chung_lu", "ba")[i % 3], n=n, attach=m)
            state.graphs.append(_load(_graph(kind, seed + 1 + i)))
        state.jobs = [(i % len(ns), float(rng.choice([0.02, 0.01, 0.005])), int(rng.choice([0, 10, 50])),
                       seed + i) for i in range(case["jobs"])]
    else:
        x = _graph(case, seed)
        if call == "load":
            state.csr = x
        elif call == "load_run":
            state.csr = _host_graph(x)
            state.counts = torch.zeros(x.n, dtype=torch.int32).pin_memory().numpy().view(np.uint32)
            state.btilde = torch.zeros(x.n, dtype=torch.float64).pin_memory().numpy()
        else:
            state.graph = _load(x)
            state.counts = torch.zeros(x.n, dtype=torch.int32, device=DEVICE)
            state.btilde = torch.zeros(x.n, dtype=torch.float64, device=DEVICE)
            state.totals = torch.zeros(kadabra.NSTAT, dtype=torch.int64, device=DEVICE)
    torch.cuda.synchronize()  # the library may work on a stream of its own
    return state


def _results(rs):
    """What runs return beside the counts and estimates: tau, the tests, the
    work counters and rankings; and the constants of computeDelta and the test."""
    whole = [np.concatenate([[r.tau, r.checks, r.vd], r.totals, [] if r.topk is None else r.topk]) for r in rs]
    return [np.concatenate(whole).astype(np.int64), np.array([(r.C, r.max_f, r.max_g) for r in rs])]


def run(state):
    case, call = state.case, state.case["call"]
    if call == "run":
        r = kadabra.kadabra_run(state.graph, case["lam"], DELTA, case["k"], state.seed,
                                check_interval=case["interval"], stream=state.stream, d_counts=state.counts,
                                d_btilde=state.btilde, want_host=False)
        return [state.counts, state.btilde] + _results([r])
    if call == "sample":
        state.counts.zero_()
        state.totals.zero_()
        kadabra.kadabra_sample_batch(state.graph, state.seed, 0, 0, case["samples"], state.counts, state.totals,
                                     state.stream)
        return [state.counts, state.totals]
    if call == "load":
        graph = _load(state.csr)
        vd = graph.vd
        graph.free()
        return vd
    if call == "load_run":
        graph = kadabra.kadabra_load_csr(state.csr)
        r = kadabra.kadabra_run(graph, case["lam"], DELTA, case["k"], state.seed, check_interval=case["interval"],
                                stream=state.stream, counts=state.counts, btilde=state.btilde)
        graph.free()
        return [state.counts, state.btilde] + _results([r])
    if call == "batch":
        n = case["graphs"]
        rs = state.batch.run([case["lam"]] * n, [DELTA] * n, [state.seed + i for i in range(n)],
                             stream=state.stream, d_counts=state.parts[0], d_btilde=state.parts[1], want_host=False)
        return [state.counts, state.btilde] + _results(rs)
    if call == "serve":
        ids = [kadabra.kadabra_submit(state.graphs[g], lam, DELTA, k, seed) for g, lam, k, seed in state.jobs]
        rs = [kadabra.kadabra_poll(job, state.graphs[g].n, k) for job, (g, _, k, _) in zip(ids, state.jobs)]
        return [x for r in rs for x in (r.counts, r.btilde)] + _results(rs)
    c = state.check
    return list(kadabra.kadabra_check(c.counts, c.tau, c.omega, c.ln_l, c.ln_u, c.lam))


# ---------------------------------------------------------------- the stop test's inputs and value
def _check_inputs(case, seed):
    """Counts as sampling gives them (most nodes unhit, a few hubs), and the
    per-node ln(1/delta) that computeDelta gives such counts."""
    rng = np.random.default_rng(seed)
    n, tau, omega = case["n"], 100000, 139915.0
    counts = np.minimum(rng.pareto(1.5, n) * 0.5, tau).astype(np.uint32)
    top = math.log(2.0 * n / (0.001 * DELTA))
    share = np.exp(-0.02 * counts)
    return SimpleNamespace(counts=counts, tau=tau, omega=omega, lam=0.005,
                           ln_l=3.0 + (top - 3.0) * share, ln_u=3.5 + (top - 3.5) * share)


def exact(case, seed):
    """The stop test's maxima and decision (Thm. 2).  The other cases' outputs
    follow from every random choice of their samples: a plain program takes
    minutes to retrace them."""
    if case["call"] != "check":
        return None
    c = _check_inputs(case, seed)
    t, b = float(c.tau), c.counts / float(c.tau)
    lower, upper = 1.0 / 3.0 - c.omega / t, 1.0 / 3.0 + c.omega / t
    f = c.ln_l / t * (lower + np.sqrt(lower * lower + 2.0 * b * c.omega / c.ln_l))
    g = c.ln_u / t * (upper + np.sqrt(upper * upper + 2.0 * b * c.omega / c.ln_u))
    return [bool((f <= c.lam).all() and (g <= c.lam).all()), float(f.max()), float(g.max())]


# ---------------------------------------------------------------- work
def _size(case):
    """(nodes, stored arcs of one direction, arcs a sample's search scans):
    the balanced search scans about sqrt(arcs), less where many pairs are not
    connected (directed R-MAT)."""
    if case["family"] == "rmat":
        n, m = 1 << case["scale"], 16 << case["scale"]
        return n, m, 0.56 * math.sqrt(m)
    n = case["n"]
    m = n * {"er": 8, "chung_lu": 16, "ba": 2 * case.get("attach", 10)}[case["family"]]
    return n, m, 1.5 * math.sqrt(m)


def _samples(lam):
    """Samples of a run: about half of omega at a vertex diameter of 10 to 17."""
    return 0.5 * 0.5 / lam**2 * (4 + math.log(2 / DELTA))


def work(case):
    """Bytes: each arc of a search read once (4 B), the counters and estimates
    written once (12 B per node); a load reads its CSRs once."""
    call = case["call"]
    flops = 0.0
    if call == "check":
        nbytes, flops = 20.0 * case["n"], 20.0 * case["n"]
    elif call in ("batch", "serve"):
        lo, hi = math.log(case["n_lo"]), math.log(case["n_hi"])
        ns = [math.exp(lo + (hi - lo) * (i + 0.5) / case["graphs"]) for i in range(case["graphs"])]
        jobs = case.get("jobs", case["graphs"])
        lam = case.get("lam", 0.0077)  # the served jobs' mean of 1 / lam^2
        per = sum(_samples(lam) * 4 * 1.5 * math.sqrt(20 * n) + 12.0 * n for n in ns) / len(ns)
        nbytes = jobs * per
    else:
        n, m, arcs = _size(case)
        graph = (8.0 if case["family"] == "rmat" else 4.0) * (n + m)
        if call == "load":
            nbytes = graph
        elif call == "sample":
            nbytes = case["samples"] * 4.0 * arcs + 4.0 * n
        else:
            nbytes = _samples(case["lam"]) * 4.0 * arcs + 12.0 * n + (graph if call == "load_run" else 0.0)
    return {"bytes": nbytes, "flops": flops}
