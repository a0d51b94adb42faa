"""The sampler's level scans, candidate choice and small-frontier bounds at
the sizes where they change path, against the oracle (GPU only).

Layered graphs put a chosen number of rows of a chosen length into the
touching level: rows below, at and above a 32-arc window, a step of pass 1 and
the 32 rows a step resolves at once; frontiers around the 32 nodes whose row
bounds stay in shared memory; rows without arcs between others (directed).
Complete bipartite graphs set the number of candidate edges around the splits
of the quadratic choice and beyond it.  Integers only, so equality is exact."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def kd():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1604_08553_gb300 import kadabra
    kadabra.load_library()
    return kadabra


def _layers(gg, rows, arcs, directed, gap=0):
    """hub a -> `rows` middle nodes -> `arcs` shared leaves each -> hub b, so
    that searches between the hubs' neighbourhoods expand `rows` rows of about
    `arcs` arcs; every (gap)-th middle node has no arc to the leaves."""
    a, b = 0, 1
    mid = range(2, 2 + rows)
    leaf0 = 2 + rows
    nleaf = 2 * arcs + 3
    e = [(a, m) for m in mid]
    for i, m in enumerate(mid):
        if gap and i % gap == 1:
            continue
        e += [(m, leaf0 + (i + j) % nleaf) for j in range(arcs)]
    e += [(leaf0 + j, b) for j in range(nleaf)]
    return gg.from_edges(leaf0 + nleaf, e, directed=directed, name=f"layers{rows}x{arcs}_{int(directed)}_{gap}")


def _equal(kd, orc, g, flags, count=2000):
    ref = orc.sample_paths(g, 9, 0, 0, count, max_len=64)
    for f in flags:
        G = kd.kadabra_load_csr(g)
        try:
            G.set_flags(f)
            got = kd.kadabra_sample_paths(G, 9, 0, 0, count, max_len=64)
        finally:
            G.free()
        assert np.array_equal(got.status, ref.status), (g.name, f)
        assert np.array_equal(got.st, ref.st) and np.array_equal(got.paths, ref.paths), (g.name, f)
        assert np.array_equal(got.stats, ref.stats), (g.name, f)


@pytest.mark.parametrize("rows,arcs", [(1, 31), (1, 32), (1, 33), (3, 127), (2, 129), (31, 8), (32, 9), (33, 8),
                                       (40, 2), (70, 1), (300, 1), (12, 300)])
@pytest.mark.parametrize("directed,gap", [(False, 0), (True, 0), (True, 3)])
def test_level_shapes(kd, orc, gg, rows, arcs, directed, gap):
    g = _layers(gg, rows, arcs, directed, gap)
    _equal(kd, orc, g, (0, kd.FLAG_COMPACT_TABLES, kd.FLAG_ASYNC_SCAN, kd.FLAG_LARGE_SHARED_TABLES,
                        kd.FLAG_MEDIUM_TABLES, kd.FLAG_FRONTIER_SEGMENTS))


@pytest.mark.parametrize("p,q", [(4, 8), (4, 9), (8, 8), (8, 9), (16, 16), (12, 22), (16, 33), (24, 30)])
def test_candidate_counts(kd, orc, gg, p, q):
    """K_{p,q} with a pendant node on every vertex: two pendants of opposite
    sides meet over all arcs between the two neighbourhoods."""
    e = [(i, p + j) for i in range(p) for j in range(q)]
    # one extra node joined to every left vertex and one to every right vertex
    e += [(i, p + q) for i in range(p)] + [(p + j, p + q + 1) for j in range(q)]
    e += [(p + q, p + q + 2), (p + q + 1, p + q + 3)]
    g = gg.from_edges(p + q + 4, e, name=f"K{p},{q}+")
    _equal(kd, orc, g, (0, kd.FLAG_COMPACT_TABLES, kd.FLAG_MEDIUM_TABLES, kd.FLAG_FRONTIER_SEGMENTS), count=1500)


@pytest.mark.parametrize("count", [8191, 8192, 20000])
def test_screened_batches(kd, orc, gg, count):
    """Directed graphs most of whose samples end at a root without arcs: the
    launches large enough for the screening kernel, and those just below,
    give the oracle's hits and work counters; several graphs in one launch
    give each graph's own run."""
    import torch
    g = gg.rmat(12, 8, 0.57, 0.19, 0.19, 10)
    _, c_ref, t_ref = orc.accumulate(g, 5, 0, 100, count)
    G = kd.kadabra_load_csr(g)
    try:
        c = torch.zeros(g.n, dtype=torch.int32, device="cuda")
        t = torch.zeros(kd.NSTAT, dtype=torch.int64, device="cuda")
        kd.kadabra_sample_batch(G, 5, 0, 100, count, c, t)
        kd.kadabra_sync_status(G)
    finally:
        G.free()
    assert np.array_equal(c.cpu().numpy(), c_ref)
    assert np.array_equal(t.cpu().numpy()[:8], np.asarray(t_ref)[:8])


def test_screened_batch_run(kd, gg):
    graphs = [gg.rmat(11, 8, 0.57, 0.19, 0.19, 3), gg.erdos_renyi(2000, 8.0, 1), gg.rmat(12, 6, 0.57, 0.19, 0.19, 4)]
    B = kd.Batch(graphs)
    try:
        rs = B.run([0.02] * 3, [0.1] * 3, [7, 8, 9], check_interval=4096)
        for i, r in enumerate(rs):
            one = kd.kadabra_run(B.views[i], 0.02, 0.1, 0, 7 + i, check_interval=4096)
            assert r.tau == one.tau and np.array_equal(r.counts, one.counts)
            assert np.array_equal(r.totals, one.totals) and (r.max_f, r.max_g) == (one.max_f, one.max_g)
    finally:
        B.free()


def _chain(gg, width, layers=5):
    e = [(a * width + i, (a + 1) * width + j) for a in range(layers - 1) for i in range(width) for j in range(width)]
    return gg.from_edges(layers * width, e, name=f"chain{width}")


@pytest.mark.parametrize("make", [
    lambda gg: gg.erdos_renyi(16384, 8.0, 3, lcc=False), lambda gg: gg.erdos_renyi(16385, 8.0, 3, lcc=False),
    lambda gg: gg.erdos_renyi(12000, 30.0, 5), lambda gg: _chain(gg, 11), lambda gg: _chain(gg, 12),
    lambda gg: _chain(gg, 100), lambda gg: _chain(gg, 155), lambda gg: _chain(gg, 175),
    lambda gg: gg.barabasi_albert(5000, 7, 2), lambda gg: gg.rmat(12, 8, 0.57, 0.19, 0.19, 2),
], ids=["er16384", "er16385", "er12000", "chain11", "chain12", "chain100", "chain155", "chain175", "ba5000", "rmat12"])
def test_small_layout(kd, gg, make):
    """The layouts of ctas_per_sm 5, the small one up to 16,384 nodes, against
    the default one: samples that outgrow 1,536 list nodes, and candidate sets
    around 128 (one per thread) and beyond the small layout's share of the
    buffers (about 23,000)."""
    g = make(gg)
    G = kd.kadabra_load_csr(g)
    try:
        a, b = (kd.kadabra_run(G, 0.02, 0.1, 0, 5, check_interval=1000, ctas_per_sm=c, warp_tier=-1) for c in (4, 5))
    finally:
        G.free()
    assert a.tau == b.tau and np.array_equal(a.counts, b.counts) and np.array_equal(a.totals, b.totals)
