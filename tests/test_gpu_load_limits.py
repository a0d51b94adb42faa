"""Loads at the ends of the accepted sizes (GPU only)."""

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


def _all_graphs(n, directed):
    """Every graph on n nodes with at least one arc, as edge lists."""
    pairs = [(a, b) for a in range(n) for b in range(n) if a != b and (directed or a < b)]
    for mask in range(1, 1 << len(pairs)):
        yield [p for i, p in enumerate(pairs) if mask >> i & 1]


@pytest.mark.parametrize("n,directed", [(2, False), (2, True), (3, False), (3, True), (4, False)])
def test_every_graph_of_few_nodes(kd, orc, gg, n, directed):
    """The VD bound's rounds of labelling, whose number is bounded by n."""
    for e in _all_graphs(n, directed):
        g = gg.from_edges(n, e, directed=directed, name=str(e))
        G = kd.kadabra_load_csr(g)
        vd = G.vd
        G.free()
        assert vd == orc.vd_bound(g), e


@pytest.mark.parametrize("n", [5, 6, 7, 9, 10])
def test_chains_of_few_nodes(kd, orc, gg, n):
    """Directed paths, and a cycle behind a path, labelled a node or two per round."""
    for e in ([(i, i + 1) for i in range(n - 1)],
              [(0, 1)] + [(1 + i, 1 + (i + 1) % (n - 1)) for i in range(n - 1)],
              [(0, i) for i in range(1, n)] + [(1 + i, 1 + (i + 1) % (n - 1)) for i in range(n - 1)]):
        g = gg.from_edges(n, e, directed=True, name=f"chain{n}")
        G = kd.kadabra_load_csr(g)
        vd = G.vd
        G.free()
        assert vd == orc.vd_bound(g), e


@pytest.mark.parametrize("directed", [False, True])
@pytest.mark.parametrize("n", [2, 33, 20000])
def test_graph_without_arcs(kd, orc, gg, n, directed):
    """No arcs at all: the arc passes have no chunk to take.  The bound, a run
    and a batch equal the oracle's."""
    g = gg.from_edges(n, [], directed=directed, name=f"edgeless{n}_{int(directed)}")
    ref = orc.run(g, 0.05, 0.1, seed=3, K=500)
    G = kd.kadabra_load_csr(g)
    try:
        assert G.vd == orc.vd_bound(g)
        got = kd.kadabra_run(G, 0.05, 0.1, 0, 3, check_interval=500)
    finally:
        G.free()
    B = kd.Batch([g, g])
    try:
        rb = B.run([0.05] * 2, [0.1] * 2, [3, 3], check_interval=500)
    finally:
        B.free()
    for r in (got, *rb):
        assert r.tau == ref.tau and r.C == ref.C and (r.max_f, r.max_g) == (ref.max_f, ref.max_g)
        assert np.array_equal(r.counts, ref.counts)


def _clique_rows(c, groups, tail, device="cuda"):
    """Columns of a clique's rows on ids [0, c), in order, with ids c, c + 1, ..
    appended to the lower rows: groups is a list of (rows up to, extra ids)."""
    import torch
    total = sum((hi - lo) * (c - 1 + x) for (lo, hi, x) in _ranges(groups)) + tail
    out = torch.empty(total, dtype=torch.int32, device=device)
    t = torch.arange(c - 1, dtype=torch.int32, device=device)
    at = 0
    for lo, hi, x in _ranges(groups):
        for a in range(lo, hi, 2000):
            u = torch.arange(a, min(a + 2000, hi), dtype=torch.int32, device=device)[:, None]
            m = t + (t >= u).to(torch.int32)
            if x:
                m = torch.cat([m, torch.arange(c, c + x, dtype=torch.int32, device=device).expand(len(u), x)], 1)
            out[at:at + m.numel()] = m.reshape(-1)
            at += m.numel()
    return out, at


def _ranges(groups):
    lo = 0
    for hi, x in groups:
        yield lo, hi, x
        lo = hi


def _offsets(deg):
    import torch
    rp = np.concatenate([[0], np.cumsum(deg, dtype=np.int64)])
    return torch.from_numpy(rp.astype(np.int32)).cuda(), int(rp[-1])


# a clique of 46,000 nodes and 1,000 pendant nodes, pendant j joined to the
# clique's nodes [0, 15,765) or, from the 824th on, [0, 15,764)
CLIQUE, PENDANTS, JOINED, LONGER = 46000, 1000, 15764, 823


@pytest.fixture(scope="module")
def largest(kd):
    """An undirected graph of 2^31 - 2 arcs on the device, the most there can be."""
    import torch
    groups = [(JOINED, PENDANTS), (JOINED + 1, LONGER), (CLIQUE, 0)]
    q = np.full(PENDANTS, JOINED) + (np.arange(PENDANTS) < LONGER)
    col, at = _clique_rows(CLIQUE, groups, int(q.sum()))
    for k in q:
        torch.arange(int(k), dtype=torch.int32, device="cuda", out=col[at:at + int(k)])
        at += int(k)
    deg = np.concatenate([np.full(hi - lo, CLIQUE - 1 + x) for lo, hi, x in _ranges(groups)] + [q])
    rp, m = _offsets(deg)
    assert m == at == col.numel() == 2 ** 31 - 2
    G = kd.kadabra_load_csr_device(CLIQUE + PENDANTS, rp, col)
    yield G, col
    G.free()
    del col, rp
    kd.kadabra_release_cached()
    torch.cuda.empty_cache()


def test_most_arcs_undirected(kd, largest):
    """Loads; node 0 is adjacent to all others, so the bound is 2 * 1 + 1.
    With the last arc changed, an id out of range, it is refused."""
    G, col = largest
    assert G.vd == 3
    kept = int(col[-1])
    try:
        col[-1] = CLIQUE + PENDANTS
        with pytest.raises(kd.KadabraError) as e:
            kd.kadabra_load_csr_device(CLIQUE + PENDANTS, G._keepalive[0], col)
        assert e.value.status == kd.ERR_CSR
        col[-1] = JOINED  # a node whose row does not hold the last pendant
        with pytest.raises(kd.KadabraError) as e:
            kd.kadabra_load_csr_device(CLIQUE + PENDANTS, G._keepalive[0], col)
        assert e.value.status == kd.ERR_CSR
    finally:
        col[-1] = kept


@pytest.mark.parametrize("sink", [False, True])
def test_most_arcs_directed(kd, sink):
    """2^31 - 1 arcs: a clique of both arcs and, at the end of the forward
    rows, 41 nodes with arcs into it, or, at the end of the reverse rows, one
    node with 41,707 arcs from it (whose row makes the condensation's passes go
    by arc).  Two components one behind the other, weighing 3 and 1."""
    import torch
    c = 46341
    if sink:
        q = np.array([2 ** 31 - 1 - c * (c - 1)])
        groups = [(int(q[0]), 1), (c, 0)]
    else:
        q = np.concatenate([np.full(40, 1020), [2 ** 31 - 1 - c * (c - 1) - 40 * 1020]])
        groups = [(int(q[-1]), 41), (1020, 40), (c, 0)]
    n = c + len(q)
    plain, _ = _clique_rows(c, [(c, 0)], int(q.sum()))  # the clique, then the other nodes' rows
    at = c * (c - 1)
    for k in q:
        torch.arange(int(k), dtype=torch.int32, device="cuda", out=plain[at:at + int(k)])
        at += int(k)
    joined, at2 = _clique_rows(c, groups, 0)
    rp_plain, m = _offsets(np.concatenate([np.full(c, c - 1), q]))
    rp_joined, m2 = _offsets(np.concatenate([np.full(hi - lo, c - 1 + x) for lo, hi, x in _ranges(groups)] +
                                            [np.zeros(len(q), np.int64)]))
    assert m == m2 == at == at2 == 2 ** 31 - 1
    fwd, rev = ((rp_joined, joined), (rp_plain, plain)) if sink else ((rp_plain, plain), (rp_joined, joined))
    G = kd.kadabra_load_csr_device(n, *fwd, True, *rev)
    try:
        assert G.vd == 4
    finally:
        G.free()
        kd.kadabra_release_cached()
        del plain, joined, fwd, rev
        torch.cuda.empty_cache()


@pytest.mark.parametrize("flags", ["", "LARGE_SHARED_TABLES", "MEDIUM_TABLES", "GLOBAL_TABLES"])
def test_rows_beyond_2_30_arcs(kd, largest, flags):
    """Samples whose rows lie up to 2^31 into the column array: distances,
    path counts and paths follow from the construction."""
    G, _ = largest
    count = 4000 if not flags else 600
    G.set_flags(getattr(kd, "FLAG_" + flags) if flags else 0)
    try:
        got = kd.kadabra_sample_paths(G, 1, 0, 0, count, max_len=4)
    finally:
        G.set_flags(0)
    assert not got.status.any()
    width = JOINED + (np.arange(PENDANTS) < LONGER)  # clique nodes a pendant is joined to: [0, width)
    seen = set()
    for (s, t), path, length, dist, sigma in zip(got.st, got.paths, got.path_len, got.stat("dist"),
                                                 got.stat("sigma_lo")):
        w = [int(width[x - CLIQUE]) if x >= CLIQUE else CLIQUE for x in (s, t)]
        pend = (s >= CLIQUE) + (t >= CLIQUE)
        common = min(w)
        near = pend == 0 or (pend == 1 and min(s, t) < common)
        assert (dist, sigma) == ((1, 1) if near else (2, common)), (s, t)
        assert length == dist + 1 and path[0] == s and path[length - 1] == t
        assert near or 0 <= path[1] < common
        seen.add((int(pend), bool(near)))
    assert {(0, True), (1, True), (1, False)} <= seen
