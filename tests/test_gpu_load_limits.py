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
