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
