"""The n-sized tables on graphs of few nodes (GPU only): candidate sets beyond
the 256 that are ranked pairwise, whose selection keeps its histogram in a
frontier array of fewer than 384 entries, against the oracle, and graphs
sampled with the same workspace after them."""

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


def _equal(kd, orc, g, flags):
    ref = orc.sample_paths(g, 4, 0, 0, 1000, max_len=24)
    G = kd.kadabra_load_csr(g)
    try:
        G.set_flags(flags)
        got = kd.kadabra_sample_paths(G, 4, 0, 0, 1000, max_len=24)
    finally:
        G.free()
    assert np.array_equal(got.status, ref.status) and np.array_equal(got.paths, ref.paths), g.name
    assert np.array_equal(got.stats, ref.stats), g.name
    return int(ref.stat("pi").max())


@pytest.mark.parametrize("side", [16, 17, 20, 24, 70, 120, 169])
def test_selection_on_few_nodes(kd, orc, gg, side):
    """Two sides joined completely, each with 20 nodes joined to all of it: two
    of those, one of each side, meet over side^2 candidate edges."""
    k, hubs = side, 20
    e = [(i, k + j) for i in range(k) for j in range(k)]
    e += [(i, 2 * k + h) for i in range(k) for h in range(hubs)]
    e += [(k + j, 2 * k + hubs + h) for j in range(k) for h in range(hubs)]
    joined = gg.from_edges(2 * (k + hubs), e, name=f"joined{k}")
    kd.kadabra_release_cached()  # a workspace of this graph's size
    assert _equal(kd, orc, joined, kd.FLAG_GLOBAL_TABLES) == k * k
    for n in (4, 60):  # in the same workspace, with tables that have to be empty
        _equal(kd, orc, gg.cycle_graph(n), kd.FLAG_GLOBAL_TABLES)
    assert _equal(kd, orc, joined, kd.FLAG_MEDIUM_TABLES) == k * k
