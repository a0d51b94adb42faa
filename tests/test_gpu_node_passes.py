"""The passes over all nodes of a run (compaction of the warm-up hits, top-k
selection, b~) at node counts around their rows of 256 nodes and groups of
eight rows, with counts on both sides of the 256 that b~ looks up, against
the oracle (GPU only).  b~ is one FP64 division on both sides and everything
else is integers or the oracle's own expression trees, so equality is exact."""

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


GRAPHS = [("star2048", lambda gg: gg.star_graph(2048)), ("star2049", lambda gg: gg.star_graph(2049)),
          ("cycle2047", lambda gg: gg.cycle_graph(2047)), ("ba4097", lambda gg: gg.barabasi_albert(4097, 3, 5)),
          ("K257", lambda gg: gg.complete_graph(257)), ("K2", lambda gg: gg.complete_graph(2)),
          ("rmat13", lambda gg: gg.rmat(13, 6, 0.57, 0.19, 0.19, 8))]


@pytest.mark.parametrize("name,make", GRAPHS, ids=[g[0] for g in GRAPHS])
@pytest.mark.parametrize("k", [0, 1, 9, 256])
def test_node_passes(kd, orc, gg, name, make, k):
    g = make(gg)
    lam = 0.04
    G = kd.kadabra_load_csr(g)
    try:
        got = kd.kadabra_run(G, lam, 0.1, k, 11, check_interval=500)
    finally:
        G.free()
    ref = (orc.run_topk(g, lam, 0.1, k, seed=11, K=500) if k else orc.run(g, lam, 0.1, seed=11, K=500))
    assert got.tau == ref.tau and got.C == ref.C
    assert np.array_equal(got.counts, ref.counts)
    assert np.array_equal(got.btilde, got.counts.astype(np.float64) / float(got.tau))
    assert (got.max_f, got.max_g) == (ref.max_f, ref.max_g)
    if k:
        assert np.array_equal(got.topk, np.asarray(ref.topk)[:len(got.topk)])
