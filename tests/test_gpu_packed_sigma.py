"""Path counts that outgrow the packed table entries' 24 bits inside a level
small enough to insert and test for touches in one pass, against the oracle
(GPU only).  Integers only, so equality is exact."""

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


SOURCES, ENDS = 600, 600


def _fan(gg, fan):
    """Sources, layers joined completely (4095^2 = 16,769,025 paths to a single
    node, just below 2^24), `fan` arcs to as many nodes that all enter one
    node, whose count so carries `fan` - 1 times beyond its 24 bits, and behind
    it a node with so many in-arcs that the forward search gets there."""
    e, n = [], 0

    def new(k):
        nonlocal n
        n += k
        return range(n - k, n)
    last = new(SOURCES)
    for w in (3, 3, 5, 7, 13, 3, 3, 5, 7, 13, 1):
        cur = new(w)
        e += [(a, b) for a in last for b in cur]
        last = cur
    mid, z, gate = new(fan), new(1)[0], new(1)[0]
    e += [(last[0], x) for x in mid] + [(x, z) for x in mid] + [(z, gate)]
    e += [(x, gate) for x in new(1500)]
    e += [(gate, x) for x in new(ENDS)]
    return gg.from_edges(n, e, directed=True, name=f"fan{fan}")


@pytest.mark.parametrize("fan", [1, 2, 127, 129, 192, 256, 257])
def test_carry_in_one_pass_level(kd, orc, gg, fan):
    g = _fan(gg, fan)
    ref = orc.sample_paths(g, 3, 0, 0, 4000, max_len=64)
    assert ((ref.st[:, 0] < SOURCES) & (ref.st[:, 1] >= g.n - ENDS)).sum() > 50
    G = kd.kadabra_load_csr(g)
    try:
        for f in (0, kd.FLAG_COMPACT_TABLES, kd.FLAG_LARGE_SHARED_TABLES, kd.FLAG_MEDIUM_TABLES, kd.FLAG_WARP_TIER):
            G.set_flags(f)
            got = kd.kadabra_sample_paths(G, 3, 0, 0, 4000, max_len=64)
            assert np.array_equal(got.status, ref.status) and np.array_equal(got.paths, ref.paths), f
            assert np.array_equal(got.stats, ref.stats), f
        # the small layout, which only runs take
        G.set_flags(0)
        r = kd.kadabra_run(G, 0.02, 0.1, 0, 5, check_interval=1000, ctas_per_sm=5, warp_tier=-1)
    finally:
        G.free()
    o = orc.run(g, 0.02, 0.1, seed=5, K=1000)
    assert r.tau == o.tau and np.array_equal(r.counts, o.counts) and (r.max_f, r.max_g) == (o.max_f, o.max_g)
