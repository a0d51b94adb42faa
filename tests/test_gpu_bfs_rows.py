"""Long rows that a bottom-up level of the load's BFS searches in vain, or to
their last arc (GPU only): the bound against the oracle at row lengths around
a lane's share, a warp's and an item's, and the load's time."""

import time

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


def _hub(gg, length, place, steps, directed):
    """A root with 6,000 chains of five nodes, so that every level is a wide
    one, and a path of `steps` nodes from it to a hub with `length` more arcs,
    whose other ends the search only reaches through the hub.  The path's last
    node stands first, in the middle or last in the hub's row; a tail behind
    the hub makes the bound depend on the hub's distance."""
    gate = 1 + {"first": 0, "middle": length // 2, "last": length}[place]
    far = [x for x in range(1, length + 2) if x != gate]
    path = [0, *range(length + 2, length + 1 + steps), gate]
    hub = length + 1 + steps
    tail = [hub + i for i in range(7)]
    first, width = tail[-1] + 1, 6000
    e = list(zip(path, path[1:] + [hub])) + list(zip(tail, tail[1:]))
    e += [(0, first + i) for i in range(width)] + [(first + i, first + i + width) for i in range(4 * width)]
    if directed:  # strongly connected; the hub's long row is that of its in-arcs
        e += [(tail[-1], x) for x in far] + [(x, hub) for x in far]
        e += [(first + 4 * width + i, 0) for i in range(width)] + [(hub, 0)]
    else:
        e += [(hub, x) for x in far]
    return gg.from_edges(first + 5 * width, e, directed=directed, name=f"hub{length}_{place}_{steps}")


@pytest.mark.parametrize("length", [63, 64, 65, 96, 1087, 1088, 1089, 1120, 5000])
@pytest.mark.parametrize("directed", [False, True])
def test_rows_of_unreached_hubs(kd, orc, gg, length, directed):
    for place in ("first", "middle", "last"):
        for steps in (1, 2, 4):
            g = _hub(gg, length, place, steps, directed)
            G = kd.kadabra_load_csr(g)
            vd = G.vd
            G.free()
            assert vd == orc.vd_bound(g), (place, steps)


def test_far_hub_costs_no_more_than_its_arcs(kd, gg):
    """A hub of 100,000 arcs that two bottom-up levels do not reach, beside
    the same graph with one of those arcs.  The hub's row is 1 % of the arcs;
    read by one thread it took 30 times the whole load."""
    import torch
    d = 100_000
    l1, l2, l3, hub = 1 + np.arange(d), 1 + d + np.arange(2 * d), 1 + 3 * d + np.arange(d), 1 + 4 * d
    n = hub + 1 + 40 * d
    times = []
    for joined in (1, d):
        e = np.concatenate([np.stack(x, 1) for x in (
            (np.zeros(d, np.int64), l1), (np.repeat(l1, 2), l2), (l2[::2], l3),
            (l3[:joined], np.full(joined, hub)), (np.repeat(l3, 40), hub + 1 + np.arange(40 * d)))])
        e = np.concatenate([e, e[:, ::-1]])
        key = torch.from_numpy(e[:, 0] * n + e[:, 1]).cuda().sort().values
        rp = torch.searchsorted(key, torch.arange(n + 1, device="cuda") * n).to(torch.int32)
        col = (key % n).to(torch.int32)
        best = 1e9
        for _ in range(5):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            G = kd.kadabra_load_csr_device(n, rp, col)
            best = min(best, time.perf_counter() - t0)
            assert G.vd == 9
            G.free()
        times.append(best)
    assert times[1] < 4 * times[0], times
