"""The load's arc passes (CSR checks, mirror test, VD bound) at the sizes where
they change path (GPU only): rows, and runs of rows without arcs, around the
32 rows and 32 arcs of a window and the 512 arcs of a chunk; components that
many nodes enter; a graph beyond the L2, whose mirror test searches pivots.
The VD bound equals the oracle's; a CSR with one entry changed is refused."""

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


def _vd(kd, g):
    G = kd.kadabra_load_csr(g)
    try:
        return G.vd
    finally:
        G.free()


def _directed(gg, n, edges, name):
    return gg.from_edges(n, edges, directed=True, name=name)


@pytest.mark.parametrize("row,empty", [(1, 0), (1, 31), (1, 32), (1, 33), (31, 1), (32, 40), (33, 100), (511, 3),
                                       (512, 70), (513, 1)])
def test_rows_and_gaps(kd, orc, gg, row, empty):
    """Every (empty + 1)-th node has `row` out-arcs to the nodes after it."""
    step, n = empty + 1, 3000
    e = [(u, (u + 1 + 7 * j) % n) for u in range(0, n, step) for j in range(row) if (7 * j + 1) % n]
    g = _directed(gg, n, e[:60000], f"rows{row}_{empty}")
    assert _vd(kd, g) == orc.vd_bound(g)


def test_components(kd, orc, gg):
    """Chains of cycles of several sizes behind thousands of sources, and a
    root's component that is a single node with many entering arcs."""
    e, base = [], 0
    for size in (5, 40, 3, 700, 1, 12):  # components in topological order
        e += [(base + i, base + (i + 1) % size) for i in range(size) if size > 1]
        e.append((base + size - 1, base + size))
        base += size
    n = base + 1 + 4000
    e += [(base + 1 + i, i % base) for i in range(4000)]
    g = _directed(gg, n, e, "cycles")
    assert _vd(kd, g) == orc.vd_bound(g)
    star = _directed(gg, 5000, [(i, 0) for i in range(1, 4000)] + [(0, i) for i in range(4000, 5000)] +
                     [(i, i + 1) for i in range(4000, 4999)], "star")
    assert _vd(kd, star) == orc.vd_bound(star)
    und = gg.from_edges(4000, [(0, i) for i in range(1, 2000)] + [(i, i + 1) for i in range(2000, 3999)],
                        name="star and path")
    assert _vd(kd, und) == orc.vd_bound(und)


@pytest.mark.parametrize("hub", [0, 1024, 1025])
def test_outside_the_core(kd, orc, gg, hub):
    """A large component, nodes before and behind it with rows of 0 to 40
    arcs, a second component behind it that chains into more nodes, and a
    node with `hub` in-arcs, whose row decides whether the passes over the
    other components go by node or by arc."""
    rng = np.random.default_rng(11)
    core, out, src = 2500, 3000, 1500
    e = [(i, (i + 1) % core) for i in range(core)] + [(0, i) for i in range(2, core)] + [(i, 0) for i in range(3, core)]
    for i in range(out):  # behind the core: i % 41 in-arcs from it, some from the nodes before
        y = core + i
        e += [(int(u), y) for u in rng.choice(core, i % 41, replace=False)]
        e += [(core + i - k, y) for k in (1, 7, 32) if i >= k and i % (k + 2) == 0]
    base = core + out
    e += [(base + i, (base + (i + 1) % 50)) for i in range(50)] + [(5, base), (base + 3, base + 50)]
    e += [(base + 50 + i, base + 51 + i) for i in range(60)]
    first = base + 111
    for i in range(src):  # before it
        e += [(first + i, int(u)) for u in rng.choice(core + out, i % 19, replace=False)]
    n = first + src + 1
    e += [(int(u), n - 1) for u in rng.choice(core, hub, replace=False)]
    g = _directed(gg, n, e, f"core{hub}")
    assert _vd(kd, g) == orc.vd_bound(g)


@pytest.mark.parametrize("directed", [False, True])
def test_changed_entry_is_refused(kd, gg, directed):
    rng = np.random.default_rng(3)
    g = (gg.rmat(11, 8, 0.57, 0.19, 0.19, 5) if directed else gg.chung_lu(3000, 2.5, 12.0, 300.0, 6))
    _refused_after_changes(kd, g, rng, 12)


def test_changed_entry_is_refused_beyond_l2(kd, gg):
    import torch
    g = gg.rmat(20, 18, 0.57, 0.19, 0.19, 4)
    l2 = torch.cuda.get_device_properties(0).L2_cache_size
    assert 8 * (g.n + 1 + g.m) > l2, "the graph has to exceed the L2"
    G = kd.kadabra_load_csr(g)  # accepted as it is
    G.free()
    _refused_after_changes(kd, g, np.random.default_rng(7), 8)


@pytest.mark.parametrize("offset", [0, 1])
def test_device_csr_beyond_l2(kd, gg, offset):
    """Borrowed device arrays, aligned to 32 bytes or not, with a number of
    arcs that is no multiple of 8; the very last entry changed is refused."""
    import torch
    g = gg.rmat(20, 18, 0.57, 0.19, 0.19, 4)
    assert g.m % 8, "the last group of 8 has to be a partial one"

    def dev(a):
        t = torch.empty(a.size + offset, dtype=torch.int32, device="cuda")[offset:]
        t.copy_(torch.from_numpy(a))
        return t
    rp, col, rrp, rcol = (dev(a) for a in (g.row_ptr, g.col, g.rrow_ptr, g.rcol))
    G = kd.kadabra_load_csr_device(g.n, rp, col, True, rrp, rcol)
    vd = G.vd
    G.free()
    assert vd == _vd(kd, g)
    last = int(g.rcol[-1])
    deg = np.diff(g.rrow_ptr)
    row = int(np.nonzero(deg)[0][-1])
    rcol[-1] = last + 1 if last + 1 != row and last + 1 < g.n else last - 1
    with pytest.raises(kd.KadabraError) as e:
        kd.kadabra_load_csr_device(g.n, rp, col, True, rrp, rcol)
    assert e.value.status == kd.ERR_CSR


def _refused_after_changes(kd, g, rng, changes):
    """Moves one entry of the searched CSR to a free id between its
    neighbours, in short and long rows, one at a time."""
    import copy
    rp, col = (g.rrow_ptr, g.rcol) if g.directed else (g.row_ptr, g.col)
    deg = np.diff(rp)
    rows = np.concatenate([np.argsort(deg)[-changes // 2:], rng.choice(np.nonzero(deg > 0)[0], changes)])
    done = 0
    for v in rows:
        a, b = int(rp[v]), int(rp[v + 1])
        row = col[a:b].astype(np.int64)
        lo = np.concatenate([[-1], row[:-1]])
        free = np.nonzero((row - lo > 1) & (row - 1 != v))[0]
        if free.size == 0:
            continue
        at = a + int(rng.choice(free))
        h = copy.copy(g)
        bad = col.copy()
        bad[at] -= 1
        if g.directed:
            h.rcol = bad
        else:
            h.col = bad
        with pytest.raises(kd.KadabraError) as e:
            kd.kadabra_load_csr(h)
        assert e.value.status == kd.ERR_CSR, (int(v), at)
        done += 1
        if done == changes:
            break
    assert done >= changes // 2
