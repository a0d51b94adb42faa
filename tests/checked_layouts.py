"""Parity cases run against the KADABRA_CHECKED build of the library in a child
process (test_gpu_checked_layouts.py), for what checked_cases.py leaves out:
the compact and the small tier-S layout, row searches in segmented frontiers,
and candidate sets that fill the shared buffer and go on behind it.  Results
must equal the oracle's and no index check may fail."""

import os
import sys

import numpy as np

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)
sys.path.insert(0, os.path.dirname(os.path.abspath(__file__)))


def main(lib_path):
    from paper_1604_08553_gb300 import _build
    _build.build_kadabra = lambda *a, **k: lib_path
    from paper_1604_08553_gb300 import kadabra as kd, graphgen as gg
    import oracle as orc
    assert kd.load_library()._name == lib_path
    kb = gg.from_edges(200, [(i, 100 + j) for i in range(100) for j in range(100)], name="K100,100")
    # two hubs' neighbourhoods joined completely: candidate sets of 576 and 4,900 edges
    joined = [gg.from_edges(2 * k + 4, [(i, k + j) for i in range(k) for j in range(k)] +
                            [(i, 2 * k) for i in range(k)] + [(k + j, 2 * k + 1) for j in range(k)] +
                            [(2 * k, 2 * k + 2), (2 * k + 1, 2 * k + 3)], name=f"joined{k}") for k in (24, 70)]
    graphs = [gg.erdos_renyi(2000, 8.0, 1), gg.rmat(12, 16, 0.57, 0.19, 0.19, 1), gg.barabasi_albert(9000, 6, 3), kb,
              *joined]
    cases = 0
    for g in graphs:
        ref = orc.sample_paths(g, 3, 0, 100, 600, max_len=64)
        G = kd.kadabra_load_csr(g)
        try:
            for f in (kd.FLAG_COMPACT_TABLES, kd.FLAG_ASYNC_SCAN | kd.FLAG_FRONTIER_SEGMENTS,
                      kd.FLAG_COMPACT_TABLES | kd.FLAG_FRONTIER_SEGMENTS,
                      kd.FLAG_ASYNC_SCAN | kd.FLAG_LARGE_SHARED_TABLES):
                G.set_flags(f)
                got = kd.kadabra_sample_paths(G, 3, 0, 100, 600, max_len=64)
                assert np.array_equal(got.status, ref.status), (g.name, f)
                assert np.array_equal(got.paths, ref.paths) and np.array_equal(got.stats, ref.stats), (g.name, f)
                cases += 1
            G.set_flags(0)
            r = kd.kadabra_run(G, 0.04, 0.1, 0, 2, check_interval=500, ctas_per_sm=5, warp_tier=-1)  # the small layout
            o = orc.run(g, 0.04, 0.1, seed=2, K=500)
            assert r.tau == o.tau and np.array_equal(r.counts, o.counts), g.name
        finally:
            G.free()
    print(f"checked layouts: {cases} forced cases and {len(graphs)} runs equal to the oracle")


if __name__ == "__main__":
    main(sys.argv[1])
