"""What a call launches (GPU only), read from PyTorch's profiler in a child
process: choices that no result shows, only the time."""

import json
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PRELUDE = """
import json, sys
sys.path.insert(0, sys.argv[1])
import torch
from torch.profiler import profile, ProfilerActivity
from paper_1604_08553_gb300 import kadabra as kd, graphgen as gg

def count(call, *names):
    with profile(activities=[ProfilerActivity.CPU, ProfilerActivity.CUDA]) as p:
        call()
        torch.cuda.synchronize()
    keys = p.key_averages()
    return [sum(k.count for k in keys if n in k.key) for n in names]

torch.zeros(1, device="cuda")
count(lambda: torch.zeros(8, device="cuda") + 1, "x")  # the first profile of a process may stay empty
"""


def _child(code):
    out = subprocess.run([sys.executable, "-c", PRELUDE + code, ROOT], capture_output=True, text=True, timeout=300)
    assert out.returncode == 0, out.stderr[-3000:]
    return json.loads([x for x in out.stdout.splitlines() if x.startswith("[")][-1])


def test_loop_graph_serves_every_interval():
    """The main loop's CUDA graph is built by the first run, not again by runs
    with other numbers of samples between two tests."""
    first, same, other, chosen = _child("""
g = gg.erdos_renyi(2000, 8.0, 1)
G = kd.kadabra_load_csr(g)
run = lambda lam, K: kd.kadabra_run(G, lam, 0.1, 0, 1, check_interval=K, ctas_per_sm=4, warp_tier=-1)
names = ("cudaGraphInstantiate", "cudaGraphLaunch")
print(json.dumps([count(lambda: run(0.01, 1000), *names), count(lambda: run(0.01, 1000), *names),
                  count(lambda: run(0.01, 1013), *names), count(lambda: run(0.009, 0), *names)]))
""")
    assert first == [1, 1] and same == [0, 1]
    assert other == [0, 1] and chosen == [0, 1]


def test_screening_goes_by_the_launch_s_samples():
    """The screening kernel runs where a quarter of a launch's samples are
    expected to end at a root without arcs: not in a batch or among served
    jobs because one graph of many is of that kind."""
    alone, few, mixed, most, served, served_mixed = _child("""
rmat = [gg.rmat(12, 8, 0.57, 0.19, 0.19, s) for s in (3, 4, 5)]
ba = [gg.barabasi_albert(20000, 5, s) for s in range(7)]
names = ("k_screen", "k_sample<2")
def batch(graphs, K):
    B = kd.Batch(graphs)
    run = lambda: B.run([0.01] * len(graphs), [0.1] * len(graphs), [1] * len(graphs), check_interval=K)
    run()
    c = count(run, *names)
    B.free()
    return c
def serve(graphs):
    G = [kd.kadabra_load_csr(g) for g in graphs]
    def run():
        ids = [kd.kadabra_submit(g, 0.01, 0.1, 0, 1, check_interval=16384) for g in G]
        for i, g in zip(ids, G):
            kd.kadabra_poll(i, g.n)
    run()
    c = count(run, *names)
    kd.kadabra_serve_shutdown()
    for g in G:
        g.free()
    return c
print(json.dumps([batch(rmat, 16384), batch(rmat[:1], 1000), batch(rmat[:1] + ba, 8192), batch(rmat + ba[:1], 8192),
                  serve(rmat), serve(rmat[:1] + ba)]))
""")
    assert alone[0] > 0 and most[0] > 0 and served[0] > 0
    assert few[0] == 0 and mixed[0] == 0
    assert served_mixed[0] <= served_mixed[1] // 2  # the last rounds may be the screened graph's job alone


def test_batch_tunes_the_layout_it_runs():
    """A batch's setup is timed with the launches the batch makes: the small
    layout only if all its graphs are small, and whatever a run on the probed
    graph alone has chosen before."""
    small, large, alone, large_again = _child("""
dense = gg.erdos_renyi(8000, 100.0, 1)   # the most arcs, few nodes
wide = gg.erdos_renyi(20000, 8.0, 2)
tiny, compact = "k_sample<0, 2", "k_sample<0, 1"
def batch(graphs):
    B = kd.Batch(graphs)
    c = count(lambda: B.run([0.05] * len(graphs), [0.1] * len(graphs), [1] * len(graphs)), tiny, compact)
    return B, c
S, small = batch([dense, dense])
L, large = batch([dense, wide])
alone = count(lambda: kd.kadabra_run(L.views[0], 0.05, 0.1, 0, 1, check_interval=1024), tiny, compact)
for B in (S, L):
    B.free()
L, again = batch([dense, wide])
L.free()
print(json.dumps([small, large, alone, again]))
""")
    assert small[0] > 0 and small[1] == 0
    assert large[0] == 0 and large[1] > 0
    assert alone[0] > 0 and alone[1] == 0
    assert large_again[0] == 0 and large_again[1] <= large[1]  # tuned before
