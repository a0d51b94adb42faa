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
    return json.loads(out.stdout.strip().splitlines()[-1])


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
