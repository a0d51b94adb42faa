"""The KADABRA_CHECKED build runs checked_layouts.py in a child process (GPU
only, slow): the layouts and buffers that the forced-tier cases leave out."""

import os
import subprocess
import sys

import pytest

pytestmark = [pytest.mark.gpu, pytest.mark.slow]

HERE = os.path.dirname(os.path.abspath(__file__))


def test_checked_layouts():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1604_08553_gb300 import _build
    lib = _build.build_checked()
    out = subprocess.run([sys.executable, os.path.join(HERE, "checked_layouts.py"), lib], capture_output=True, text=True,
                         timeout=900)
    assert out.returncode == 0, out.stdout[-2000:] + out.stderr[-4000:]
    assert "checked layouts:" in out.stdout
