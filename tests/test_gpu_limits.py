"""Calls that cannot have what they ask for: what is refused leaves nothing behind."""
import os
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def built(cuda_device):
    import __graft_entry__

    __graft_entry__.build()


def test_an_unknown_configuration_costs_no_memory(built):
    """CV_SCAN_CONFIG naming no configuration: every call is refused, and none leaves host memory behind."""
    code = """
import sys
sys.path.insert(0, sys.argv[1])
import torch
from paper_0901_1307_gb300 import cv
x, out = (torch.zeros(n, dtype=torch.uint8, device="cuda") for n in (4096, 65536))
used = lambda: int(next(l for l in open("/proc/self/status") if l.startswith("VmRSS")).split()[1])
for k in range(100):
    try:
        cv.window_signatures(x.data_ptr(), 4096, 2, out.data_ptr())
    except cv.CVError as e:
        assert e.code == cv.CV_EINVAL
    else:
        raise SystemExit("accepted")
    if k == 10:
        first = used()
print(used() - first)
"""
    r = subprocess.run([sys.executable, "-c", code, ROOT], capture_output=True, text=True, timeout=300,
                       env=dict(os.environ, CV_SCAN_CONFIG="no_such_configuration"))
    assert r.returncode == 0, r.stdout + r.stderr
    assert int(r.stdout) < 64 << 10, r.stdout  # KiB
