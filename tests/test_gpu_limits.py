"""Calls that cannot have what they ask for: what is refused leaves nothing behind, and a scan that can do
without some memory does. Allocations are refused by a stand-in for the allocator."""
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


ALLOCATOR = """
#define _GNU_SOURCE
#include <dlfcn.h>
#include <stddef.h>
size_t refuse_from = (size_t)-1, refuse_to = 0;
int refused = 0;
int cudaMallocFromPoolAsync(void** out, size_t n, void* pool, void* stream) {
  static int (*real)(void**, size_t, void*, void*);
  if (!real) *(void**)&real = dlsym(RTLD_NEXT, "cudaMallocFromPoolAsync");
  if (n >= refuse_from && n <= refuse_to) {
    refused++;
    return 2; /* out of memory */
  }
  return real(out, n, pool, stream);
}
"""


def child(tmp_path, code):
    """code in a process of its own, whose pool allocations of refuse(from, to) bytes fail."""
    src, lib = tmp_path / "allocator.c", tmp_path / "allocator.so"
    src.write_text(ALLOCATOR)
    subprocess.run(["gcc", "-O1", "-shared", "-fPIC", str(src), "-o", str(lib), "-ldl"], check=True)
    head = """
import ctypes, sys
sys.path.insert(0, sys.argv[1])
import numpy as np
import torch
from paper_0901_1307_gb300 import cv
shim = ctypes.CDLL(sys.argv[2])
def refuse(lo, hi):
    ctypes.c_size_t.in_dll(shim, "refuse_from").value = lo
    ctypes.c_size_t.in_dll(shim, "refuse_to").value = hi
def refused():
    return ctypes.c_int.in_dll(shim, "refused").value
"""
    return subprocess.run([sys.executable, "-c", head + code, ROOT, str(lib)], capture_output=True, text=True, timeout=300,
                          env=dict(os.environ, LD_PRELOAD=str(lib)))


def test_fragment_scan_without_memory_to_spare(built, tmp_path):
    """A fragment scan without memory for its masks, then without the room that an earlier scan's count
    suggests, then without room for the matches themselves, which alone is an error."""
    r = child(tmp_path, """
rng = np.random.default_rng(7)
file = rng.integers(0, 256, 64 * 300, dtype=np.uint8)
big = rng.integers(0, 256, 16 << 20, dtype=np.uint8)
for k in range(300):
    at = 50_000 * k + 4 * k
    big[at:at + 64] = file[64 * k:64 * k + 64]
small = big[:60_000].copy()
many = torch.from_numpy(np.tile(file, 300)).cuda()
big, small = torch.from_numpy(big).cuda(), torch.from_numpy(small).cuda()
for sig in (0, 1, 2):
    with cv.master_build([file, file], signature=sig, unit=cv.CV_UNIT_FRAGMENT) as m:
        with cv.scan(m, [big]) as r: want = r.matches(0)
        with cv.scan(m, [small]) as r: want_small = r.matches(0)
        assert want.size == 600 and want_small.size == 4
        tiles = -(-((len(big) - 64) // 4 + 1) // (32 * (23 if sig == 2 else 31)))
        before = refused()
        refuse(tiles * 128, tiles * 128)
        with cv.scan(m, [big]) as r: assert np.array_equal(r.matches(0), want)
        assert refused() == before + 1
        refuse(2**62, 0)
        with cv.scan(m, [many]) as r: found = r.count(0)
        assert found == 300 * 300 * 2, found
        refuse(1 << 20, 2**62)
        for _ in range(2):
            with cv.scan(m, [small]) as r: assert np.array_equal(r.matches(0), want_small)
        assert refused() == before + 2
        with cv.scan(m, [small[:64]]) as r: assert r.count(0) == 2
        try: cv.scan(m, [many]).close()
        except cv.CVError as e: assert e.code == cv.CV_ENOMEM
        else: raise SystemExit("no memory, and no error")
        refuse(2**62, 0)
        with cv.scan(m, [many]) as r: assert r.count(0) == found
        with cv.scan(m, [big], keep_on_device=True) as r:
            assert np.array_equal(cv.device_matches_to_numpy(r.matches(0)), want)
print("done")
""")
    assert r.stdout.strip() == "done", r.stdout + r.stderr
