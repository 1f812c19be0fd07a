"""What creating and destroying runs does to others' work on the device."""
import ctypes
import os
import subprocess
import sys
import time

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def P():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1508_02748_gb300 as P
    from paper_1508_02748_gb300 import build
    build.build()
    return P


def _cudart():
    """Path of the CUDA runtime that this process has loaded."""
    with open("/proc/self/maps") as f:
        return next(line.split()[-1] for line in f if "libcudart.so" in line)


class _Runs:
    """Runs made through the C interface in workspaces allocated beforehand."""

    def __init__(self, P, n):
        import torch
        self.lib, self.cfg = P.load_library(), P.Config(L=4, seed=5).to_c()
        size = ctypes.c_size_t(0)
        assert self.lib.rewl_workspace_size(ctypes.byref(self.cfg), ctypes.byref(size)) == 0
        self.size, self.stream = size.value, torch.cuda.Stream()
        self.mem = [torch.empty(self.size, dtype=torch.uint8, device="cuda") for _ in range(n)]
        self.handles = []
        torch.cuda.synchronize()

    def create(self):
        for m in self.mem:
            h = ctypes.c_void_p(0)
            rc = self.lib.rewl_create(ctypes.byref(self.cfg), None, m.data_ptr(), self.size, self.stream.cuda_stream, ctypes.byref(h))
            assert rc == 0, self.lib.rewl_last_error(None)
            self.handles.append(h)

    def destroy(self):
        for h in self.handles:
            assert self.lib.rewl_destroy(h) == 0
        self.handles = []


def test_destroying_runs_waits_for_no_one(P):
    """80 runs are destroyed while another stream is busy for 0.2 s or more."""
    import torch
    runs = _Runs(P, 80)
    runs.create()
    other = torch.cuda.Stream()
    with torch.cuda.stream(other):
        torch.cuda._sleep(400_000_000)
    t = time.perf_counter()
    runs.destroy()
    t = time.perf_counter() - t
    busy = not other.query()
    torch.cuda.synchronize()
    assert busy and t < 0.1, t


RESET = """
import ctypes, sys
sys.path.insert(0, sys.argv[2])
rt = ctypes.CDLL(sys.argv[1], mode=ctypes.RTLD_GLOBAL)
import paper_1508_02748_gb300 as P
from paper_1508_02748_gb300 import rewl as R
lib, cfg = P.load_library(), P.Config(L=4, n_win_E=2, walkers_per_window=3, seed=5, exchange_interval=500).to_c()
size = ctypes.c_size_t(0)
assert lib.rewl_workspace_size(ctypes.byref(cfg), ctypes.byref(size)) == 0
got = []
for _ in range(3):
    mem, stream, h, st, d = ctypes.c_void_p(0), ctypes.c_void_p(0), ctypes.c_void_p(0), R.rewl_status(), ctypes.c_uint64(0)
    assert rt.cudaMalloc(ctypes.byref(mem), size) == 0 and rt.cudaStreamCreate(ctypes.byref(stream)) == 0
    assert lib.rewl_create(ctypes.byref(cfg), None, mem, size, stream, ctypes.byref(h)) == 0, lib.rewl_last_error(None)
    assert lib.rewl_run_cycles(h, 5, ctypes.byref(st)) == 0, lib.rewl_last_error(h)
    assert lib.rewl_tables_digest(h, ctypes.byref(d)) == 0
    got.append((st.cycles, st.trials, d.value))
    assert lib.rewl_destroy(h) == 0
    assert rt.cudaDeviceReset() == 0
assert got[0][:2] == (5, 2500) and got[1:] == [got[0]] * 2, got
print("same")
"""


def test_runs_after_a_device_reset(P):
    """In a process of its own: the device's context is ended between runs, and
    with it all memory that the library had from it."""
    r = subprocess.run([sys.executable, "-c", RESET, _cudart(), ROOT], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip() == "same", r.stdout + r.stderr
