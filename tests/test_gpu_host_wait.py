"""On a device set to blocking synchronisation the host thread sleeps through the
waits of a step instead of polling.  In a process of its own: the flag is set
before the context exists."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SCRIPT = """
import ctypes, sys, time
cu = ctypes.CDLL("libcuda.so.1")
assert cu.cuInit(0) == 0 and cu.cuDevicePrimaryCtxSetFlags_v2(0, 4) == 0   # CU_CTX_SCHED_BLOCKING_SYNC
sys.path.insert(0, ".")
from paper_2210_03763_gb300 import native, workloads as W
g = native.TTN(5, 5, 128)
g.set_precision(native.FP64)
g.set_hamiltonian(W.square_lattice(5, 5), 20.0)
g.apply_pulse(W.random_constant_schedule(25, 1))
g.set_product_state(W.random_product_amps(25, 2))
g.step(0.02)
t, c = time.perf_counter(), time.thread_time()
g.step(0.02)
print((time.thread_time() - c) / (time.perf_counter() - t))
"""


def test_blocking_device_lets_the_host_thread_sleep():
    import __graft_entry__ as ge
    ge.build()
    out = subprocess.run([sys.executable, "-c", SCRIPT], cwd=ROOT, capture_output=True, text=True, timeout=120)
    assert out.returncode == 0, out.stderr[-2000:]
    # launches take their part of a core; polling takes all of it
    assert float(out.stdout.split()[-1]) < 0.7, out.stdout
