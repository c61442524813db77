"""The solver's host waits under the device's scheduling policy."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# Time steps on one core beside a process that is always busy there; prints the steps' share of the core.
CHILD = r"""
import ctypes as C, os, subprocess, sys, time
cu = C.CDLL("libcuda.so.1")
assert cu.cuInit(0) == 0
set_flags = getattr(cu, "cuDevicePrimaryCtxSetFlags_v2", None) or cu.cuDevicePrimaryCtxSetFlags
assert set_flags(0, 2) == 0          # CU_CTX_SCHED_YIELD, for this process's context
from synth import make_config
from paper_2403_04491_gb300 import problem_from_config
_, prob = problem_from_config(make_config(2).with_nx(48), stream=0)
prob.amg_setup()
prob.step(1)                         # first-use costs
core = max(os.sched_getaffinity(0))
os.sched_setaffinity(0, {core})
busy = subprocess.Popen([sys.executable, "-c", "import time\nt = time.time()\nwhile time.time() - t < 60: pass"])
try:
    time.sleep(0.5)
    t, cpu = time.perf_counter(), time.process_time()
    prob.step(10)
    prob.sync()
    print((time.process_time() - cpu) / (time.perf_counter() - t))
finally:
    busy.kill()
    busy.wait()
"""


def test_waits_yield_when_the_policy_says_so():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()
    r = subprocess.run([sys.executable, "-c", CHILD], capture_output=True, text=True, timeout=300,
                       env=dict(os.environ, PYTHONPATH=ROOT))
    assert r.returncode == 0, r.stderr
    # a wait that keeps its core takes its time slices: half of the core over such a wait, a fifth over a step.
    # A yielding one has the launches' own work left, under 5% of the busy process's slices between them.
    assert float(r.stdout.split()[-1]) < 0.1
