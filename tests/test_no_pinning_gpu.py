"""Stepping, waiting and reading back allocate no memory, page-locked host
memory among it: whoever steps with fdtd_step_noalloc() waits through
fdtd_synchronize().  The CUDA calls of a child process are recorded, whose
only grid is new (nothing is staged from an earlier one)."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CODE = """
import sys
sys.path.insert(0, %r)
import ctypes, torch
from torch.profiler import profile, ProfilerActivity
from paper_2207_06908_gb300 import fdtd as F, workloads as W
sc = W.random_scenario(3, n=(20, 14, 17), cpml=3, n_steps=40)

def names(work):
    with profile(activities=[ProfilerActivity.CPU, ProfilerActivity.CUDA]) as p:
        work()
    return {e.name for e in p.events()}

made = {}
def build():
    made["g"] = F.from_scenario(sc, probe_capacity=40)
print("build", sorted(names(build)))
g = made["g"]
def use():
    assert g._lib.fdtd_step_noalloc(g._h, ctypes.c_int(9)) == 0
    g.synchronize()
    g.read_probe(0, 0, 9)
    g.get_field(2)
print("use", sorted(names(use)))
g.close()
"""


def test_no_allocation_after_finalize():
    r = subprocess.run([sys.executable, "-c", CODE % ROOT], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr
    lines = dict(l.split(" ", 1) for l in r.stdout.splitlines() if l.startswith(("build ", "use ")))
    if "cuda" not in lines["use"]:
        pytest.skip("CUDA calls are not recorded here")
    assert "cudaLaunchKernel" in lines["use"] or "cuLaunchKernel" in lines["use"], lines["use"]
    for word in ("Malloc", "HostAlloc", "FreeHost", "cudaFree", "MemAlloc", "HostRegister"):
        assert word not in lines["use"], lines["use"]
