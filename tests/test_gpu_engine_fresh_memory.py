"""The first engine of a process runs every engine kernel once without work:
that must not depend on what a fresh device allocation holds.  A child process
serves the library's memory filled with ones (a negative item index)."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = """
import numpy as np, torch
from paper_1512_03126_gb300 import inputs as I, rdsplit as rd
from oracle import oracle as O
held = {}
def alloc(n):
    x = torch.full((n,), 255, dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    held[x.data_ptr()] = x
    return x.data_ptr()
rd.rdsplit_set_allocator(alloc, lambda p: held.pop(p))
w = I.diffusion_cube(3, 1e-6, 0.2, 5, 300, 0.004, 2)
s = rd.Simulation(w.mesh, w.model, w.counts)
rd.rdsplit_ensemble_run([s.h], [w.t_end], [w.seed])
assert np.array_equal(s.counts(), O.run(w.mesh, w.model, w.counts, w.t_end, w.seed)[0])
s.close()
print("same")
"""


def test_first_engine_on_memory_that_is_not_zero():
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "same" in r.stdout, r.stderr[-2000:]
