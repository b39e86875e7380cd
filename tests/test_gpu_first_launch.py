"""The first launch of a process, whatever its size, gets the shared memory that
it asks for: the default limit holds a kernel's static and dynamic shared
memory together, and no launch before it has raised the limit.  Each case runs
in a process of its own."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = """
import sys
import numpy as np, torch
from paper_1512_03126_gb300 import inputs as I, rdsplit as rd
from oracle import oracle as O
form, S, R, n = sys.argv[1], int(sys.argv[2]), int(sys.argv[3]), int(sys.argv[4])
mesh = I.cube(n, 1e-6, 0.2, 5)
model = I.diffusion_model(1e-12, S)
if R:
    model.lhs, model.rhs, model.k = np.eye(S, dtype=np.int32)[:1], np.zeros((1, S), np.int32), np.full(1, 100.0)
counts = np.full((mesh.n_tets, S), 3, np.int32)
ref = O.run(mesh, model, counts, np.inf, 4, max_periods=2)[0]
sim = rd.Simulation(mesh, model, counts)
if form == "engine":
    eng = rd.rdsplit_engine_create(1, mesh.n_tets)
    rd.rdsplit_engine_set_concurrency(eng, 0, 2)
    rd.rdsplit_engine_add(eng, sim.h, 10 * sim.tau, 4)
    rd.rdsplit_engine_step(eng, 2)
else:
    rd.rdsplit_set_period_kernel(sim.h, int(form), 256 if int(form) else 0)
    sim.run_periods(2, 4)
assert np.array_equal(sim.counts(), ref)
print("same")
"""


# engine on two CTAs: 9 cells a side ask for 48,128 bytes in shared memory, 13 are in global memory
@pytest.mark.parametrize("form, S, R, n", [("engine", 1, 1, 9), ("engine", 1, 0, 9), ("engine", 1, 1, 13), ("engine", 2, 0, 13),
                                           ("engine", 3, 1, 9), ("0", 1, 1, 9), ("0", 12, 1, 13), ("1", 11, 1, 9),
                                           ("1", 12, 0, 9), ("2", 12, 1, 9)])
def test_first_launch(form, S, R, n):
    r = subprocess.run([sys.executable, "-c", CHILD, form, str(S), str(R), str(n)], cwd=ROOT, capture_output=True,
                       text=True, timeout=300)
    assert r.returncode == 0 and "same" in r.stdout, r.stderr[-2000:]
