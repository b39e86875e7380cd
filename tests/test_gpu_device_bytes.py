"""Admission counts what a simulation holds: serving.device_bytes covers the
bytes that the library takes from its allocator for a mesh, its model and its
place in an engine, and no tenth more."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = """
import numpy as np, torch
from paper_1512_03126_gb300 import inputs as I, rdsplit as rd, serving as SV
held = {}
def alloc(n):
    x = torch.empty(n, dtype=torch.uint8, device="cuda")
    held[x.data_ptr()] = x
    return x.data_ptr()
def free(p):
    torch.cuda.synchronize()
    held.pop(p)
rd.rdsplit_set_allocator(alloc, free)
for n in (3, 17):
    mesh = I.cube(n, 1e-6, 0.2, 5)
    for S in range(1, 17):
        eng = rd.rdsplit_engine_create(1, mesh.n_tets)
        before = sum(x.numel() for x in held.values())
        model = I.diffusion_model(1e-12, S)
        model.lhs, model.rhs, model.k = np.eye(S, dtype=np.int32), np.zeros((S, S), np.int32), np.full(S, 1.0)
        model.mask = np.ones((S, mesh.n_tets), np.uint8)
        sim = rd.Simulation(mesh, model)
        rd.rdsplit_engine_add(eng, sim.h, sim.tau, 1)
        took = sum(x.numel() for x in held.values()) - before
        told = SV.device_bytes(mesh.n_tets, S)
        assert took <= told <= 1.1 * took + 8192, (n, S, took, told)
        rd.rdsplit_engine_destroy(eng)
        sim.close()
print("covered")
"""


def test_device_bytes_cover_what_the_library_takes():
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "covered" in r.stdout, r.stderr[-2000:]
