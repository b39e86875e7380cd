"""Periods in one call cost what they cost in calls of one period each: a warp
whose lanes have taken in different inbox words goes through the reaction
phase together."""
import numpy as np
import pytest

from paper_1512_03126_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rd():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1512_03126_gb300 import build
    build.build()
    from paper_1512_03126_gb300 import rdsplit
    return rdsplit


@pytest.mark.parametrize("mode", [0, 1])
def test_time_of_eight_periods(rd, mode):
    """Eleven species, 30 reactions, some hundred events a tet in the first
    periods (a millisecond and more each, so that a call's own cost is small).
    With the lanes one by one the call of eight periods took 1.8 times as long as
    eight calls; they share all work but the calls' own, and 1.2 is allowed."""
    import torch
    mesh = I.kuhn_box(12, 12, 12, (2.4e-6, 2.4e-6, 2.4e-6), 0.2, 4)
    model = I.random_model(mesh, 11, np.random.Generator(np.random.PCG64(9011)))
    counts = I.place_by_volume(mesh, [I.molecules(30e-6, float(np.sum(mesh.vol)))] * 11, 1)
    ms, ends = {}, {}
    with rd.Simulation(mesh, model, counts) as sim:
        rd.rdsplit_set_period_kernel(sim.h, mode, 0)
        for a_call in (1, 8, 1, 8):
            sim.set_counts(counts)
            rd.rdsplit_set_time(sim.h, 0.0, 0)
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            torch.cuda.synchronize()
            a.record()
            for _ in range(8 // a_call):
                sim.run_periods(a_call, 7)
            b.record()
            b.synchronize()
            ms[a_call] = a.elapsed_time(b)
            ends[a_call] = sim.counts()
    assert np.array_equal(ends[1], ends[8])
    assert ms[8] < 1.2 * ms[1], ms
