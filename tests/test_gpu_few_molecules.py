"""One species without reactions, warps whose tets hold at most eight molecules
(drawn in registers) beside warps with more: resident runs, one launch a period
and two passes give the oracle's counts, also for a species that does not move."""
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


@pytest.mark.parametrize("mode, block", [(0, 0), (1, 0), (1, 256), (2, 64)])
@pytest.mark.parametrize("D", [1e-12, 0.0])
def test_few_molecules(rd, oracle, mode, block, D):
    mesh = I.kuhn_box(12, 11, 12, (1.2e-6, 1.1e-6, 1.2e-6), 0.2, 5)     # 9,504 tets: more than one cluster holds
    rng = np.random.Generator(np.random.PCG64(3))
    counts = rng.integers(0, 9, size=(mesh.n_tets, 1)).astype(np.int32)
    counts[2000:4000] = 0
    counts[4000:4064] = 8
    counts[5000:5200, 0] = rng.choice([0, 1, 8, 9, 130, 5000], size=200)
    model = I.diffusion_model(1e-12, 1)
    model.D[0] = D
    with rd.Simulation(mesh, model, counts) as sim:
        rd.rdsplit_set_period_kernel(sim.h, mode, block)
        if D == 0.0:                       # no period length: one period to the end
            sim.run(1e-3, 6)
            assert np.array_equal(sim.counts(), counts)
            return
        sim.run_periods(1, 6)
        assert np.array_equal(sim.counts(), oracle.run(mesh, model, counts, np.inf, 6, max_periods=1)[0])
        sim.run_periods(7, 6)
        assert np.array_equal(sim.counts(), oracle.run(mesh, model, counts, np.inf, 6, max_periods=8)[0])
