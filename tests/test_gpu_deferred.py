"""Tets that the rounds leave to the pass with the double-precision samplers:
binomial draws (4,096 molecules or more), whole-warp draws from 2,048 on, and
reaction phases that single precision does not follow.  Counts equal the
oracle's where nearly every tet of a mesh is such a tet, and the pass keeps its
lanes busy: its time is compared with that of the same draws laid out so that
lanes could not be shared."""
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


def best_ms(fn, reset, repeats=5):
    import torch
    out = []
    for _ in range(repeats + 1):
        reset()
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        a.record()
        fn()
        b.record()
        b.synchronize()
        out.append(a.elapsed_time(b))
    return min(out[1:])


def test_binomial_draws_of_a_warp_run_side_by_side(rd):
    """A period with 50,000 molecules in every tet against one with them in
    every 32nd tet (one a warp): one after another the first takes up to 32
    times as long, side by side the slowest of 32 draws (a quarter of 32 is
    asked for)."""
    mesh = I.kuhn_box(12, 12, 11, (1.2e-6, 1.2e-6, 1.1e-6), 0.2, 5)    # 9,504 tets
    every = np.full((mesh.n_tets, 1), 50000, np.int32)
    one = np.where(np.arange(mesh.n_tets)[:, None] % 32 == 0, every, 0).astype(np.int32)
    ms = {}
    for name, counts in (("every", every), ("one", one)):
        with rd.Simulation(mesh, I.diffusion_model(1e-12, 1), counts) as sim:
            ms[name] = best_ms(lambda: sim.run_periods(1, 3), lambda: sim.set_counts(counts))
    assert ms["every"] < 8.0 * ms["one"], ms
