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


@pytest.mark.parametrize("S, N", [(1, 5000), (1, 2500), (3, 4500)])
@pytest.mark.parametrize("cluster", [1, 4, 8])
def test_engine_where_nearly_every_tet_is_left_to_the_pass(rd, oracle, cluster, S, N):
    """One species in shared memory (8 CTAs; 4 CTAs) and in global memory (1
    CTA), several species in global memory; several bitmap words a warp."""
    mesh = I.kuhn_box(16, 15, 17, (1.6e-6, 1.5e-6, 1.7e-6), 0.2, 6)    # 24,480 tets
    model = I.diffusion_model(1e-12, S)
    counts = np.random.Generator(np.random.PCG64(N)).poisson(N, (mesh.n_tets, S)).astype(np.int32)
    counts[100:228] = 1
    periods = 2
    ref = oracle.run(mesh, model, counts, np.inf, 5, max_periods=periods)[0]
    with rd.Simulation(mesh, model, counts) as sim:
        eng = rd.rdsplit_engine_create(1, mesh.n_tets)
        rd.rdsplit_engine_set_concurrency(eng, 0, cluster)
        rd.rdsplit_engine_add(eng, sim.h, 10 * periods * sim.tau, 5)
        rd.rdsplit_engine_step(eng, periods)
        got = sim.counts()
        rd.rdsplit_engine_destroy(eng)
    assert np.array_equal(got, ref)


def test_engine_pass_fills_its_rounds(rd):
    """On 8 CTAs a warp's words are a quarter of those on 2, so a period of
    nothing but such tets takes a quarter of the time; with a round for each bit of
    a lane's own word it took 0.8 of it (half is asked for)."""
    mesh = I.cube(16, 1e-6, 0.2, 5)
    model = I.diffusion_model(1e-12, 3)
    counts = np.full((mesh.n_tets, 3), 5000, np.int32)
    ms = {}
    with rd.Simulation(mesh, model) as sim:
        for cluster in (2, 8):
            eng = rd.rdsplit_engine_create(1, mesh.n_tets)
            rd.rdsplit_engine_set_concurrency(eng, 0, cluster)

            def reset():
                sim.set_counts(counts)
                rd.rdsplit_set_time(sim.h, 0.0, 0)
                rd.rdsplit_engine_add(eng, sim.h, 1.5 * sim.tau, 5)

            def step():
                rd.rdsplit_engine_step(eng, 2)
                rd.rdsplit_engine_poll(eng)

            ms[cluster] = best_ms(step, reset, 3)
            rd.rdsplit_engine_destroy(eng)
    assert ms[8] < 0.5 * ms[2], ms
