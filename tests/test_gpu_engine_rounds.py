"""The batched engine's rounds of a simulation in global memory: bitmap words
that are full, sparse and empty, more set bits in a batch of words than the
warp's list takes at once, more words a warp than a batch, and counts on both
sides of what a round draws in registers (eight molecules) and of the whole-warp
draw.  Counts equal the oracle's."""
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


@pytest.fixture(scope="module")
def mesh():
    return I.cube(29, 1e-6, 0.2, 5)     # 146,334 tets: 286 words a warp on one CTA, the last word partial


def fill(mesh, S, kind):
    rng = np.random.Generator(np.random.PCG64(17))
    T = mesh.n_tets
    if kind == "dense":
        return rng.choice([1, 2, 4, 5, 8], size=(T, S)).astype(np.int32)
    if kind == "edges":
        c = rng.choice([0, 0, 0, 1, 3, 4, 5, 8, 9, 128, 129], size=(T, S)).astype(np.int32)
        c[1000:9000] = 0
        return c
    c = np.zeros((T, S), np.int32)
    c[rng.choice(T, 3000, replace=False)] = 2
    c[0], c[T - 1] = 8, 8
    return c


@pytest.mark.parametrize("cluster", [1, 2, 8])
@pytest.mark.parametrize("S", [1, 2])
@pytest.mark.parametrize("kind", ["dense", "edges", "sparse"])
def test_rounds_match_the_oracle(rd, oracle, mesh, kind, S, cluster):
    model = I.diffusion_model(1e-12, S)
    counts = fill(mesh, S, kind)
    periods = 3
    ref = oracle.run(mesh, model, counts, np.inf, 8, max_periods=periods)[0]
    with rd.Simulation(mesh, model, counts) as sim:
        eng = rd.rdsplit_engine_create(1, mesh.n_tets)
        rd.rdsplit_engine_set_concurrency(eng, 0, cluster)
        rd.rdsplit_engine_add(eng, sim.h, 10 * periods * sim.tau, 8)
        rd.rdsplit_engine_step(eng, 1)
        rd.rdsplit_engine_step(eng, periods - 1)
        got = sim.counts()
        visited = rd.rdsplit_engine_stats(eng)[1]
        rd.rdsplit_engine_destroy(eng)
    assert np.array_equal(got, ref)
    assert visited >= periods * int(np.count_nonzero(counts.any(axis=1))) // 2
