"""The warp's period step at the sizes where its parts meet: Philox blocks of
four molecules, whole-warp draws, the switch to the binomial sampler, species
counts on both sides of the inbox forms (values, 8-bit and 16-bit masks), the
capped draw, and tets whose single-precision reaction phase has to hand over
to double precision (more events than it follows, counts beyond its bound).
Every count equals the oracle's (tolerance 0: counts are whole numbers from
the same streams)."""
import numpy as np
import pytest

from paper_1512_03126_gb300 import inputs as I

pytestmark = pytest.mark.gpu

EDGES = [0, 1, 3, 4, 5, 31, 33, 127, 128, 129, 132, 4095, 4096, 4097, 9000]


@pytest.fixture(scope="module")
def rd():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1512_03126_gb300 import build
    build.build()
    from paper_1512_03126_gb300 import rdsplit
    return rdsplit


def both(rd, oracle, mesh, model, counts, periods, seed, rule, mode):
    with rd.Simulation(mesh, model, counts, rule=rule) as sim:
        rd.rdsplit_set_period_kernel(sim.h, mode, 0)
        sim.run_periods(periods, seed)
        first = sim.counts()
        sim.run_periods(periods, seed)          # a second run starts from cleared inboxes
        second = sim.counts()
        end = sim.time[0]
    ref = oracle.run(mesh, model, counts, np.inf, seed, max_periods=2 * periods, rule=rule)[0]
    half = oracle.run(mesh, model, counts, np.inf, seed, max_periods=periods, rule=rule)[0]
    # the batched engine on the same two stretches at once
    with rd.Simulation(mesh, model, counts, rule=rule) as sim:
        rd.rdsplit_ensemble_run([sim.h], [end], [seed])
        batched = sim.counts()
    assert np.array_equal(first, half) and np.array_equal(second, ref) and np.array_equal(batched, ref)


@pytest.mark.parametrize("mode", [0, 2])
@pytest.mark.parametrize("S", [1, 2, 3, 8, 9, 16])
def test_draw_edges(rd, oracle, S, mode):
    mesh = I.kuhn_box(3, 2, 5, (3e-7, 2e-7, 5e-7), 0.2, 7)       # 180 tets: a partial last warp
    model = I.diffusion_model(1e-12, S)
    model.D[S - 1] = 0.0 if S > 2 else model.D[S - 1]
    rng = np.random.Generator(np.random.PCG64(S))
    counts = rng.choice(EDGES, size=(mesh.n_tets, S)).astype(np.int32)
    both(rd, oracle, mesh, model, counts, 5, 3, 0, mode)


@pytest.mark.parametrize("rule", [0, 1, 2])
@pytest.mark.parametrize("mode", [0, 2])
@pytest.mark.parametrize("per_period", [0.02, 1.5, 40.0])
def test_reactions_and_capped_draws(rd, oracle, rule, mode, per_period):
    """Decay (N-bar above the count: the capped draw), influx, and doubled
    reactants, from events in few tets to more per tet than the
    single-precision pass follows."""
    mesh = I.kuhn_box(2, 3, 4, (2e-7, 3e-7, 4e-7), 0.2, 8)
    D = np.array([1e-12, 0.4e-12, 0.0])
    tau = 1e-7 ** 2 / 1e-12 / 100.0
    avv = I.AVOGADRO * 1e3 * float(np.mean(mesh.vol))
    lhs = np.array([[1, 0, 0], [0, 0, 0], [0, 2, 0], [1, 1, 0], [0, 0, 1]], np.int32)
    rhs = np.array([[0, 0, 0], [0, 3, 0], [0, 0, 1], [0, 0, 1], [1, 0, 0]], np.int32)
    k = np.array([per_period / 20 / tau, per_period / 8 / tau / avv, per_period / 200 / tau * avv,
                  per_period / 200 / tau * avv, 0.3 / tau])
    model = I.Model(D=D, lhs=lhs, rhs=rhs, k=k)
    rng = np.random.Generator(np.random.PCG64(5))
    counts = rng.choice([0, 1, 2, 12, 40], size=(mesh.n_tets, 3)).astype(np.int32)
    both(rd, oracle, mesh, model, counts, 6, 11, rule, mode)


def test_counts_beyond_the_single_precision_bound(rd, oracle):
    mesh = I.cube(2, 2e-7, 0.2, 3)
    model = I.Model(D=np.array([1e-12]), lhs=np.array([[1], [0]], np.int32), rhs=np.array([[0], [1]], np.int32),
                    k=np.array([1e-2, 1e-4]))
    counts = np.full((mesh.n_tets, 1), (1 << 20) - 1, np.int32)
    counts[::3] += 5000
    both(rd, oracle, mesh, model, counts, 2, 4, 0, 0)
