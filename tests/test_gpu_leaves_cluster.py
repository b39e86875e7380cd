"""A mesh within one cluster whose tets mostly need the double-precision samplers
is spread over the device, and comes back: counts, time and period index are
the oracle's through both switches, in rdsplit_run, in a run of so many periods
and in the allocation-free call, with the last period shortened; and such a
period takes no longer than the same period in a launch of its own."""
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


def heavy_then_light(S):
    """3,072 tets (six warps a CTA) with 4,500 molecules of each species that
    decay within a few periods to the level of an influx."""
    mesh = I.kuhn_box(8, 8, 8, (8e-7, 8e-7, 8e-7), 0.2, 5)
    tau = 1e-7 ** 2 / 1e-12 / 100.0
    avv = I.AVOGADRO * 1e3 * float(np.mean(mesh.vol))
    lhs = np.concatenate([np.eye(S, dtype=np.int32), np.zeros((1, S), np.int32)])
    rhs = np.concatenate([np.zeros((S, S), np.int32), np.eye(S, dtype=np.int32)[:1]])
    model = I.Model(D=np.linspace(1.0, 0.3, S) * 1e-12, lhs=lhs, rhs=rhs,
                    k=np.array([1.0 / tau] * S + [2.0 / tau / avv]))
    return mesh, model, np.full((mesh.n_tets, S), 4500, np.int32)


@pytest.mark.parametrize("S", [1, 3])
def test_leaving_and_coming_back(rd, oracle, S):
    import torch
    mesh, model, counts = heavy_then_light(S)
    with rd.Simulation(mesh, model, counts) as sim:
        # over the periods spread over the device and back in the cluster; the last shortened
        t_end = 200.4 * sim.tau
        launches = rd.rdsplit_kernel_launches()
        sim.run(t_end, 3)
        launches = rd.rdsplit_kernel_launches() - launches
        got, when = sim.counts(), sim.time
    ref, t, period = oracle.run(mesh, model, counts, t_end, 3)
    assert np.array_equal(got, ref) and when == (t, period)
    assert 4 <= launches <= 8          # thresholds, cluster, spread, cluster
    with rd.Simulation(mesh, model, counts) as sim:
        for n in (1, 2, 100, 40):
            sim.run_periods(n, 3)
        assert np.array_equal(sim.counts(), oracle.run(mesh, model, counts, np.inf, 3, max_periods=143)[0])
        assert sim.time[1] == 143

    def dev(a):
        return torch.from_numpy(np.ascontiguousarray(a)).cuda()
    d = dev(counts)
    for end in (t_end, 200.0 * t_end / 200.4, 0.4 * t_end / 200.4):
        d.copy_(torch.from_numpy(counts))
        t, period = rd.rdsplit_run_static(mesh.n_tets, dev(mesh.adj), dev(mesh.vol), dev(mesh.area), dev(mesh.dist), S,
                                          model.D, model.n_reactions, model.lhs, model.rhs, model.k, None, 1.0, d, 0.0,
                                          0, end, 3)
        ref = oracle.run(mesh, model, counts, end, 3)
        assert np.array_equal(d.cpu().numpy(), ref[0]) and (t, period) == ref[1:]


def test_time_of_such_periods(rd):
    """7,986 tets of 5,000 molecules.  Within the cluster a period took 2.5 times
    as long as in a launch of its own; 1.5 is allowed."""
    import torch
    mesh = I.cube(11, 1.1e-6, 0.2, 5)
    counts = np.full((mesh.n_tets, 1), 5000, np.int32)
    ms = {}
    with rd.Simulation(mesh, I.diffusion_model(1e-12, 1)) as sim:
        for mode in (0, 1, 0, 1):
            rd.rdsplit_set_period_kernel(sim.h, mode, 0)
            sim.set_counts(counts)
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            torch.cuda.synchronize()
            a.record()
            sim.run_periods(12, 7)
            b.record()
            b.synchronize()
            ms[mode] = a.elapsed_time(b)
    assert ms[0] < 1.5 * ms[1], ms
