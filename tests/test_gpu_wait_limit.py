"""A run whose grid barrier is waited for longer than the handle's limit ends with
RDSPLIT_ETIMEOUT and leaves counts, time and period index as they were before
the call; within the limit a long period is no error.  One tet has some tens of
thousands of reaction events in a period while all others wait for it."""
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


def one_busy_tet(events):
    """12,000 tets (more than one cluster holds); A <-> B, `events` a period
    for the 1,000 molecules of one tet, diffusion a thousandth of it."""
    mesh = I.kuhn_box(10, 10, 20, (1e-6, 1e-6, 2e-6), 0.2, 5)
    tau = 1e-7 ** 2 / 1e-12 / 100.0
    k = np.array([events / 1000.0 / tau] * 2)
    model = I.Model(D=np.array([1e-12, 1e-15]), lhs=np.array([[1, 0], [0, 1]], np.int32),
                    rhs=np.array([[0, 1], [1, 0]], np.int32), k=k)
    counts = np.zeros((mesh.n_tets, 2), np.int32)
    counts[4321, 1] = 1000
    return mesh, model, counts


def test_running_out_leaves_the_state_of_before_the_call(rd, oracle):
    mesh, model, counts = one_busy_tet(3e4)
    ref = oracle.run(mesh, model, counts, np.inf, 9, max_periods=3)[0]
    with rd.Simulation(mesh, model, counts) as sim:
        sim.run_periods(1, 9)
        first, when = sim.counts(), sim.time
        rd.rdsplit_set_wait_limit(sim.h, 1e-3)
        for _ in range(2):
            with pytest.raises(rd.RdsplitError) as e:
                sim.run_periods(2, 9)
            assert e.value.code == rd.RDSPLIT_ETIMEOUT
            assert np.array_equal(sim.counts(), first) and sim.time == when
        rd.rdsplit_set_wait_limit(sim.h, 60.0)
        sim.run_periods(2, 9)
        assert np.array_equal(sim.counts(), ref)


def test_a_long_period_is_no_error(rd, oracle):
    """About 300,000 events of one tet, a second and more, within the default limit."""
    mesh, model, counts = one_busy_tet(4e5)
    ref = oracle.run(mesh, model, counts, np.inf, 9, max_periods=1)[0]
    with rd.Simulation(mesh, model, counts) as sim:
        sim.run_periods(1, 9)
        assert np.array_equal(sim.counts(), ref)


def test_running_out_between_two_forms(rd, oracle):
    """3,072 tets that leave their cluster after a period, one of them busy for
    tenths of a second in the next: the wait over the device runs out with the
    cluster's next launch queued behind it.  The handle is at a point of the call
    (its counts are the oracle's there) and goes on from it."""
    mesh = I.kuhn_box(8, 8, 8, (8e-7, 8e-7, 8e-7), 0.2, 5)
    tau = 1e-7 ** 2 / 1e-12 / 100.0
    model = I.Model(D=np.array([1e-14]), lhs=np.ones((1, 1), np.int32), rhs=np.zeros((1, 1), np.int32),
                    k=np.array([0.01 / tau]))
    counts = np.full((mesh.n_tets, 1), 4500, np.int32)
    counts[777] = 200000
    with rd.Simulation(mesh, model, counts) as sim:
        rd.rdsplit_set_wait_limit(sim.h, 1e-6)
        with pytest.raises(rd.RdsplitError) as e:
            sim.run_periods(140, 9)
        assert e.value.code == rd.RDSPLIT_ETIMEOUT
        done = sim.time[1]
        assert 0 < done < 140
        assert np.array_equal(sim.counts(), oracle.run(mesh, model, counts, np.inf, 9, max_periods=done)[0])
        rd.rdsplit_set_wait_limit(sim.h, 60.0)
        sim.run_periods(3, 9)
        assert np.array_equal(sim.counts(), oracle.run(mesh, model, counts, np.inf, 9, max_periods=done + 3)[0])


def test_limits_that_are_not_positive_are_rejected(rd):
    mesh, model, counts = one_busy_tet(1e3)
    with rd.Simulation(mesh, model, counts) as sim:
        for bad in (0.0, -1.0, float("nan")):
            with pytest.raises(rd.RdsplitError) as e:
                rd.rdsplit_set_wait_limit(sim.h, bad)
            assert e.value.code == rd.RDSPLIT_EINVAL
