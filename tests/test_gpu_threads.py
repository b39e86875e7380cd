"""Handles of different species counts in different threads: a kernel's limit of
dynamic shared memory belongs to the function, not to a launch, so no thread's
launch may depend on what another thread has just launched.  (With a limit set
to each launch's own size, launches of the larger handle failed.)"""
import threading

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


def conversions(S):
    """S species, each converted into the next."""
    lhs, rhs = np.eye(S, dtype=np.int32)[:-1], np.eye(S, dtype=np.int32)[1:]
    return I.Model(D=np.linspace(0.1, 1.0, S) * 1e-12, lhs=lhs, rhs=rhs, k=np.full(S - 1, 1e3))


# period kernel in blocks of 256 threads (one pass, two passes); automatic (resident) runs
@pytest.mark.parametrize("mode, block", [(1, 256), (2, 256), (0, 0)])
def test_handles_of_different_species_counts_in_threads(rd, mode, block):
    import torch
    mesh = I.kuhn_box(3, 2, 5, (3e-7, 2e-7, 5e-7), 0.2, 7)
    runs, periods = 12, 1500           # a few ten thousand launches a thread
    errors, ends = [], {12: [], 16: []}

    def work(S, n):
        try:
            counts = I.place_by_volume(mesh, [400] * S, S)
            with rd.Simulation(mesh, conversions(S), counts, stream=torch.cuda.Stream()) as sim:
                rd.rdsplit_set_period_kernel(sim.h, mode, block)
                for _ in range(n):
                    sim.set_counts(counts)
                    rd.rdsplit_set_time(sim.h, 0.0, 0)
                    sim.run_periods(periods, 5)
                    ends[S].append(sim.counts())
        except Exception as e:   # reported below, in the test's thread
            errors.append(e)

    for S in ends:                     # alone
        work(S, 1)
    threads = [threading.Thread(target=work, args=(S, runs)) for S in ends]
    for th in threads:
        th.start()
    for th in threads:
        th.join()
    assert not errors, errors[0]
    for S in ends:
        assert len(ends[S]) == 1 + runs and all(np.array_equal(x, ends[S][0]) for x in ends[S])
