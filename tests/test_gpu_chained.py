"""Chained launches must not lengthen a step: a step of a run takes no longer than
its kernels one by one (timed with an event before each)."""
import time

import pytest

from paper_1811_05474_gb300 import mt, synth

from .test_gpu_parity import PRECISIONS

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", PRECISIONS)
@pytest.mark.parametrize("dim,n,L", [(1, 5000, 37.0), (1, 20000, 147.0), (1, 30000, 220.0),
                                     (1, 40208, 296.0), (1, 70000, 515.0), (2, 38000, 195.0),
                                     (2, 60000, 245.0), (2, 77000, 277.0)])
def test_a_step_is_no_longer_than_its_kernels(dim, n, L, precision):
    """Dense 1-d systems (tiles) and 2-d ones.  Launches overlap in the run and
    not in the profile, so the run is the shorter one by some microseconds; it
    may be 15 % longer here."""
    p = mt.mt_params_init(dim=dim, n=n, L=(L,) * dim, react=0, precision=precision)
    sim = mt.Simulation(p)
    sim.upload(synth.uniform_positions(n, L, dim=dim, seed=1), *synth.uniform_masses(n, seed=1))
    sim.run(4)
    sim.sync()
    run = float("inf")
    for _ in range(3):
        t = time.perf_counter()
        sim.run(40)
        sim.sync()
        run = min(run, (time.perf_counter() - t) / 40 * 1e3)
    mt.mt_set_profiling(sim.h, 1)
    kernels = float("inf")
    for _ in range(3):
        sim.step()
        sim.sync()
        kernels = min(kernels, sum(ms for _, ms in mt.mt_read_profile(sim.h)))
    sim.close()
    assert run <= 1.15 * kernels, (run, kernels)
