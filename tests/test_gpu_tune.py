"""mt_autotune times what a long run replays, and no graph's construction."""
import pytest

from paper_1811_05474_gb300 import mt, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("observe", [0, 64])
@pytest.mark.parametrize("warmup,steps", [(3, 10), (3, 12), (12, 13), (1, 1)])
def test_the_time_does_not_depend_on_the_counts(warmup, steps, observe):
    """N = 2000 (no wall layer): a step after three or twelve others costs what it
    costs in a run of hundreds.  A graph built between the events adds 40 % and
    more to 12 steps; the least of three tunings varies by a few per cent (the
    start of the first launch: half a step of one timed step)."""
    n = 2000
    x = synth.uniform_positions(n, float(n), seed=51)
    A, B = synth.uniform_masses(n, seed=51)
    p = mt.mt_params_init(n=n, L=(float(n),), precision=mt.MT_MIXED_DF32, observe_cap=observe)
    ms = [min(mt.autotune(p, x, A, B, warmup=w, steps=s)[1] for _ in range(3))
          for w, s in ((warmup, steps), (48, 240))]
    assert ms[0] <= 1.25 * ms[1], ms
