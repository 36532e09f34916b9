"""mt_run's graphs of several steps against the same steps launched one by one:
positions, masses and observables bit for bit, for plain steps, segments that
only the second tier can take (particles piled against a wall), steps that
only the general pipeline can do, batches, and step counts around the graph's."""
import numpy as np
import pytest

from paper_1811_05474_gb300 import mt, synth

from .test_gpu_parity import PRECISIONS

pytestmark = pytest.mark.gpu


def compare(p, x, A, B, runs, batch=None):
    sims = [mt.Simulation(p, batch=batch) for _ in range(2)]
    for s in sims:
        s.upload(x, A, B)
    for n in runs:
        sims[0].run(n)
        sims[1].step(n)
        assert np.array_equal(sims[0].ticks(), sims[1].ticks()), n
        for a, b in zip(sims[0].masses(), sims[1].masses()):
            assert np.array_equal(a, b), n
        assert sims[0].steps_done() == sims[1].steps_done()
        if p.observe_cap:
            assert np.array_equal(sims[0].observables(), sims[1].observables()), n
    for s in sims:
        s.close()


@pytest.mark.parametrize("precision", PRECISIONS)
@pytest.mark.parametrize("observe", [0, 40])
@pytest.mark.parametrize("n,L,v,pile", [
    (1000, 1000.0, 0.0, 0),       # first tier only
    (20011, 18000.0, 0.5, 0),
    (3000, 3000.0, 0.5, 600),     # second tier from the first step
    (4000, 4000.0, 6.0, 0),       # ... on the way
    (9000, 9000.0, 0.5, 7000),    # general pipeline
])
def test_equals_single_steps(precision, observe, n, L, v, pile):
    p = mt.mt_params_init(n=n, L=(L,), v=(v, 0.0), precision=precision, observe_cap=observe, seed=4)
    x = synth.uniform_positions(n, L, seed=1)
    x[0, :pile] = L - 1e-3 * x[0, :pile] / L
    A, B = synth.uniform_masses(n, seed=2)
    compare(p, x, A, B, [12, 1, 30, 5, 24] if pile < 1000 else [13])


@pytest.mark.parametrize("precision", PRECISIONS)
def test_batch(precision):
    ns, Ls = [700, 1, 2500, 33], [700.0, 2.0, 2000.0, 40.0]
    p = mt.mt_params_init(dim=1, v=(1.0, 0.0), precision=precision, observe_cap=40, seed=3)
    x = np.concatenate([synth.uniform_positions(n, L, seed=5)[0] for n, L in zip(ns, Ls)])[None]
    A, B = synth.uniform_masses(sum(ns), seed=6)
    compare(p, x, A, B, [25, 2, 36], batch=mt.make_batch(ns, Ls))


@pytest.mark.parametrize("precision", PRECISIONS)
def test_step_waits_for_its_predicted_segments(precision):
    """A large system whose wall layer keeps the predicted-segment kernel busy
    longer than the first tier: the state after graph steps without observables
    is the one with them (whose kernel, behind the predicted segments, the
    step's end waits for)."""
    n, L = 700000, 700000.0
    x = synth.uniform_positions(n, L, seed=1)
    x[0, :900] = L - 0.25 * synth.rng(5).exponential(size=900)
    A, B = synth.uniform_masses(n, seed=2)
    out = []
    for observe in (0, 8):
        p = mt.mt_params_init(n=n, L=(L,), v=(0.5, 0.0), precision=precision, seed=4,
                              observe_cap=observe)
        sim = mt.Simulation(p)
        sim.upload(x, A, B)
        sim.run(8)
        out.append((sim.ticks(), *sim.masses()))
        sim.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("n", [1000, 400000])  # graphs of several steps; of one step
def test_checkpoint_without_the_graph_words(tmp_path, n):
    """A file from before the control block held the words of the several-step
    graphs (bytes 184 on of its 256, the workspace's first) has anything there."""
    p = mt.mt_params_init(n=n, L=(float(n),), v=(0.5,), precision=mt.MT_MIXED, seed=9)
    a, b = mt.Simulation(p), mt.Simulation(p)
    a.upload(synth.uniform_positions(n, float(n), seed=1), *synth.uniform_masses(n, seed=1))
    a.run(14)
    path = tmp_path / "old.ckpt"
    a.save(path)
    data = bytearray(path.read_bytes())
    at = len(data) - a.nbytes
    data[at + 184:at + 256] = b"\xa5" * 72
    path.write_bytes(data)
    a.run(26)
    b.load(path)
    b.run(26)
    assert np.array_equal(a.ticks(), b.ticks())
    for u, v in zip(a.masses(), b.masses()):
        assert np.array_equal(u, v)
