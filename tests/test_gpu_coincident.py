"""Periodic walls in 1-d with particles at one place: the cell list's walks go
around the domain and must not meet a particle twice where a whole realisation
lies within the cutoff of one point and its lowest (or highest) position is
shared.  Against the oracle: the computed weights, the stored ones (with and
without entries past the band), tracers and batches, and the pair sets."""
import numpy as np
import pytest

import oracle as O
from paper_1811_05474_gb300 import mt, synth

from .test_gpu_parity import PRECISIONS, TOL, assert_masses

pytestmark = pytest.mark.gpu

L = 20.0
# positions of one realisation, the cutoff being 1.9: all at one place, the
# lowest tied, the highest tied, either side of the wall, and a full domain
PLACES = {
    "two": [7.0, 7.0],
    "three": [7.0, 7.0, 7.0],
    "low": [7.0, 7.0, 7.5, 8.25],
    "high": [6.5, 7.0, 8.0, 8.0],
    "zero": [0.0, 0.0, 0.0],
    "seam": [0.0, 0.0, 0.5, 19.5, 19.5],
    "spread": [0.0, 0.0, 5.0, 10.0, 15.0, 19.0, 19.0],
    "many": [3.0] * 40 + [4.0] * 40,
}
FORMS = [dict(), dict(stored_p=1), dict(stored_p=3), dict(species=5)]


def step(places, precision, norm=mt.MT_NORM_SYM, batch=False, **form):
    """One step without a walk against the oracle of each realisation."""
    xs = [np.array(PLACES[k])[None, :] for k in places]
    n = sum(x.shape[1] for x in xs)
    p = mt.mt_params_init(n=n, L=(L,), D_rw=0.0, react=0, precision=precision, norm=norm,
                          walls=mt.MT_WALLS_PERIODIC, frac_bits=27, **form)
    b = mt.make_batch([x.shape[1] for x in xs], [L] * len(xs)) if batch else None
    sim = mt.Simulation(p, batch=b)
    species = form.get("species", 2)
    M = [synth.uniform_masses(n, seed=s)[0] for s in range(species)]
    sim.upload(np.concatenate(xs, axis=1), M[0], M[1])
    for s in range(2, species):
        sim.set_species(s, M[s])
    sim.step()
    got = [*sim.masses()] + [sim.species(s) for s in range(2, species)]
    pairs = list(zip(*[v.tolist() for v in sim.pairs()]))
    r = sim.params
    po = O.params(frac_bits=r.frac_bits, L=(L,), D_rw=0.0, smax=r.cutoff, norm=norm, react=0,
                  walls=O.WALLS_PERIODIC)
    sim.close()
    off = 0
    want, wpairs = [[] for _ in M], []
    for x in xs:
        m, X = x.shape[1], O.quantize(x, 27)
        t = O.mass_transfer(po, X, [v[off:off + m] for v in M])
        for s in range(species):
            want[s].append(t[s])
        oi, oj = O.pairs_brute(po, X)
        wpairs += list(zip((oi + off).tolist(), (oj + off).tolist()))
        off += m
    for s in range(species):
        assert_masses(got[s], np.concatenate(want[s]), TOL[precision], f"species {s}")
    assert sorted(pairs) == sorted(wpairs)


@pytest.mark.parametrize("form", FORMS, ids=["walk", "stored", "band3", "tracers"])
@pytest.mark.parametrize("precision", PRECISIONS)
@pytest.mark.parametrize("place", PLACES)
def test_one_system(place, precision, form):
    step([place], precision, **form)
    step([place], precision, norm=mt.MT_NORM_ROW, **form)


@pytest.mark.parametrize("form", FORMS[:2], ids=["walk", "stored"])
@pytest.mark.parametrize("precision", PRECISIONS)
def test_batch(precision, form):
    step(list(PLACES), precision, batch=True, **form)
