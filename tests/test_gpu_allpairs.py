"""The all-pairs searches' scan with candidate lists (csrc/mt_allpairs.cu)
against the oracle: sizes around its tiles and rows per warp, one and eight
rows per warp, lists that overflow, both walls, one and two dimensions, the
cutoff and the full matrix, tracers, each precision."""
import numpy as np
import pytest

import oracle as O
from paper_1811_05474_gb300 import mt, synth

from .test_gpu_parity import MREF, PRECISIONS, TOL

pytestmark = pytest.mark.gpu


def check(n, L, precision, search, dim=1, walls=0, norm=mt.MT_NORM_SYM, species=2, sample=None,
          cutoff=0.0):
    p = mt.mt_params_init(dim=dim, n=n, L=(L,) * dim, v=(0.3, 0.0), search=search, walls=walls,
                          precision=precision, norm=norm, react=0, species=species, cutoff=cutoff,
                          frac_bits=27)
    sim = mt.Simulation(p)
    r = sim.params
    full = search == mt.MT_SEARCH_FULL
    # sampled rows of the full matrix: the oracle with a cutoff of 6, beyond
    # which the weights (below e^-45) change nothing at these tolerances
    po = O.params(dim=dim, frac_bits=r.frac_bits, L=(L,) * dim, v=(0.3, 0.0),
                  smax=6.0 if full and sample else r.cutoff, norm=norm, react=0, walls=walls,
                  search=O.SEARCH_FULL if full and not sample else O.SEARCH_CUTOFF)
    x = synth.uniform_positions(n, L, dim=dim, seed=n)
    x[:, : n // 50] = x[:, n // 3: n // 3 + n // 50]  # coincident particles
    M = list(synth.uniform_masses(n, seed=n)) + [synth.uniform_masses(n, seed=n + s)[0]
                                                  for s in range(2, species)]
    xi = synth.normals(1, dim, n, seed=n)[0]
    sim.upload(x, M[0], M[1])
    for s in range(2, species):
        sim.set_species(s, M[s])
    sim.set_noise(xi)
    sim.step()
    X = O.move(po, O.quantize(x, int(r.frac_bits)), xi)
    assert np.array_equal(sim.ticks(), X)
    idx = np.arange(n) if sample is None else np.linspace(0, n - 1, sample).astype(np.int64)
    want = (O.mass_transfer_sample(po, X, M, idx) if sample else O.mass_transfer(po, X, M))
    for s in range(species):
        got = (sim.masses()[s] if s < 2 else sim.species(s))[idx]
        err = np.abs(got - want[s]) / np.maximum(np.abs(want[s]), MREF)
        assert err.max() <= TOL[precision], (s, err.max())
    sim.close()


@pytest.mark.parametrize("n", [1, 2, 33, 1023, 1025, 2056])
@pytest.mark.parametrize("precision", PRECISIONS)
@pytest.mark.parametrize("search", [mt.MT_SEARCH_BRUTE, mt.MT_SEARCH_FULL])
def test_sizes(n, precision, search):
    check(n, 200.0 + n, precision, search)


@pytest.mark.parametrize("precision", PRECISIONS)
@pytest.mark.parametrize("search", [mt.MT_SEARCH_BRUTE, mt.MT_SEARCH_FULL])
@pytest.mark.parametrize("dim,walls", [(1, 0), (1, 1), (2, 0), (2, 1)])
def test_eight_rows_per_warp(precision, search, dim, walls):
    n = 19461  # above two CTAs of eight rows per warp on 152 multiprocessors; a ragged last warp
    check(n, float(n) if dim == 1 else 1000.0, precision, search, dim=dim, walls=walls, sample=200)


@pytest.mark.parametrize("precision", PRECISIONS)
@pytest.mark.parametrize("walls", [0, 1])
def test_small_2d_periodic_and_row(precision, walls):
    check(700, 120.0, precision, mt.MT_SEARCH_FULL, dim=2, walls=walls, norm=mt.MT_NORM_ROW)


@pytest.mark.parametrize("precision", PRECISIONS)
@pytest.mark.parametrize("L", [120.0, 30.0])
def test_lists_overflow(precision, L):
    """Hundreds of candidates per row (and, on 30 units, the direct form of
    the binary32 weights)."""
    check(1500, L, precision, mt.MT_SEARCH_FULL)
    check(1500, L, precision, mt.MT_SEARCH_BRUTE, cutoff=5.0)


@pytest.mark.parametrize("precision", PRECISIONS)
def test_tracers(precision):
    check(900, 900.0, precision, mt.MT_SEARCH_FULL, species=5)
