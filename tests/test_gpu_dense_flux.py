"""The flux sums of the dense exchange (1-d tiles) at the ends of the masses' range."""
import numpy as np
import pytest

from paper_1811_05474_gb300 import mt, synth

from .test_gpu_parity import PRECISIONS

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("norm", [mt.MT_NORM_SYM, mt.MT_NORM_ROW])
@pytest.mark.parametrize("precision", PRECISIONS)
def test_masses_near_the_largest_number(precision, norm):
    """Masses of 0 and nearly the largest number of the masses' format at 100
    particles per unit length (380 neighbours): the results, weighted means of
    the two, are finite and equal those of the masses scaled by 2^-40.  The
    binary64 sums are within (380 + 2) 2^-53 = 4.3e-14 of the largest mass
    (the sum of a row's weights is about 1), twice that in the difference of
    two; the double-binary32 ones (2^-48 per term) within 380 2^-48 = 1.4e-12."""
    n, L = 3000, 30.0
    top, tol = (3.3e38, 3e-12) if precision == mt.MT_MIXED_DF32 else (1.79e308, 1e-13)
    p = mt.mt_params_init(n=n, L=(L,), D_mt=0.1, D_rw=0.0, dt=1.0, precision=precision, norm=norm,
                          react=0)
    x = synth.uniform_positions(n, L, seed=8)
    g = np.random.default_rng(8)
    A = np.where(g.random(n) < 0.1, 0.0, top)
    B = np.where(g.random(n) < 0.5, 0.0, top)
    out = []
    for scale in (1.0, 2.0 ** -40):
        sim = mt.Simulation(p)
        sim.upload(x, A * scale, B * scale)
        sim.step()
        out.append([m * (2.0 ** -40 / scale) for m in sim.masses()])
        sim.close()
    for big, small in zip(*out):
        assert np.isfinite(big).all()
        assert np.abs(big - small).max() <= tol * top * 2.0 ** -40
