"""The binary64 weights within the cutoff (Eq. 3), evaluated with 64-bit
integer arithmetic from the exact squared separation (exp_fix in
csrc/mt_pair.cuh): the table and the polynomial against 200-bit evaluations,
the recipe replayed on integers, and the weights the library applies on the
GPU, read back through the exchange of two particles."""
import math
import random
import re
from pathlib import Path

import numpy as np
import pytest

from paper_1811_05474_gb300 import mt

mp = pytest.importorskip("mpmath")
SRC = Path(__file__).resolve().parents[1] / "paper_1811_05474_gb300" / "csrc" / "mt_pair.cuh"
M64 = 2 ** 64 - 1


def table_and_coefficients():
    text = SRC.read_text()
    body = re.search(r"kExp2Neg\[256\] = \{(.*?)\};", text, re.S).group(1)
    tab = [int(v, 16) for v in re.findall(r"0x([0-9a-f]+)ull", body)]
    b = [int(re.search(rf"kExpB{i} = 0x([0-9a-f]+)u", text).group(1), 16) for i in range(1, 5)]
    return tab, b


def constants(inv8, k, S):
    """exp_constants (csrc/mt_api.cu): (ec, eq, eib)."""
    a = math.ldexp(inv8, -2 * k)
    R = min(S * S, int(746.0 / a))
    q = 64 - R.bit_length()
    ib = 1
    while 2.0 ** (ib - 1) <= R * a * 1.4426950408889634 * (1 + 1e-9):
        ib += 1
    m, e = math.frexp(inv8)
    P, sh = int(m * 2 ** 53) * 0xB8AA3B295C17F0BC, e - 53 - 2 * k - 63 + 128 - ib - q
    ec = P << sh if sh >= 0 else (P + (1 << (-sh - 1))) >> -sh
    assert ec <= M64
    return ec, q, ib


def replay(R2, ec, q, ib, tab, b):
    """(mantissa, m): the weight is mantissa 2^-53 2^-m."""
    V = ((R2 << q) * ec) >> 64
    m, F = V >> (64 - ib), (V << ib) & M64
    X = (F << 8) & M64
    xh = X >> 32
    t3 = b[2] - ((xh * b[3]) >> 32)
    t2 = b[1] - ((xh * t3) >> 32)
    t1 = b[0] - (((X * t2) >> 64) << 4)
    r = tab[F >> 56] - ((tab[F >> 56] * ((X * t1) >> 64)) >> 64)
    return (r + 512) >> 10, m


def test_table_and_polynomial():
    mp.mp.prec = 200
    tab, b = table_and_coefficients()
    assert len(tab) == 256
    for j, t in enumerate(tab):
        assert t == int(mp.nint(mp.mpf(2) ** (63 - mp.mpf(j) / 256))), j
    for i in range(257):  # 1 - 2^(-x/256) on [0, 1]
        x = mp.mpf(i) / 256
        p = x * (b[0] / mp.mpf(2) ** 64 - x * (b[1] - x * (b[2] - x * b[3])) / mp.mpf(2) ** 60)
        assert abs(p - (1 - mp.mpf(2) ** (-x / 256))) < mp.mpf(2) ** -56


@pytest.mark.parametrize("D,dt,cutoff", [(0.1, 1.0, 0.0), (0.5, 0.1, 0.0), (0.1, 1.0, 20.0),
                                         (3.0, 7.0, 0.01), (0.01, 0.1, 0.9)])
def test_replay_is_within_1_2_half_units(D, dt, cutoff):
    mp.mp.prec = 200
    tab, b = table_and_coefficients()
    p = mt.mt_resolve(mt.mt_params_init(n=10, L=(100.0,), D_mt=D, dt=dt, cutoff=cutoff))
    k, inv8 = p.frac_bits, 1.0 / (8.0 * D * dt)
    S = math.floor(math.ldexp(p.cutoff, k))
    c = constants(inv8, k, S)
    rng = random.Random(1)
    # truncation 2^-56, the product's and the exponent's last bits (frac bits
    # 64 - eib, at least 53 for exponents below 2^10), the final rounding 2^-53
    tol = mp.mpf(2) ** -53 * (1 + mp.mpf(2) ** -2) + mp.mpf(2) ** (c[2] - 64)
    for d in [0, 1, S, S - 1] + [rng.randrange(S) for _ in range(2000)]:
        q, m = replay(d * d, *c, tab, b)
        assert 2 ** 52 <= q <= 2 ** 53
        exact = mp.e ** (-mp.mpf(d) ** 2 * mp.mpf(inv8) * mp.mpf(2) ** (-2 * k))
        assert abs(q * mp.mpf(2) ** (-53 - m) - exact) <= tol * exact, d
    assert replay(0, *c, tab, b) == (2 ** 53, 0)  # coincident particles: exactly 1


@pytest.mark.gpu
@pytest.mark.parametrize("dim", [1, 2])
@pytest.mark.parametrize("cutoff", [0.0, 12.0, 40.0])
def test_weights_on_the_gpu(dim, cutoff):
    """Pairs of particles with masses 0 and 1: after one transfer without walk
    or reaction the first holds w / (1 + w) / 2.  Its relative error is the
    weight's (the replay's bound above) plus the row sum's, the reciprocal's,
    the normalisation's and the exchange's roundings: 8 2^-53 in all."""
    mp.mp.prec = 200
    pairs, L = 64, 400.0
    p = mt.mt_params_init(dim=dim, n=2 * pairs, L=(L * pairs, L), D_rw=0.0, cutoff=cutoff, react=0)
    sim = mt.Simulation(p)
    k, smax = int(sim.params.frac_bits), sim.params.cutoff
    inv8 = 1.0 / (8.0 * 0.1)
    g = np.random.default_rng(3)
    s = np.concatenate([[0.0, smax * (1 - 1e-6)], g.uniform(0, smax, pairs - 2)])
    a = g.uniform(0, 2 * np.pi, pairs) if dim == 2 else np.zeros(pairs)
    x0 = L * np.arange(pairs) + 100.0
    x = np.stack([np.concatenate([x0, x0 + s * np.cos(a)]),
                  np.concatenate([np.full(pairs, 200.0), 200.0 + s * np.sin(a)])])[:dim]
    A = np.concatenate([np.zeros(pairs), np.ones(pairs)])
    sim.upload(x, A, A)
    X = sim.ticks()
    sim.step()
    got = sim.masses()[0][:pairs]
    for i in range(pairs):
        R2 = sum(int(X[c, pairs + i] - X[c, i]) ** 2 for c in range(dim))
        t = mp.mpf(R2) * mp.mpf(inv8) * mp.mpf(2) ** (-2 * k)
        w = mp.e ** -t if R2 <= math.floor(math.ldexp(smax, k)) ** 2 else mp.mpf(0)
        want = w / (1 + w) / 2
        if t < 700:
            assert abs(mp.mpf(float(got[i])) - want) <= 8 * mp.mpf(2) ** -53 * want, (i, t)
        else:  # below the normal range
            assert abs(got[i] - float(want)) <= 1e-300
    sim.close()
