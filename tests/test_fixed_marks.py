"""Small masses beside large ones in MT_MIXED's integer flux sums
(csrc/mt_fixed.cuh): which rows the integers take and how exact those are, the
recipe replayed on Python integers, and the library on the GPU by linearity."""
import math
import random
from fractions import Fraction

import numpy as np
import pytest

from paper_1811_05474_gb300 import mt, synth

from .test_fixed_flux import bits, exponent, fix_p, value, wrap96


def to_fix(b, E):
    e = exponent(b)
    m = ((b & (2 ** 52 - 1)) | ((1 if e else 0) << 52)) << 8
    sh = E - (e if e else 1)
    v = m >> min(sh, 63)
    if sh > 7 and m and (sh > 16 or v << sh != m):
        v |= 1
    return -v if b >> 63 else v


def fix_rest(b, E):
    e = exponent(b)
    m = ((b & (2 ** 52 - 1)) | ((1 if e else 0) << 52)) << 8
    sh = E - (e if e else 1)
    if sh <= 7 or not m:
        return np.float32(0.0)
    v, f = m >> min(sh, 63), np.float32(0.0)
    if sh < 64:
        f = np.float32(m << (64 - sh) >> 32 & 0xFFFFFFFF) * np.float32(2.0 ** -32)
    elif sh < 150:
        f = np.float32(m >> 32) * np.float32(2.0 ** (32 - sh))
    if not v & 1 and (sh > 16 or v << sh != m):
        f -= np.float32(1.0)
    return -f if b >> 63 else f


@pytest.mark.parametrize("E", [1023, 1400])
def test_rests(E):
    """A mass is its integer and its rest, to 2^-24 of the unit."""
    rng = random.Random(2)
    u = Fraction(2) ** (E - 1083)
    for _ in range(4000):
        x = math.ldexp(rng.choice([rng.random(), rng.randrange(1, 64) / 64.0]),
                       E - 1022 - rng.randrange(0, 100)) * rng.choice([1, -1])
        b = bits(x)
        if exponent(b) > E:
            continue
        rest = fix_rest(b, E)
        assert abs(rest) <= 1.0
        assert abs(Fraction(x) / u - to_fix(b, E) - Fraction(float(rest))) <= Fraction(2) ** -24


@pytest.mark.parametrize("kind", ["edge", "decades", "signed", "clean", "smooth", "zeros"])
def test_kept_rows_are_as_exact_as_one_rounding(kind):
    """Rows of up to 200 neighbours with a large mass at the cutoff's edge, with
    masses over 30 decades, of both signs, with few significant bits, and nearly
    equal ones: where the integer sum is kept, the new mass M' is within its rests'
    error (2^-15 of a unit for up to 512 terms) and the terms' (2^-30 of one each),
    together at most 2^-53 M' (1 + 2^-5), and the sum's and the update's rounding
    (2^-53 each of |M'| and the sum)."""
    rng = random.Random(7)
    kept = 0
    for _ in range(400):
        c = rng.choice([2, 10, 200])
        M = [rng.random() for _ in range(c + 1)]
        P = [math.exp(-rng.uniform(0, 1)) / (c + 1) for _ in range(c)]
        if kind == "edge":
            M = [m * 1e-6 for m in M]
            M[1], P[0] = 0.9, math.exp(-rng.uniform(0, 6.9)) / (c + 1)
        elif kind == "decades":
            M = [m * 10 ** rng.uniform(-30, 0) for m in M]
        elif kind == "signed":
            M = [m * 10 ** rng.uniform(-6, 0) * rng.choice([1, -1]) for m in M]
        elif kind == "clean":
            M = [rng.randrange(1, 64) * 2.0 ** rng.choice([-57, -20, -6]) for _ in M]
        elif kind == "zeros":
            tiny = 1e-17 * rng.random()
            M = [0.0 if rng.random() < 0.99 else tiny for _ in M]
        else:
            M = [0.7 + 1e-9 * m for m in M]
        P = [float(np.float32(p)) for p in P]
        top = 1.0 if rng.random() < 0.5 else max(abs(m) for m in M)  # another staged mass
        E = exponent(bits(max(top, max(abs(m) for m in M)))) or 1023
        f = [to_fix(bits(m), E) for m in M]
        rest = [fix_rest(bits(m), E) for m in M]
        acc, sum_rest = 0, np.float32(0.0)
        for i in range(c):
            p, s = fix_p(P[i])
            acc = wrap96(acc + ((f[i + 1] - f[0]) * p >> s))
            sum_rest = np.float32(P[i] * float(rest[i + 1] - rest[0]) + float(sum_rest))
        acc = wrap96(acc + round(float(sum_rest) * 2.0 ** 29))
        exact = sum(Fraction(P[i]) * (Fraction(M[i + 1]) - Fraction(M[0])) for i in range(c))
        total = value(acc, E)
        new = M[0] + 0.5 * total
        size = abs((f[0] >> 3) + (acc >> 33))  # |M'| in units of 8 u
        zero = f[0] == 0 and acc == 0 and min(f) >= 0  # (P is at least 2^-18 here)
        if size < 2 ** 35 and not zero:
            continue  # summed in binary64
        kept += 1
        bound = Fraction(2) ** -53 * (2 * abs(Fraction(new)) + abs(exact)) * Fraction(33, 32)
        assert abs(Fraction(new) - (Fraction(M[0]) + exact / 2)) <= bound
    assert kept > 20


def large(n):
    m = np.zeros(n)
    m[n // 5:: n // 5] = 0.9
    return m


@pytest.mark.gpu
@pytest.mark.parametrize("L", [2000.0, 10.0])
@pytest.mark.parametrize("norm", [mt.MT_NORM_SYM, mt.MT_NORM_ROW])
@pytest.mark.parametrize("kind", ["generic", "few bits"])
def test_small_masses_beside_large_ones(kind, norm, L):
    """Small masses with a few large ones among them (species A), the small ones
    alone (B), and, in a second run, the large ones alone: the same weights, so
    the first result is the sum of the others.  Two of the three sums are of
    terms that are exact or far smaller; the first one's binary64 roundings, one
    per term (up to 930), within half a unit of the partial sums, 2^-53 of the
    terms' total T, and independent, have a root mean square of at most
    sqrt(930 / 3) 2^-53 T = 17.6 2^-53 T, and its update and the others' less
    than two more: 20.  Rows with a large mass near the cutoff, where its weight
    is least, and rows with none, each on their own."""
    n = 2000
    p = mt.mt_params_init(n=n, L=(L,), D_rw=0.0, react=0, norm=norm, precision=mt.MT_MIXED,
                          cutoff=2.34)
    g = np.random.default_rng(4)
    x = synth.uniform_positions(n, L, seed=4)
    big = np.zeros(n)
    big[np.argsort(x[0])[[n // 5, n // 2]]] = 0.9
    small = 1e-9 * g.random(n) if kind == "generic" else 2.0 ** -59 * g.integers(1, 64, n)
    small[big > 0] = 0.0
    out = []
    for A in (small + big, big):
        sim = mt.Simulation(p)
        sim.upload(x, A, small)
        X = sim.ticks()[0]
        sim.step()
        out.append(sim.masses())
        k = int(sim.params.frac_bits)
        S = math.floor(math.ldexp(sim.params.cutoff, k))
        sim.close()
    (both, alone), (large, _) = out
    D = X[None, :] - X[:, None]
    w = np.where(np.abs(D) <= S, np.exp(-(D * 2.0 ** -k) ** 2 / 0.8), 0.0)
    r = w.sum(1)
    P = w / r[:, None] if norm == mt.MT_NORM_ROW else 0.5 * (w / r[:, None] + w / r[None, :])
    A = small + big
    T = A + 0.5 * (P * np.abs(A[None, :] - A[:, None])).sum(1)
    off = np.abs(both - (alone + large)) / (2.0 ** -53 * T)
    nearest = np.where(big[None, :] > 0, w, 0.0).max(1)
    for rows in (nearest == 0, (nearest > 0) & (nearest < math.exp(-5.5 if L < 100 else -1))):
        assert rows.any()
        assert np.sqrt(np.mean(off[rows] ** 2)) <= 20
