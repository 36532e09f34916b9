"""MT_MIXED's flux sums in exact integer arithmetic (csrc/mt_fixed.cuh): the
recipe replayed on Python integers against exact rationals, and the library
on the GPU against a binary64 reference for masses over many decades, of both
signs, zero, near the ends of binary64's range, infinite and NaN, in the
sparse (one-kernel step) and the dense (tiled) exchange."""
import math
import pathlib
import random
import re
import struct
from fractions import Fraction

import numpy as np
import pytest

from paper_1811_05474_gb300 import mt, synth

M64 = 2 ** 64 - 1


def bits(x):
    return struct.unpack("<Q", struct.pack("<d", x))[0]


def exponent(b):
    return (b >> 52) & 0x7FF


def to_fix(b, E):
    e = exponent(b)
    m = ((b & (2 ** 52 - 1)) | ((1 if e else 0) << 52)) << 8
    sh = E - (e if e else 1)
    v = m >> min(sh, 63) if sh < 64 else 0
    if sh > 7 and m:
        lost = sh >= 63 or (v << sh) & M64 != m or v & 1
        v = (v & ~1) | (1 if lost else 0)
    return -v if b >> 63 else v


def fix_p(P):
    u = struct.unpack("<I", struct.pack("<f", P))[0]
    return ((u & 0x7FFFFF) | 0x800000) << 7, 128 - (u >> 23)


def wrap96(v):
    v &= 2 ** 96 - 1
    return v - 2 ** 96 if v >> 95 else v


def value(acc, E):
    a = abs(acc)
    if a == 0:
        return 0.0
    t = a.bit_length() - 1
    top96 = a << (95 - t)
    top = (top96 >> 32) | (1 if top96 & 0xFFFFFFFF else 0)
    q = ((top + 0x3FF + ((top >> 11) & 1)) & M64) >> 11
    mant = q | (2 ** 53 if top > 0xFFFFFFFFFFFFFBFF else 0)
    b = ((((t + E - 90) << 52) + mant) & M64) | ((1 if acc < 0 else 0) << 63)
    return struct.unpack("<d", struct.pack("<Q", b))[0]


@pytest.mark.parametrize("kind", ["near", "decades", "signed", "smooth"])
def test_replay_is_no_less_exact_than_binary64(kind):
    """For the rows the integer form takes: its error is one rounding of the
    sum, a unit 2^(E - 1083) for each marked mass times its P, and a 2^-29 unit
    per term (the shift); the mean square of the errors relative to the row's
    largest term is below that of the binary64 form (a difference and a fused
    multiply-add per term)."""
    rng = random.Random(5)
    err = {"fix": [], "f64": []}
    for _ in range(4000):
        c = rng.randrange(1, 12)
        M = [rng.random() for _ in range(c + 1)]
        if kind != "near":
            M = [m * 10 ** rng.uniform(-4, 0) for m in M]
        if kind == "signed":
            M = [m * rng.choice([1, -1]) for m in M]
        if kind == "smooth":
            M = [0.7 + 1e-9 * m for m in M]
        else:
            M = [0.0 if rng.random() < 0.4 else m for m in M]
        P = [float(np.float32(math.exp(-rng.uniform(0, 4.5)) / rng.uniform(1, 20)))
             for _ in range(c)]
        E = exponent(bits(max([abs(m) for m in M] + [0.9 * rng.random()])))
        f = [to_fix(bits(m), E) for m in M]
        size = 0
        for v in f:
            h = (v >> 32) & 0xFFFFFFFF
            size |= h ^ (0xFFFFFFFF if v < 0 else 0)
        if any(v & 1 for v in f) and not size >> 26:
            continue  # summed in binary64
        acc, ref, exact, largest = 0, 0.0, Fraction(0), 0.0
        for i in range(c):
            p, s = fix_p(P[i])
            acc = wrap96(acc + ((f[i + 1] - f[0]) * p >> s))
            ref = float(Fraction(P[i]) * Fraction(M[i + 1] - M[0]) + Fraction(ref))
            term = Fraction(P[i]) * (Fraction(M[i + 1]) - Fraction(M[0]))
            exact += term
            largest = max(largest, abs(float(term)))
        if largest == 0.0:
            assert acc == 0
            continue
        unit = Fraction(2) ** (E - 1083)
        bound = Fraction(2) ** -53 * abs(exact) + c * unit / 2 ** 29
        bound += sum(Fraction(P[i]) * ((f[i + 1] & 1) + (f[0] & 1)) * unit for i in range(c))
        assert abs(Fraction(value(acc, E)) - exact) <= bound * Fraction(1001, 1000)
        err["fix"].append(abs(float(Fraction(value(acc, E)) - exact)) / largest)
        err["f64"].append(abs(float(Fraction(ref) - exact)) / largest)
    assert np.mean(np.square(err["fix"])) <= max(np.mean(np.square(err["f64"])), 2.0 ** -108)


def test_smallest_weights_stay_in_the_shift():
    """The dispatch's bound on the weights and on a realisation's particles
    keeps P's shift below a word's 32 bits, down to the row normalisation's
    smallest P (a far neighbour of all the others at one place)."""
    src = (pathlib.Path(mt.__file__).parent / "csrc" / "mt_api.cu").read_text()
    limit = float(re.search(r"d\.fix = .* <= ([0-9.]+) \?", src).group(1))
    most = 1 << int(re.search(r"R\.n > \(1LL << (\d+)\)\) d\.fix", src).group(1))
    P = math.exp(-limit) * (1 - 1e-5) / most  # (binary32 rounding: < 1e-6)
    assert 0 <= fix_p(P)[1] <= 31


def masses(kind, n, g):
    m = g.uniform(0.0, 1.0, n)
    if kind == "decades":
        m *= 10.0 ** g.uniform(-25, 0, n)
    elif kind == "signed":
        m *= 10.0 ** g.uniform(-6, 0, n) * g.choice([1.0, -1.0], n)
    elif kind == "spike":  # nearly all tiny or zero, a few of order one
        m = np.where(g.random(n) < 0.5, 0.0, 1e-13 * m)
        m[:: n // 7] = 1.0
    elif kind == "zeros":
        m[:] = 0.0
    elif kind == "huge":
        m *= 1e306
    elif kind == "tiny":
        m *= 1e-290
    elif kind == "smooth":
        m = 0.7 + 1e-9 * m
    elif kind == "inf":
        m[n // 3] = np.inf
        m[2 * n // 3] = np.nan
    return m


@pytest.mark.gpu
@pytest.mark.parametrize("L", [2000.0, 30.0])
@pytest.mark.parametrize("norm", [mt.MT_NORM_SYM, mt.MT_NORM_ROW])
@pytest.mark.parametrize("kind", ["unit", "decades", "signed", "spike", "zeros", "huge", "tiny",
                                  "smooth", "inf"])
def test_exchange_on_the_gpu(kind, norm, L):
    """One transfer without walk or reaction against a dense binary64 matrix.
    Bound per particle: binary32 weights and row sums are within 2^-20 of the
    exact ones (an exponential, up to 500 compensated terms, a reciprocal and
    two products of 2^-24 each), relative to the sum of the terms' magnitudes,
    plus the update's rounding."""
    n = 2000
    p = mt.mt_params_init(n=n, L=(L,), D_rw=0.0, react=0, norm=norm, precision=mt.MT_MIXED)
    sim = mt.Simulation(p)
    g = np.random.default_rng(11)
    x = synth.uniform_positions(n, L, seed=3)
    A, B = masses(kind, n, g), masses("unit", n, g)
    sim.upload(x, A, B)
    X = sim.ticks()[0]
    sim.step()
    k, S = int(sim.params.frac_bits), math.floor(math.ldexp(sim.params.cutoff, int(sim.params.frac_bits)))
    D = X[None, :] - X[:, None]
    w = np.where(np.abs(D) <= S, np.exp(-(D * 2.0 ** -k) ** 2 / 0.8), 0.0)
    r = w.sum(1)
    P = w / r[:, None] if norm == mt.MT_NORM_ROW else 0.5 * (w / r[:, None] + w / r[None, :])
    for M, got in zip((A, B), sim.masses()):
        with np.errstate(invalid="ignore", over="ignore"):
            terms = np.where(P > 0, P * (M[None, :] - M[:, None]), 0.0)
            np.fill_diagonal(terms, 0.0)
            want = M + 0.5 * terms.sum(1)
            tol = 2.0 ** -20 * 0.5 * np.abs(terms).sum(1) + 2.0 ** -51 * np.abs(M) + 1e-320
        ok = np.isfinite(want)
        off = np.abs(np.where(ok, got, 0.0) - np.where(ok, want, 0.0))
        assert np.array_equal(np.isnan(want), np.isnan(got))
        assert np.array_equal(want[~ok & ~np.isnan(want)], got[~ok & ~np.isnan(want)])
        assert np.all(off[ok] <= tol[ok]), np.max(off[ok] / tol[ok])
    sim.close()


@pytest.mark.gpu
@pytest.mark.parametrize("norm", [mt.MT_NORM_SYM, mt.MT_NORM_ROW])
@pytest.mark.parametrize("precision", [mt.MT_FP64, mt.MT_MIXED])
def test_masses_near_the_largest_binary64(precision, norm):
    """One-kernel step with masses of 0 and 1.79e308: the results, weighted
    means of the two, are finite, and equal those of the masses scaled by
    2^-40 (sums of at most ~30 terms in binary64, or in integers: within
    1e-13 of the largest mass)."""
    n, L = 3000, 1000.0
    p = mt.mt_params_init(n=n, L=(L,), D_mt=0.1, D_rw=0.0, dt=1.0, precision=precision, norm=norm,
                          react=0)
    x = synth.uniform_positions(n, L, seed=8)
    g = np.random.default_rng(8)
    A = np.where(g.random(n) < 0.1, 0.0, 1.79e308)
    B = np.where(g.random(n) < 0.5, 0.0, 1.79e308)
    out = []
    for scale in (1.0, 2.0 ** -40):
        sim = mt.Simulation(p)
        sim.upload(x, A * scale, B * scale)
        sim.step()
        out.append([m * (2.0 ** -40 / scale) for m in sim.masses()])
        sim.close()
    for big, small in zip(*out):
        assert np.isfinite(big).all()
        assert np.abs(big - small).max() <= 1e-13 * 1.79e308 * 2.0 ** -40
