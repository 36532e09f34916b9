"""The all-pairs searches where much of the matrix is nonzero: dense systems and
particles piled at one place, in each of the scan's dispatch bands (one, four
and sixteen rows per warp), against a binary64 matrix formed by torch, and
their time against the same pairs on a small domain."""
import time

import numpy as np
import pytest

from paper_1811_05474_gb300 import mt, synth

from .test_gpu_parity import MREF, PRECISIONS, TOL

pytestmark = pytest.mark.gpu


def bands():
    """Sizes in the bands of one, four and sixteen rows per warp, each with
    several tiles and a ragged last warp."""
    import torch

    sms = torch.cuda.get_device_properties(0).multi_processor_count
    return {1: 32 * sms - 5, 4: 128 * sms - 9, 16: 128 * sms + 7}


def positions(kind, n, L, dim, rng):
    x = rng.uniform(0.0, L, (dim, n))
    if kind == "pile":  # all within a few cutoffs
        x = 0.5 * L + rng.uniform(0.0, 6.0, (dim, n))
    elif kind == "half":  # the first half piled, the rest spread: tiles of both kinds
        x[:, : n // 2] = 0.25 * L + rng.uniform(0.0, 3.0, (dim, n // 2))
    elif kind == "seam":  # across a wall
        x = (rng.uniform(-3.0, 3.0, (dim, n))) % L
    elif kind == "place":  # one point
        x[:] = 0.3 * L
    return x


def reference(X, k, S, L, Ms, norm, periodic, cut, idx):
    """dM of the rows idx by a binary64 matrix, row sums of every particle."""
    import torch

    X = torch.tensor(X, device="cuda")
    Lq = int(round(L * 2.0 ** k))
    n = X.shape[1]

    def weights(rows):
        d2 = torch.zeros((len(rows), n), dtype=torch.float64, device="cuda")
        near = torch.ones((len(rows), n), dtype=torch.bool, device="cuda")
        for a in range(X.shape[0]):
            D = X[a][None, :] - X[a][rows][:, None]
            if periodic:
                D = torch.where(2 * D > Lq, D - Lq, torch.where(2 * D <= -Lq, D + Lq, D))
            d2 += (D.double() * 2.0 ** -k) ** 2
        if cut:
            near = d2 <= (S * 2.0 ** -k) ** 2
        return torch.where(near, torch.exp(-d2 / 0.8), torch.zeros_like(d2))

    r = torch.cat([weights(b).sum(1) for b in torch.arange(n, device="cuda").split(1024)])
    w = weights(idx)
    P = w / r[idx][:, None]
    if norm == mt.MT_NORM_SYM:
        P = 0.5 * (P + w / r[None, :])
    out = []
    for M in Ms:
        M = torch.tensor(M, device="cuda")
        out.append((M[idx] + 0.5 * ((P * M[None, :]).sum(1) - P.sum(1) * M[idx])).cpu().numpy())
    return out


@pytest.mark.parametrize("rows", [1, 4, 16])
@pytest.mark.parametrize("precision", PRECISIONS)
@pytest.mark.parametrize("kind,dim,walls,search,norm,species", [
    ("pile", 1, 0, mt.MT_SEARCH_FULL, mt.MT_NORM_SYM, 2),
    ("pile", 1, 0, mt.MT_SEARCH_BRUTE, mt.MT_NORM_ROW, 2),
    ("half", 1, 0, mt.MT_SEARCH_FULL, mt.MT_NORM_ROW, 5),
    ("half", 2, 0, mt.MT_SEARCH_BRUTE, mt.MT_NORM_SYM, 2),
    ("seam", 1, 1, mt.MT_SEARCH_BRUTE, mt.MT_NORM_SYM, 3),
    ("seam", 2, 1, mt.MT_SEARCH_FULL, mt.MT_NORM_SYM, 2),
    ("place", 2, 0, mt.MT_SEARCH_FULL, mt.MT_NORM_ROW, 2),
    ("spread", 1, 1, mt.MT_SEARCH_FULL, mt.MT_NORM_ROW, 4),
    ("spread", 2, 0, mt.MT_SEARCH_BRUTE, mt.MT_NORM_SYM, 2),
])
def test_against_a_matrix(kind, dim, walls, search, norm, species, precision, rows):
    import torch

    n = bands()[rows]
    L = 1000.0 if kind != "spread" else (n / 4.0 if dim == 1 else 300.0)
    rng = np.random.default_rng(n + dim)
    x = positions(kind, n, L, dim, rng)
    M = [rng.uniform(0.0, 1.0, n) for _ in range(species)]
    p = mt.mt_params_init(dim=dim, n=n, L=(L,) * dim, D_rw=0.0, search=search, walls=walls,
                          precision=precision, norm=norm, react=0, species=species, frac_bits=27)
    sim = mt.Simulation(p)
    sim.upload(x, M[0], M[1])
    for s in range(2, species):
        sim.set_species(s, M[s])
    X = sim.ticks()
    sim.step()
    got = [*sim.masses()] + [sim.species(s) for s in range(2, species)]
    S = int(np.floor(np.ldexp(sim.params.cutoff, 27)))
    sim.close()
    idx = torch.unique(torch.cat([torch.linspace(0, n - 1, 200, device="cuda").long(),
                                  torch.arange(n - 70, n, device="cuda")]))
    want = reference(X, 27, S, L, M, norm, walls == 1, search == mt.MT_SEARCH_BRUTE, idx)
    for s in range(species):
        err = np.abs(got[s][idx.cpu().numpy()] - want[s]) / np.maximum(np.abs(want[s]), MREF)
        assert err.max() <= TOL[precision], (s, err.max())


@pytest.mark.parametrize("precision", [mt.MT_MIXED, mt.MT_MIXED_DF32])
@pytest.mark.parametrize("n", [8000, 20000, 50000])
def test_a_pile_costs_no_more_than_its_pairs(n, precision):
    """The same positions, all within 20 units, on a domain of 20 units and on one
    of n: the same nonzero weights, so the same time (a quarter is allowed)."""
    x = 20.0 * np.random.default_rng(3).random((1, n))
    A, B = synth.uniform_masses(n, seed=3)
    took = []
    for L in (20.0, float(n)):
        p = mt.mt_params_init(n=n, L=(L,), D_rw=0.0, search=mt.MT_SEARCH_FULL, precision=precision,
                              frac_bits=27)
        sim = mt.Simulation(p)
        sim.upload(x, A, B)
        sim.run(2)
        sim.sync()
        best = float("inf")
        for _ in range(3):
            t = time.perf_counter()
            sim.run(2)
            sim.sync()
            best = min(best, time.perf_counter() - t)
        took.append(best)
        sim.close()
    assert took[1] <= 1.25 * took[0], took
