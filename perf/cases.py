"""What a user of this library has it compute, as cases that can be timed and checked.

A pass is what a program does with a handle it keeps: load a state, advance it
some time steps, read the state back (and the observables where it tracks
them).  The sizes are those of the benchmark's and the tests' workloads:
uniform particles at one per unit length (1-d) or on [0, 10 sqrt(N)]^2 (2-d),
the paper's densities, its full-matrix form, ensembles and served requests.
"""
import math
import random

import numpy as np
import torch

from paper_1811_05474_gb300 import mt, synth

PREC = {"fp64": mt.MT_FP64, "mixed": mt.MT_MIXED, "df32": mt.MT_MIXED_DF32}
SEARCH = {"cell": mt.MT_SEARCH_CELL, "full": mt.MT_SEARCH_FULL}


def _system(**kw):
    """One system; every field of a case of this kind, with its usual value."""
    c = dict(kind="system", dim=1, n=1000, L=0.0, search="cell", precision="fp64", v=0.0,
             D=0.1, dt=1.0, norm="sym", walls="reflect", species=2, react=True, elapsed=0,
             observe=False, steps=100)
    c.update(kw)
    if not c["L"]:  # one particle per unit length, or per 100 units of area
        c["L"] = float(c["n"]) if c["dim"] == 1 else 10.0 * math.sqrt(c["n"])
    return c


def _dense(**kw):
    """The paper's own densities (Sec. 3, Sec. 6): D split between transfer and
    walk, no reaction (conservative components), hundreds of neighbours."""
    return _system(D=0.5, dt=0.1, react=False, **kw)


def listed():
    return [
        # the smallest simulation, 100 steps: launches and latency are what it costs
        dict(_system(n=1000, steps=100), name="cell_1e3_fp64"),
        # the same system with the paper's full matrix, its reference form
        dict(_system(n=1000, search="full", steps=20), name="full_1e3_fp64"),
        # an ordinary 1-d simulation in binary64
        dict(_system(n=100000, steps=50), name="cell_1e5_fp64"),
        # the headline workload in the middle of its run: drift, the layer at the wall,
        # mean A tracked
        dict(_system(n=1000000, precision="mixed", v=0.5, elapsed=500, observe=True, steps=40),
             name="cell_1e6_mixed"),
        # an odd size with the literal row normalisation in the fast binary32 variant
        dict(_system(n=300007, L=330001.5, precision="df32", norm="row", steps=40),
             name="cell_3e5_df32"),
        # an ensemble of 256 uneven realisations advanced together
        dict(kind="batch", count=256, n_lo=1000, n_hi=100000, per_length=1.0, D=0.1, dt=1.0,
             precision="mixed", react=True, observe=True, steps=10, sizes=0, name="batch_256_mixed"),
        # the paper's accuracy problem: 75 realisations on [0, 50]
        dict(kind="batch", count=75, n_lo=5000, n_hi=5000, per_length=100.0, D=0.5, dt=0.1,
             precision="fp64", react=False, observe=False, steps=5, sizes=0,
             name="ensemble_75_fp64"),
        # the paper's density at its largest size (Sec. 6: 10^6 particles on [0, 5000])
        dict(_dense(n=1000000, L=5000.0, precision="mixed", steps=5), name="dense_1e6_mixed"),
        # a 2-d system of a served request's shape
        dict(_system(dim=2, n=1000000, precision="mixed", steps=20), name="cell2d_1e6_mixed"),
        # tracers beside the reaction on a periodic domain (multi-kernel pipeline)
        dict(_system(n=400009, precision="mixed", walls="periodic", species=4, v=0.5, steps=20),
             name="tracers_4e5_periodic"),
        # the full matrix at the largest size the paper quotes it for
        dict(_system(n=100000, search="full", precision="mixed", steps=1), name="full_1e5_mixed"),
        # served requests of mixed sizes and dimensions, host arrays in and out
        dict(kind="serve", requests=10, n_lo=1000, n_hi=1000000, steps_lo=25, steps_hi=100,
             precision="mixed", sizes=1, name="serve_10_mixed"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """A case of the same ranges: 1-d and 2-d cell lists, the full matrix, dense
    systems, tracers, ensembles and requests."""
    prec = rng.choice(["fp64", "mixed", "mixed", "df32"])
    norm = rng.choice(["sym", "sym", "sym", "row"])
    k = rng.choice(["cell", "cell", "cell", "cell2d", "cell2d", "full", "dense", "tracers",
                    "batch", "ensemble", "serve"])
    if k == "cell":
        n = _log(rng, 1000, 1000000)
        v = rng.choice([0.0, 0.5])
        return _system(n=n, L=round(n * rng.uniform(0.8, 1.3), 3), precision=prec, norm=norm, v=v,
                       elapsed=rng.randrange(0, 1000) if v else 0, observe=rng.random() < 0.5,
                       steps=rng.randrange(10, 60))
    if k == "cell2d":
        n = _log(rng, 1000, 1000000)
        return _system(dim=2, n=n, precision=prec, norm=norm, v=rng.choice([0.0, 0.5]),
                       walls=rng.choice(["reflect", "reflect", "periodic"]),
                       observe=rng.random() < 0.5, steps=rng.randrange(5, 20))
    if k == "full":
        n = _log(rng, 1000, 60000)
        prec = prec if n < 4000 else rng.choice(["mixed", "df32"])
        return _system(n=n, search="full", precision=prec, norm=norm,
                       steps=1 if n >= 4000 else rng.randrange(1, 12))
    if k == "dense":
        n = _log(rng, 20000, 1000000)
        return _dense(n=n, L=round(n / rng.uniform(40.0, 200.0), 3), norm=norm,
                      precision=rng.choice(["mixed", "mixed", "df32", "fp64"] if n < 300000 else
                                           ["mixed", "df32"]),
                      steps=rng.randrange(1, 5))
    if k == "tracers":
        return _system(n=_log(rng, 1000, 400000), precision=prec, species=rng.randrange(2, 9),
                       walls=rng.choice(["reflect", "periodic"]), v=rng.choice([0.0, 0.5]),
                       steps=rng.randrange(5, 20))
    if k == "batch":
        return dict(kind="batch", count=rng.randrange(8, 200), n_lo=1000,
                    n_hi=_log(rng, 2000, 100000), per_length=1.0, D=0.1, dt=1.0, precision=prec,
                    react=True, observe=rng.random() < 0.5, steps=rng.randrange(2, 10),
                    sizes=rng.randrange(1 << 20))
    if k == "ensemble":
        n = rng.choice([500, 1000, 2500, 5000])
        return dict(kind="batch", count=rng.randrange(10, 76), n_lo=n, n_hi=n,
                    per_length=n / 50.0, D=0.5, dt=0.1, precision=rng.choice(["fp64", "mixed"]),
                    react=False, observe=False, steps=rng.randrange(1, 5),
                    sizes=rng.randrange(1 << 20))
    return dict(kind="serve", requests=rng.randrange(3, 11), n_lo=1000,
                n_hi=_log(rng, 10000, 1000000), steps_lo=25, steps_hi=60, precision=prec,
                sizes=rng.randrange(1 << 20))


# ---------------------------------------------------------------- inputs --

def _sizes(case):
    """A batch's (n, L) per realisation."""
    rng = random.Random(case["sizes"])
    lo, hi = case["n_lo"], case["n_hi"]
    ns = [lo if lo == hi else _log(rng, lo, hi) for _ in range(case["count"])]
    return ns, [n / case["per_length"] for n in ns]


def _requests(case):
    """The served requests as system cases."""
    rng = random.Random(case["sizes"])
    out = []
    for _ in range(case["requests"]):
        out.append(_system(dim=rng.choice([1, 2]), n=_log(rng, case["n_lo"], case["n_hi"]),
                           precision=case["precision"], observe=True,
                           steps=rng.randrange(case["steps_lo"], case["steps_hi"] + 1)))
    return out


def _uniform(seed, stream, *shape):
    g = torch.Generator(device="cuda")
    g.manual_seed((int(seed) * 1000003 + stream) & (2**62 - 1))
    return torch.rand(shape, generator=g, device="cuda", dtype=torch.float64)


def _inputs(case, seed):
    """x (dim, n) and the masses (species, n) of a system on the GPU: uniform,
    or as a run with drift has them after `elapsed` steps (particles that
    reached the wall in a layer D / v thick, one reactant left per particle)."""
    n, L = case["n"], case["L"]
    x = _uniform(seed, 1, case["dim"], n) * L
    M = _uniform(seed, 2, case["species"], n)
    if case["elapsed"]:
        t = case["elapsed"] * case["dt"]
        x += case["v"] * t
        layer = L + torch.log(1.0 - _uniform(seed, 3, case["dim"], n)) * (case["D"] / case["v"])
        x = torch.where(x > L, layer, x).clamp_(0.0, L)
        left = (M[0] - M[1]) * (1.0 + t) ** -0.25
        M[0], M[1] = left.clamp(min=0.0), (-left).clamp(min=0.0)
    return x, M


def _batch_inputs(case, seed):
    ns, Ls = _sizes(case)
    per = torch.repeat_interleave(torch.tensor(Ls, dtype=torch.float64, device="cuda"),
                                  torch.tensor(ns, device="cuda"))
    x = (_uniform(seed, 1, 1, sum(ns)) * per).contiguous()
    if case["react"]:
        M = _uniform(seed, 2, 2, sum(ns))
    else:  # the accuracy problem's segregated components
        left = (x[0] < 0.5 * per).double()
        M = torch.stack([left, 1.0 - left])
    return ns, Ls, x, M


def _host_inputs(req, seed, i):
    L = req["L"]
    x = synth.uniform_positions(req["n"], L, dim=req["dim"], seed=seed * 64 + i)
    return x, np.stack(synth.uniform_masses(req["n"], seed=seed * 64 + i))


def _params(case, seed):
    return mt.mt_params_init(
        dim=case["dim"], n=case["n"], L=(case["L"],) * case["dim"], v=(case["v"], 0.0),
        D_mt=case["D"], D_rw=case["D"], dt=case["dt"], search=SEARCH[case["search"]],
        precision=PREC[case["precision"]],
        norm=mt.MT_NORM_SYM if case["norm"] == "sym" else mt.MT_NORM_ROW,
        react=int(case["react"]), seed=int(seed),
        walls=mt.MT_WALLS_REFLECT if case["walls"] == "reflect" else mt.MT_WALLS_PERIODIC,
        species=case["species"], observe_cap=case["steps"] if case["observe"] else 0)


# ---------------------------------------------------------- prepare / run --

def prepare(case, seed):
    if case["kind"] == "serve":
        reqs = _requests(case)
        return {"case": case, "reqs": reqs, "params": [_params(r, seed + i) for i, r in enumerate(reqs)],
                "data": [_host_inputs(r, seed, i) for i, r in enumerate(reqs)],
                "server": mt.Server(1 << 30, max_active=16, chunk_steps=25)}
    batch = None
    if case["kind"] == "batch":
        ns, Ls, x, M = _batch_inputs(case, seed)
        batch = mt.make_batch(ns, Ls)
        p = mt.mt_params_init(dim=1, D_mt=case["D"], D_rw=case["D"], dt=case["dt"],
                              precision=PREC[case["precision"]], react=int(case["react"]),
                              seed=int(seed), observe_cap=case["steps"] if case["observe"] else 0)
    else:
        x, M = _inputs(case, seed)
        p = _params(case, seed)
    sim = mt.Simulation(p, batch=batch)
    torch.cuda.current_stream().synchronize()  # the handle works on a stream of its own
    return {"case": case, "sim": sim, "x": x, "M": M, "out_x": torch.empty_like(x),
            "out_M": torch.empty_like(M)}


def run(state):
    case = state["case"]
    if case["kind"] == "serve":
        s = state["server"]
        ids = [s.submit(p, x, M[0], M[1], r["steps"])
               for p, r, (x, M) in zip(state["params"], state["reqs"], state["data"])]
        s.drain()
        out = [s.result(i) for i in ids]
        for i in ids:
            s.release(i)
        return [{"A": A, "B": B, "observables": o} for A, B, o in out]
    sim, x, M = state["sim"], state["x"], state["M"]
    ox, om = state["out_x"], state["out_M"]
    mt.mt_upload(sim.h, x.data_ptr(), M[0].data_ptr(), M[1].data_ptr(), mt.MT_MEM_DEVICE)
    for s in range(2, M.shape[0]):
        mt.mt_set_species(sim.h, s, M[s].data_ptr(), mt.MT_MEM_DEVICE)
    sim.run(case["steps"])
    mt.mt_read_masses(sim.h, om[0].data_ptr(), om[1].data_ptr(), mt.MT_MEM_DEVICE)
    for s in range(2, M.shape[0]):
        mt.mt_read_species(sim.h, s, om[s].data_ptr(), mt.MT_MEM_DEVICE)
    mt.mt_read_positions(sim.h, ox.data_ptr(), mt.MT_MEM_DEVICE)
    out = {"x": ox, "M": om}
    if case["observe"]:
        out["observables"] = sim.observables()
    return out


# ----------------------------------------------------------------- work --

def _neighbours(case, n, L):
    """Expected neighbours within the cutoff of a particle of a uniform system."""
    s = 3.0 * math.sqrt(4.0 * case["D"] * case["dt"])
    if case.get("search") == "full":
        return n - 1.0
    return 2.0 * s * n / L if case.get("dim", 1) == 1 else math.pi * s * s * n / (L * L)


def _work(case, n, L):
    """A step reads and writes each particle's position and masses once; an
    ordered pair costs a weight (counted as 8 operations, half of it its own)
    and, per species, a difference, a product and a sum; a particle its walk."""
    dim, species = case.get("dim", 1), case.get("species", 2)
    pairs = n * _neighbours(case, n, L)
    steps = case["steps"]
    state = 8.0 * n * (dim + species)
    return steps * 2.0 * state + 2.0 * state, steps * (pairs * (6.0 + 3.0 * species) + n * 30.0 * dim)


def work(case):
    if case["kind"] == "serve":
        parts = [_work(r, r["n"], r["L"]) for r in _requests(case)]
    elif case["kind"] == "batch":
        parts = [_work(case, n, L) for n, L in zip(*_sizes(case))]
    else:
        parts = [_work(case, case["n"], case["L"])]
    return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}


# ---------------------------------------------------------------- exact --
# The same steps in 64 bits: positions as whole grid ticks x = X 2^-k (k the
# largest with s_max 2^k < 2^30 and L 2^k < 2^61), the walk's Philox4x32-10
# numbers with Box-Muller in binary64, everything else in binary64.

_M32 = 0xFFFFFFFF


def _normals(loc, step, real, seed, dim):
    c = [loc, torch.full_like(loc, step & _M32), torch.full_like(loc, (step >> 32) & _M32), real]
    k0, k1 = seed & _M32, (seed >> 32) & _M32
    for _ in range(10):
        p0, p1 = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57
        c = [((p1 >> 32) & _M32) ^ c[1] ^ k0, p1 & _M32, ((p0 >> 32) & _M32) ^ c[3] ^ k1, p0 & _M32]
        k0, k1 = (k0 + 0x9E3779B9) & _M32, (k1 + 0xBB67AE85) & _M32
    u1 = ((c[0] >> 8) + 1).double() * 2.0**-24
    u2 = (c[1] >> 8).double() * 2.0**-24
    rad, ang = torch.sqrt(-2.0 * torch.log(u1)), 2.0 * math.pi * u2 - math.pi
    return [rad * torch.cos(ang), rad * torch.sin(ang)][:dim]


def _pairs(X, base, Lq, S, periodic):
    """Unordered pairs (i, j) within S ticks and their squared separations in
    ticks (binary64).  X: (dim, n) ticks; base: the start of each particle's
    realisation on the shared axis; Lq: domain length per axis."""
    dim, n = X.shape
    x0, order = torch.sort(X[0] + base)
    if periodic:  # particles near 0 again beyond the far wall
        near = order[X[0][order] <= S]
        x0, order = torch.cat([x0, X[0][near] + Lq[0]]), torch.cat([order, near])
    at = torch.arange(n, device=X.device)
    I, J, R2 = [], [], []
    k = 1
    while True:
        at = at[at + k < x0.numel()]
        dx = x0[at + k] - x0[at]
        keep = dx <= S
        at, dx = at[keep], dx[keep]
        if not at.numel():
            break
        i, j = order[at], order[at + k]
        d2 = dx * dx
        if dim == 2:
            dy = X[1][j] - X[1][i]
            if periodic:
                dy = torch.remainder(dy + Lq[1] // 2, Lq[1]) - Lq[1] // 2
            d2 = d2 + dy * dy
            ok = (dy.abs() <= S) & (d2 <= S * S)
            i, j, d2 = i[ok], j[ok], d2[ok]
        I.append(i), J.append(j), R2.append(d2.double())
        k += 1
    if not I:
        z = torch.zeros(0, dtype=torch.int64, device=X.device)
        return z, z, z.double()
    return torch.cat(I), torch.cat(J), torch.cat(R2)


def _transfer(M, i, j, w, row):
    r = torch.ones_like(M[0]).index_add_(0, i, w).index_add_(0, j, w)
    pi, pj = (w / r[i], w / r[j]) if row else (0.5 * (w / r[i] + w / r[j]),) * 2
    out = []
    for m in M:
        d = m[j] - m[i]
        out.append(m + 0.5 * torch.zeros_like(m).index_add_(0, i, pi * d).index_add_(0, j, -pj * d))
    return torch.stack(out)


def _transfer_full(M, x, inv8, row):
    n, rows = x.numel(), max(1, (1 << 27) // x.numel())
    w = lambda a: torch.exp(-((x[a:a + rows, None] - x[None, :]) ** 2) * inv8)  # noqa: E731
    r = torch.cat([w(a).sum(1) for a in range(0, n, rows)])
    out = torch.empty_like(M)
    for a in range(0, n, rows):
        P = w(a)
        P = P / r[a:a + rows, None] if row else 0.5 * (P / r[a:a + rows, None] + P / r[None, :])
        for s, m in enumerate(M):
            out[s, a:a + rows] = m[a:a + rows] + 0.5 * (P * (m[None, :] - m[a:a + rows, None])).sum(1)
    return out


def _exact_steps(x, M, L, parts, *, v, D, dt, steps, seed, row, react, periodic, full):
    """parts: particles per realisation; L: per axis, or per realisation in a batch."""
    dim, n = x.shape
    smax = 3.0 * math.sqrt(4.0 * D * dt)
    Lmax = max(L)
    k = 62
    while math.ldexp(smax, k) >= 2.0**30 or math.ldexp(Lmax, k) >= 2.0**61:
        k -= 1
    S = math.floor(math.ldexp(smax, k))
    X = torch.round(x * 2.0**k).to(torch.int64)
    counts = torch.tensor(parts, device=x.device)
    real = torch.repeat_interleave(torch.arange(len(parts), device=x.device), counts)
    off = torch.cumsum(counts, 0) - counts
    loc = torch.arange(n, device=x.device) - off[real]
    if len(parts) > 1:
        Lq = torch.tensor([round(math.ldexp(v_, k)) for v_ in L], device=x.device)
        base = (torch.cumsum(Lq + 2 * S, 0) - (Lq + 2 * S))[real]
        Lp = [Lq[real]]
    else:
        Lp = [round(math.ldexp(L[a], k)) for a in range(dim)]
        base = torch.zeros_like(loc)
    drift = [round(math.ldexp(v * dt, k)), 0]
    b = math.ldexp(math.sqrt(2.0 * D * dt), k)
    obs = []
    for t in range(steps):
        for a, z in enumerate(_normals(loc, t, real, seed, dim)):
            y = X[a] + drift[a] + torch.round(b * z).to(torch.int64)
            if periodic:
                y = torch.remainder(y, Lp[a])
            else:
                for _ in range(4):
                    y = torch.where(y < 0, -y, y)
                    y = torch.where(y > Lp[a], 2 * Lp[a] - y, y)
            X[a] = y
        if full:
            M = _transfer_full(M, X[0].double() * 2.0**-k, 1.0 / (8.0 * D * dt), row)
        else:
            i, j, d2 = _pairs(X, base, Lp, S, periodic)
            M = _transfer(M, i, j, torch.exp(-d2 * (2.0**(-2 * k) / (8.0 * D * dt))), row)
        if react:
            m = torch.minimum(M[0], M[1])
            M[0] -= m
            M[1] -= m
        sums = torch.zeros(2, len(parts), dtype=torch.float64, device=x.device).index_add_(1, real, M[:2])
        obs.append(torch.stack([sums[0], sums[1], sums[0] - sums[1], sums[0] / counts], 1))
    return X.double() * 2.0**-k, M, torch.stack(obs)


def exact(case, seed):
    if case["kind"] == "serve":
        out = []
        for i, r in enumerate(_requests(case)):
            x, M = (torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in _host_inputs(r, seed, i))
            _, M, obs = _exact_steps(x, M, [r["L"]] * r["dim"], [r["n"]], v=r["v"], D=r["D"],
                                     dt=r["dt"], steps=r["steps"], seed=seed + i, row=False,
                                     react=r["react"], periodic=False, full=False)
            out.append({"A": M[0], "B": M[1], "observables": obs[:, 0]})
        return out
    if case["kind"] == "batch":
        ns, Ls, x, M = _batch_inputs(case, seed)
        x, M, obs = _exact_steps(x, M, Ls, ns, v=0.0, D=case["D"], dt=case["dt"],
                                 steps=case["steps"], seed=seed, row=False, react=case["react"],
                                 periodic=False, full=False)
    else:
        x, M = _inputs(case, seed)
        x, M, obs = _exact_steps(x, M, [case["L"]] * case["dim"], [case["n"]], v=case["v"],
                                 D=case["D"], dt=case["dt"], steps=case["steps"], seed=seed,
                                 row=case["norm"] == "row", react=case["react"],
                                 periodic=case["walls"] == "periodic",
                                 full=case["search"] == "full")
        obs = obs[:, 0]
    out = {"x": x, "M": M}
    if case["observe"]:
        out["observables"] = obs
    return out
