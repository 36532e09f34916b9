"""Checkpoints of format version 1, whose workspace held two regions more (a word
per cell; 32 MiB in large MT_FP64 one-kernel systems), load and continue."""
import ctypes
import re
import struct
from pathlib import Path

import numpy as np
import pytest

from paper_1811_05474_gb300 import mt, synth

pytestmark = pytest.mark.gpu

SRC = (Path(mt.__file__).parent / "csrc" / "mt_internal.cuh").read_text()


def constant(name):
    return eval(re.search(rf"constexpr int {name} = ([^;]+);", SRC).group(1),
                {"kThreads": 256, "kScanItems": 16})


def region(nbytes):
    return (nbytes + 255) // 256 * 256


def old_file(path, sim, n, dim, species, cap):
    """The version-1 form of the file that sim saves: (bytes, sizes of the two regions)."""
    p = sim.params
    raw = path.read_bytes()
    head = 16 + ctypes.sizeof(mt.mt_params)
    steps, rt_bytes, ws_bytes = struct.unpack_from("<qQQ", raw, head)
    ws = raw[head + 24 + rt_bytes:]
    assert len(ws) == ws_bytes and struct.unpack_from("<I", raw, 8)[0] == 2
    Lq = [int(np.rint(np.ldexp(p.L[a], p.frac_bits))) for a in range(dim)]
    ncell = int(np.prod([(v >> p.cell_shift) + 1 for v in Lq])) if p.search == mt.MT_SEARCH_CELL else 0
    status = region(256) + 2 * region(dim * n * 8) + 2 * region(n * 4) + 2 * region(species * n * 8)
    status += region(n * 4) + region(n * 8) + region(ncell * 4) + region((ncell + 1) * 4)
    cursor = region(ncell * 4)
    fused = p.seg_target > 0
    nseg = -(-n // p.seg_target) if fused else 0
    pred = status + region(-(-ncell // constant("kScanTile")) * 8)
    pred += region((n // (constant("kSmallCell") + 1) + 1) * 4) + region(cap * 32)
    pred += 2 * region((ncell + 1) * 4 if fused else 0) + 2 * region((nseg + 1) * 4 if fused else 0)
    pred += region(nseg * 4)
    wc = 32 << 20 if fused and p.precision == mt.MT_FP64 and n >= 1 << 17 else 0
    ws = ws[:status] + b"\xa5" * cursor + ws[status:pred] + b"\xa5" * wc + ws[pred:]
    out = raw[:8] + struct.pack("<I", 1) + raw[12:head]
    out += struct.pack("<qQQ", steps, rt_bytes, len(ws)) + raw[head + 24:head + 24 + rt_bytes] + ws
    return out, cursor + wc


@pytest.mark.parametrize("kw", [
    dict(n=200000, L=(200000.0,), precision=mt.MT_FP64, v=(0.5,), observe_cap=40),
    dict(n=200000, L=(200000.0,), precision=mt.MT_MIXED, observe_cap=40),
    dict(n=3000, L=(3000.0,), walls=mt.MT_WALLS_PERIODIC, species=3),
    dict(n=20000, L=(500.0, 400.0), dim=2, precision=mt.MT_MIXED_DF32, observe_cap=40),
    dict(n=2000, L=(20.0,), precision=mt.MT_FP64),
    dict(n=1500, L=(1500.0,), search=mt.MT_SEARCH_FULL),
])
def test_version_1_continues(kw, tmp_path):
    n, dim, species = kw["n"], kw.get("dim", 1), kw.get("species", 2)
    p = mt.mt_params_init(seed=9, **kw)
    sim = mt.Simulation(p)
    sim.upload(synth.uniform_positions(n, kw["L"] if dim == 2 else kw["L"][0], dim=dim, seed=5),
               *synth.uniform_masses(n, seed=5))
    sim.run(14)
    sim.save(tmp_path / "new")
    raw, extra = old_file(tmp_path / "new", sim, n, dim, species, kw.get("observe_cap", 0))
    (tmp_path / "old").write_bytes(raw)
    sim.run(15)
    want = [sim.ticks(), *[sim.species(s) for s in range(species)], sim.observables()]
    sim.close()
    assert mt.mt_checkpoint_params(tmp_path / "old").n == n
    other = mt.Simulation(mt.mt_checkpoint_params(tmp_path / "old"))
    other.load(tmp_path / "old")
    other.run(15)
    got = [other.ticks(), *[other.species(s) for s in range(species)], other.observables()]
    for a, b in zip(got, want):
        assert np.array_equal(a, b)
    if extra:  # the regions' bytes are part of the file's size check
        (tmp_path / "cut").write_bytes(raw[:-256])
        with pytest.raises(mt.MtError):
            other.load(tmp_path / "cut")
    other.close()
