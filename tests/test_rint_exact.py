"""rint_exact (csrc/mt_internal.cuh), the walk's rounding to the grid with
integer operations, replayed on its bit patterns: equal to rounding to the
nearest integer, ties to even, wherever it does not hand over to the
conversion instruction."""
import random
import struct

import numpy as np
import pytest


def rint_exact(v):
    u = struct.unpack("<Q", struct.pack("<d", v))[0]
    sh = 1075 - ((u >> 52) & 0x7FF)
    if sh < 1 or sh > 53:
        return None  # the conversion instruction
    m = (u & (2 ** 52 - 1)) | 2 ** 52
    q = ((m + (2 ** (sh - 1) - 1) + ((m >> sh) & 1)) & (2 ** 64 - 1)) >> sh
    return -q if u >> 63 else q


@pytest.mark.parametrize("scale", [0.5, 1.0, 3.0, 1e3, 2.0 ** 31, 2.0 ** 50, 2.0 ** 51])
def test_rint_exact(scale):
    rng = random.Random(3)
    vals = [scale * rng.uniform(1, 2) * rng.choice([1, -1]) for _ in range(3000)]
    vals += [s * (k + 0.5) for k in range(2000) for s in (1, -1)]  # ties
    vals += [s * v for v in (0.5, np.nextafter(0.5, 1), np.nextafter(1.5, 0), 2.0 ** 52 - 0.5)
             for s in (1, -1)]
    for v in vals:
        got = rint_exact(float(v))
        assert got is None or got == int(np.rint(v)), v
    assert rint_exact(2.0 ** 52) is None and rint_exact(0.49) is None
