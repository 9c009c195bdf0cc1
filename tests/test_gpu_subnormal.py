"""The FP64 spectrum on charges below the smallest normal number: the vacuum
solve is linear, so integers times 2^-1074 give the potential of the integers
times 2^-1074.

Tolerance: sources of 30 bits whose unit is that of the subnormal numbers lose
at most four of them where a line of up to 2048 points is scaled, so 2^-26 of a
transform's line, and 1e-6 leaves a factor of 60."""
import numpy as np
import pytest

import synth
from test_gpu_fix64 import GRIDS, _solve, lib  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bc,n", GRIDS[:4])
def test_subnormal_charges(lib, bc, n):  # noqa: F811
    g = synth.Grid(n[0], n[1], n[2], 0.4, 0.4, 0.4, bc)
    a = np.random.default_rng(6).integers(-(1 << 30), 1 << 30, g.shape).astype(float)
    w = _solve(lib, g, np.ldexp(a, -1074))
    ref = np.ldexp(_solve(lib, g, a), -1074)
    assert np.abs(ref).max() < np.finfo(float).tiny
    err, ref = np.ldexp(w - ref, 600), np.ldexp(ref, 600)   # squares of subnormal numbers vanish
    assert np.linalg.norm(err) <= 1e-6 * np.linalg.norm(ref)
