"""The FP64 spectrum's 64-bit fixed-point transforms at the places where block
floating point can go wrong: sources of every crest factor (one point, noise,
a smooth charge), values far from 1, zero and non-finite input, and the
lengths at the edges of each kernel (register-resident 64 .. 1024,
shared-memory radices 2, 3, 5, 16, the rescaled stages above 512 points).

Tolerance: either side rounds its five passes at about 2^-53 of each line, and
the kernel weighs the error like the source (white for the point and the
noise, whose low wavevectors carry the potential), so 4e-15 in relative L2
norm leaves a factor of three to ten; powers of two must come out bit for
bit."""
import numpy as np
import pytest

import synth
from oracle.green import VacuumSolver

pytestmark = pytest.mark.gpu

GRIDS = [
    (synth.BC_PERIODIC, (64, 30, 128)),
    (synth.BC_FREE, (32, 27, 64)),
    (synth.BC_SURFACE, (48, 256, 32)),
    (synth.BC_WIRE, (40, 64, 50)),
    (synth.BC_PERIODIC, (1024, 8, 12)),
    (synth.BC_PERIODIC, (8, 2048, 10)),
    (synth.BC_PERIODIC, (10, 8, 1024)),
    (synth.BC_PERIODIC, (4096, 4, 6)),
    (synth.BC_PERIODIC, (6, 4, 2400)),
]


def _source(kind, g):
    rng = np.random.default_rng(5)
    if kind == "point":
        a = np.zeros(g.shape)
        a[g.nz // 3, g.ny // 2, 1] = 1.0
    elif kind == "smooth":
        z, y, x = np.meshgrid(*[np.arange(m) - 0.45 * m for m in g.shape], indexing="ij")
        a = np.exp(-0.05 * (x * x + y * y + z * z))
    else:
        a = rng.standard_normal(g.shape)
    return a


@pytest.fixture(scope="module")
def lib():
    from paper_1509_00680_gb300 import build
    build.build()
    from paper_1509_00680_gb300 import gps
    ctx = gps.Context(0)
    yield gps, ctx
    ctx.close()


def _solve(lib, g, a):
    import torch
    gps, ctx = lib
    w = torch.zeros(g.npts, dtype=torch.float64, device="cuda")
    ctx.vacuum_solve(gps.grid_from(g), torch.from_numpy(a.ravel()).cuda(), w)
    return w.cpu().numpy().reshape(g.shape)


@pytest.mark.parametrize("bc,n", GRIDS)
def test_crest_factors_and_scaling(lib, bc, n):
    g = synth.Grid(n[0], n[1], n[2], 0.4, 0.4, 0.4, bc)
    vac = VacuumSolver(g)
    for kind in ("point", "smooth", "noise"):
        a = _source(kind, g)
        w = _solve(lib, g, a)
        ref = vac.apply(a)
        assert np.linalg.norm(w - ref) <= 4e-15 * np.linalg.norm(ref), kind
        for k in (-300, 250):
            assert np.array_equal(_solve(lib, g, np.ldexp(a, k)), np.ldexp(w, k)), (kind, k)


@pytest.mark.parametrize("bc,n", [GRIDS[0], GRIDS[1], (synth.BC_PERIODIC, (20, 18, 30))])
def test_zero_and_non_finite(lib, bc, n):
    g = synth.Grid(n[0], n[1], n[2], 0.4, 0.4, 0.4, bc)
    assert not _solve(lib, g, np.zeros(g.shape)).any()
    for bad in (np.nan, np.inf):
        a = _source("noise", g)
        a[2, 3, 1] = bad
        assert np.isnan(_solve(lib, g, a)).all()
