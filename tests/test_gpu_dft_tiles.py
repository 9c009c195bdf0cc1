"""The tiled order-16 passes and the logarithm of the polarization charge at
their edges: grids smaller than a tile, one point past it and several tiles on
each axis, fields over many decades, dielectrics on both sides of the
logarithm's range, and values that are not finite.

Tolerance 1e-12 of the largest value, as for the other DFT-facing passes: two
sums of 16 terms per axis in different order, rounded at 2^-53."""
import numpy as np
import pytest

import synth
from oracle import dft

pytestmark = pytest.mark.gpu

GRIDS = [
    (synth.BC_PERIODIC, (8, 8, 8)),
    (synth.BC_FREE, (5, 9, 4)),
    (synth.BC_SURFACE, (36, 8, 5)),
    (synth.BC_WIRE, (32, 16, 12)),
    (synth.BC_PERIODIC, (64, 10, 9 * 2)),
    (synth.BC_FREE, (45, 25, 27)),
]


@pytest.fixture(scope="module")
def lib():
    from paper_1509_00680_gb300 import build
    build.build()
    from paper_1509_00680_gb300 import gps
    ctx = gps.Context(0)
    yield gps, ctx
    ctx.close()


def _run(lib, g, rho, eps, phi, deps):
    import torch
    gps, ctx = lib
    d = [torch.from_numpy(np.ascontiguousarray(a).ravel()).cuda() for a in (rho, eps, phi, deps)]
    pol, v = torch.zeros_like(d[0]), torch.zeros_like(d[0])
    gr = gps.grid_from(g)
    ctx.polarization_charge(gr, d[0], d[1], d[2], pol)
    ctx.v_eps(gr, d[3], d[2], v)
    e = ctx.electrostatic_energy(gr, d[0], d[1], d[2])
    return pol.cpu().numpy().reshape(g.shape), v.cpu().numpy().reshape(g.shape), e


def _close(a, b):
    return np.abs(a - b).max() <= 1e-12 * np.abs(b).max()


@pytest.mark.parametrize("decades", [0, 6])
@pytest.mark.parametrize("bc,n", GRIDS)
def test_tiles(lib, bc, n, decades):
    g = synth.Grid(n[0], n[1], n[2], 0.4, 0.35, 0.5, bc)
    rng = np.random.default_rng(21)
    rho = rng.standard_normal(g.shape)
    phi = rng.standard_normal(g.shape) * 10.0 ** rng.uniform(-decades, 0, g.shape)
    # eps from 1e-4 to 1e4: the table's range, its ends, and log() beyond
    eps = 10.0 ** rng.uniform(-4, 4, g.shape) if decades else 1.0 + 10.0 ** rng.uniform(-16, 2, g.shape)
    deps = np.where(rng.random(g.shape) < 0.3, -np.abs(rho), 0.0)
    pol, v, e = _run(lib, g, rho, eps, phi, deps)
    assert _close(pol, dft.polarization_charge(g, rho, eps, phi))
    assert _close(v, dft.v_eps(g, deps, phi))
    ref = dft.electrostatic_energy(g, rho, eps, phi)
    assert abs(e[1] - ref[1]) <= 1e-12 * abs(ref[1])


def test_not_finite_stays_local(lib):
    """A NaN or an infinity reaches the points whose stencils hold it, no others."""
    g = synth.Grid(72, 20, 24, 0.4, 0.4, 0.4, synth.BC_PERIODIC)
    rng = np.random.default_rng(22)
    rho, eps = rng.standard_normal(g.shape), 1.0 + 40.0 * rng.random(g.shape)
    phi, deps = rng.standard_normal(g.shape), -np.ones(g.shape)
    good = _run(lib, g, rho, eps, phi, deps)[1]
    for bad in (np.nan, np.inf):
        phi2 = phi.copy()
        phi2[10, 11, 40] = bad
        v = _run(lib, g, rho, eps, phi2, deps)[1]
        with np.errstate(invalid="ignore"):
            ref = dft.v_eps(g, deps, phi2)
        assert np.array_equal(np.isfinite(v), np.isfinite(ref))
        ok = np.isfinite(ref)
        assert np.abs(v[ok] - good[ok]).max() <= 1e-12 * np.abs(good).max()


def test_log_is_accurate(lib):
    """ln eps through the polarization charge of a ramp: with one point's eps
    changed at a time the result is a coefficient times ln eps; compared with
    numpy's log at 4 units in the last place of the coefficient's product."""
    import torch
    gps, ctx = lib
    n = 512
    g = gps.make_grid(n, 8, 8, 1.0, 1.0, 1.0, gps.GPS_BC_PERIODIC)
    rng = np.random.default_rng(23)
    x = np.concatenate([2.0 ** rng.uniform(-7, 8, 12), 1.0 + 10.0 ** -np.arange(1.0, 16.0, 2.0),
                        1.0 - 10.0 ** -np.arange(1.0, 16.0, 2.0)])
    eps = np.ones((8, 8, n))
    at = 20 + 17 * np.arange(len(x))
    assert at[-1] + 20 < n
    eps[:, :, at] = x
    phi = np.broadcast_to(np.arange(n, dtype=float), (8, 8, n)).copy()
    out = torch.zeros(eps.size, dtype=torch.float64, device="cuda")
    T = lambda a: torch.from_numpy(np.ascontiguousarray(a).ravel()).cuda()
    ctx.polarization_charge(g, T(np.zeros_like(eps)), T(eps), T(phi), out)
    got = out.cpu().numpy().reshape(eps.shape)[0, 0, at - 1] * 4.0 * np.pi / (8.0 / 9.0)
    assert np.abs(got - np.log(x)).max() <= 4 * np.finfo(float).eps * np.abs(np.log(x)).max()
