"""Potentials whose values within one tile are many decades apart: v_eps at
every point against the gradient in extended precision.

Tolerance: a derivative is within 2^-49 of the largest value of its stencil
(16 terms, coefficients that sum to 2.7, rounded at 2^-53 in a chain of eight),
and v_eps is a sum of squares of three of them, rounded four times."""
import numpy as np
import pytest

import synth
from test_host_device_code import _derivative, _spread

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["rough", "spike", "decay", "patch", "tiny", "zero"])
def test_v_eps_follows_each_stencil(kind):
    import torch
    from paper_1509_00680_gb300 import build
    build.build()
    from paper_1509_00680_gb300 import gps
    g = synth.Grid(40, 24, 20, 0.4, 0.35, 0.5, synth.BC_PERIODIC)
    phi = _spread(kind, g.shape)
    if kind == "tiny":
        phi = phi * 1e160                    # squares stay normal; 1e-140 beside zeros
    ctx = gps.Context(0)
    out = torch.zeros(g.npts, dtype=torch.float64, device="cuda")
    ctx.v_eps(gps.grid_from(g), torch.full((g.npts,), -8.0 * np.pi, dtype=torch.float64, device="cuda"),
              torch.from_numpy(phi.ravel()).cuda(), out)
    got = out.cpu().numpy().reshape(g.shape)
    ctx.close()
    u = phi.astype(np.longdouble)
    ref, err = np.zeros_like(u), np.zeros_like(u)
    for axis, h in enumerate((g.hx, g.hy, g.hz)):
        d = _derivative(u, axis) / h
        big = np.max([np.abs(np.roll(u, s * j, 2 - axis)) for j in range(1, 9) for s in (-1, 1)], axis=0)
        e = 2.0 ** -49 * big / h
        ref += d * d
        err += 2 * np.abs(d) * e + e * e
    assert (np.abs(got - ref) <= err + 2.0 ** -50 * ref).all()
