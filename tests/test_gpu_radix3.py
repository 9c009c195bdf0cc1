"""White noise on axes with many factors of 3, whose butterflies halve: the FP64
spectrum against the oracle, with the tolerance of test_gpu_fix64 (4e-15 in
relative L2 norm: both sides round five passes at about 2^-53 of each line,
which the kernel weighs like the source)."""
import numpy as np
import pytest

import synth
from oracle.green import VacuumSolver
from test_gpu_fix64 import _solve, lib  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bc,n", [(synth.BC_FREE, (54, 81, 54)), (synth.BC_SURFACE, (54, 18, 81)),
                                  (synth.BC_PERIODIC, (486, 54, 18)), (synth.BC_PERIODIC, (6, 1458, 18))])
def test_noise(lib, bc, n):  # noqa: F811
    g = synth.Grid(n[0], n[1], n[2], 0.4, 0.4, 0.4, bc)
    vac = VacuumSolver(g)
    for seed in range(3):
        a = np.random.default_rng(seed).standard_normal(g.shape)
        ref = vac.apply(a)
        err = _solve(lib, g, a) - ref
        print(bc, n, seed, np.linalg.norm(err) / np.linalg.norm(ref))
        assert np.linalg.norm(err) <= 4e-15 * np.linalg.norm(ref)
