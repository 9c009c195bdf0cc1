"""The fixed-point elementary functions on the GPU, element by element, and
outside their fixed-point ranges (where they are CUDA's own)."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

import synth
from test_host_device_code import division_arguments, log_arguments, same_bits, ulp_error

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    out = str(tmp_path_factory.mktemp("fixed") / "libfixed.so")
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17",
                    "-shared", "-Xcompiler", "-fPIC", "-I", os.path.join(ROOT, "include"),
                    "-I", os.path.join(ROOT, "paper_1509_00680_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "fixed_math_check.cu"), "-o", out], check=True)
    return ctypes.CDLL(out)


def _on_gpu(run, *arrays):
    """run(inputs .., output, n) on the GPU."""
    import torch
    a = [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in arrays]
    out = torch.empty_like(a[0])
    assert run(*[ctypes.c_void_p(t.data_ptr()) for t in a], ctypes.c_void_p(out.data_ptr()), out.numel()) == 0
    return out.cpu().numpy()


def test_logarithm(lib):
    """One unit in the last place, that of CUDA's log."""
    x = np.concatenate([log_arguments(200000), [1e-300, 1e300, 2.0 ** 8, 2.0 ** -7.5, 5e-324]])
    assert ulp_error(_on_gpu(lib.run_fixed_log, x), np.log(x.astype(np.longdouble))) < 1.0
    got = _on_gpu(lib.run_fixed_log, np.array([0.0, -1.0, np.inf, np.nan, 1.0]))
    assert got[0] == -np.inf and np.isnan(got[1]) and got[2] == np.inf and np.isnan(got[3]) and got[4] == 0.0


def test_division_is_correctly_rounded(lib):
    a, b = division_arguments(300000)
    with np.errstate(all="ignore"):
        assert same_bits(_on_gpu(lib.run_fixed_divide, a, b), a / b)


def test_polarization_charge_divides_exactly():
    """A constant potential leaves -((eps - 1)/eps) rho, whose division IEEE
    arithmetic fixes; with rho = 1 nothing else rounds."""
    import torch
    from paper_1509_00680_gb300 import build
    build.build()
    from paper_1509_00680_gb300 import gps
    g = synth.Grid(32, 24, 20, 0.4, 0.4, 0.4, synth.BC_PERIODIC)
    eps = 1.0 + 80.0 * np.random.default_rng(36).random(g.npts) ** 3
    one = torch.ones(g.npts, dtype=torch.float64, device="cuda")
    out = torch.empty_like(one)
    ctx = gps.Context(0)
    ctx.polarization_charge(gps.grid_from(g), one, torch.from_numpy(eps).cuda(), one, out)
    got = out.cpu().numpy()
    ctx.close()
    assert np.array_equal(got, -((eps - 1.0) / eps))
