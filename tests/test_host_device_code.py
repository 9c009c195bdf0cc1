"""Device headers run on the host, a thread per CUDA thread (host_cuda.h): the
order of their shared accesses under schedules that the hardware may take, and
their arithmetic against exact references."""
import ctypes
import math
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _cuda_include():
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    return os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    inc = _cuda_include()
    if not (shutil.which("g++") and os.path.exists(os.path.join(inc, "cuda_runtime.h"))):
        pytest.skip("needs g++ and the CUDA headers")
    out = str(tmp_path_factory.mktemp("host") / "libhost.so")
    subprocess.run(["g++", "-O1", "-std=c++20", "-w", "-shared", "-fPIC", "-pthread", "-ffp-contract=off",
                    "-I", os.path.join(ROOT, "tests"), "-I", os.path.join(ROOT, "include"),
                    "-I", os.path.join(ROOT, "paper_1509_00680_gb300", "csrc"), "-I", inc,
                    os.path.join(ROOT, "tests", "host_device_code.cpp"), "-o", out], check=True)
    return ctypes.CDLL(out)


class Stencil16(ctypes.Structure):
    _fields_ = [("n", ctypes.c_int * 3), ("per", ctypes.c_int * 3), ("ih", ctypes.c_double * 3),
                ("d", ctypes.c_double * 9)]


def _coefficients():
    f = math.factorial
    return [0.0] + [(-1) ** (j + 1) * f(8) ** 2 / (j * f(8 - j) * f(8 + j)) for j in range(1, 9)]


def _stencil(n, per):
    return Stencil16((ctypes.c_int * 3)(*n), (ctypes.c_int * 3)(*[per] * 3), (ctypes.c_double * 3)(1, 1, 1),
                     (ctypes.c_double * 9)(*_coefficients()))


def _ptr(a):
    return a.ctypes.data_as(ctypes.c_void_p)


def _derivative(u, axis):
    """sum_j d_j (u_(i+j) - u_(i-j)) on a periodic axis of u[z, y, x]."""
    return sum(c * (np.roll(u, -j, 2 - axis) - np.roll(u, j, 2 - axis))
               for j, c in enumerate(_coefficients()) if j)


@pytest.mark.parametrize("finite", [True, False])
@pytest.mark.parametrize("axis", [0, 1, 2])
def test_tile_maximum_is_not_lost(lib, axis, finite):
    """The largest exponent of a field is posted by warps 1 to 7 while thread 0
    still finishes the derivative before (of a field with a NaN or without):
    nothing may erase it."""
    rng = np.random.default_rng(31)
    n = (32, 8, 8)
    u0 = rng.standard_normal(n[::-1])
    if not finite:
        u0[2, 3, 4] = np.nan
    u1 = rng.standard_normal(n[::-1]) * np.ldexp(1.0, np.where(np.arange(8) > 0, 30, 0))[None, :, None]
    d0, d1 = np.zeros_like(u0), np.zeros_like(u1)
    lib.derivative_pair(ctypes.byref(_stencil(n, 1)), axis, _ptr(u0), _ptr(u1), _ptr(d0), _ptr(d1))
    ref = _derivative(u1, axis)
    assert np.abs(d1 - ref).max() <= 1e-14 * np.abs(u1).max()
    if finite:
        assert np.abs(d0 - _derivative(u0, axis)).max() <= 1e-14 * np.abs(u0).max()
