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


def test_conversions_underflow_gradually(lib):
    """Subnormal doubles keep their value, and results below the smallest normal
    number round to the nearest multiple of 2^-1074, ties away from zero."""
    rng = np.random.default_rng(33)
    d = np.concatenate([np.ldexp(rng.integers(1, 1 << 52, 4000).astype(float), -1074), np.ldexp(rng.random(4000), -1022),
                        [0.0, 5e-324, np.finfo(float).tiny, np.finfo(float).max, 1.0]])
    d = np.concatenate([d, -d])
    out = np.zeros_like(d)
    for drop in (0, 9):
        lib.fixed_round_trip(_ptr(d), _ptr(out), d.size, drop, 0)
        assert np.array_equal(out, d)
    m = rng.integers(1 << 52, 1 << 53, 4000)
    x = np.ldexp(m.astype(float), -52)
    got = np.zeros_like(x)
    for k in range(-1090, -1022):            # x 2^k = m 2^(k - 52): the bits below 2^-1074 go
        s = min(-1074 - (k - 52), 62)
        ref = np.ldexp(((m + (1 << (s - 1))) >> s).astype(float), -1074)
        for sign in (1.0, -1.0):
            lib.fixed_round_trip(_ptr(sign * x), _ptr(got), x.size, 0, k)
            assert np.array_equal(got, sign * ref), k


def _spread(kind, shape):
    rng = np.random.default_rng(32)
    u = rng.standard_normal(shape)
    if kind == "spike":                      # one value far above its tile
        u[4, 3, 11] = 1e13
    elif kind == "decay":                    # 24 decades along each axis
        z, y, x = np.meshgrid(*[np.linspace(0, 1, m) for m in shape], indexing="ij")
        u = 10.0 ** (-24 * np.abs(x - 0.4) - 24 * np.abs(y - 0.5) - 24 * np.abs(z - 0.3)) * (1 + 0.1 * u)
    elif kind == "patch":                    # zero but for a corner of one and a value of 1e-30
        u[:, :, :] = 0.0
        u[:3, :3, :5] = 1.0
        u[6, 5, 20] = 1e-30
    elif kind == "tiny":
        u = u * 1e-300
        u[5, 5, 5] = 0.0
    elif kind == "zero":
        u = 0.0 * u
    return u


@pytest.mark.parametrize("kind", ["rough", "spike", "decay", "patch", "tiny", "zero"])
@pytest.mark.parametrize("axis", [0, 1, 2])
def test_tile_derivatives_follow_their_stencils(lib, axis, kind):
    """Each derivative against the largest value of its own stencil, whatever
    else the tile holds: 2^-49 of it covers the rounding of 16 terms with
    coefficients that sum to 2.7 in either arithmetic."""
    n = (32, 24, 24)
    u = _spread(kind, n[::-1])
    d = np.zeros((8, 8, 32))
    scratch = np.zeros_like(d)
    lib.derivative_pair(ctypes.byref(_stencil(n, 1)), axis, _ptr(u), _ptr(u), _ptr(scratch), _ptr(d))
    ul = u.astype(np.longdouble)
    ref = _derivative(ul, axis)[:8, :8]
    big = np.max([np.abs(np.roll(u, s * j, 2 - axis)) for j in range(1, 9) for s in (-1, 1)], axis=0)[:8, :8]
    assert (np.abs(d - ref) <= 2.0 ** -49 * big).all()


def log_arguments(n):
    """Arguments of the fixed-point logarithm: its whole range, around 1, both
    sides of the table's interval edges and of the near-1 branch."""
    rng = np.random.default_rng(34)
    edges = 1.0 + np.arange(129) / 128.0
    edges = np.concatenate([np.ldexp(edges, k) for k in range(-7, 8)])
    edges = np.concatenate([np.nextafter(edges, 0.0), edges, np.nextafter(edges, 1e3)])
    x = np.concatenate([2.0 ** rng.uniform(-7, 8, n), 1.0 + rng.uniform(-0.02, 0.02, n),
                        1.0 + rng.choice([-1.0, 1.0], n) * 10.0 ** rng.uniform(-15.9, -1.5, n),
                        1.0 + 2.0 ** -7 * (1.0 + rng.uniform(0, 0.01, n)), edges])
    return x[(x >= 2.0 ** -7) & (x < 2.0 ** 8)]


def ulp_error(got, exact):
    """Largest distance from `exact` (extended precision) in units in the last
    place of the exact value."""
    ref = np.abs(exact.astype(float))
    return float(np.max(np.abs(got - exact) / np.spacing(np.where(ref > 0, ref, 1.0))))


def test_logarithm(lib):
    """Every result within one unit in the last place, near 1 in particular."""
    x = log_arguments(200000)
    got = np.zeros_like(x)
    lib.fixed_log(_ptr(x), _ptr(got), x.size)
    assert ulp_error(got, np.log(x.astype(np.longdouble))) < 1.0


def division_arguments(n):
    """Random mantissas at near and far exponents, quotients of small whole
    numbers, numbers a few units apart and next to powers of two, and what is not a normal
    number."""
    rng = np.random.default_rng(35)
    a, b = rng.uniform(1, 2, (2, n)) * 2.0 ** rng.integers(-40, 40, (2, n)) * rng.choice([-1.0, 1.0], (2, n))
    far = np.ldexp(rng.uniform(1, 2, (2, n)), rng.integers(-1070, 1023, (2, n)))
    whole = rng.integers(-1000, 1000, (2, n)).astype(float)
    m = rng.integers(1 << 52, 1 << 53, n)
    close = np.array([m, np.clip(m + rng.integers(-4, 5, n), 1 << 52, (1 << 53) - 1)]).astype(float)
    edge = np.ldexp(1.0 + rng.integers(-3, 4, (2, n)) * 2.0 ** -52, rng.integers(-3, 4, (2, n)))
    odd = np.array([0.0, -0.0, 1.0, -3.0, 5e-324, 2.2e-308, 1.7e308, np.inf, -np.inf, np.nan])
    pairs = np.array([(x, y) for x in odd for y in odd]).T
    return np.concatenate([(a, b), far, whole, close, edge, pairs], axis=1)


def same_bits(x, y):
    return np.array_equal(x, y, equal_nan=True) and np.array_equal(np.signbit(x)[~np.isnan(x)],
                                                                  np.signbit(y)[~np.isnan(y)])


def test_division_is_correctly_rounded(lib):
    a, b = np.ascontiguousarray(division_arguments(300000))
    got = np.zeros_like(a)
    lib.fixed_divide(_ptr(a), _ptr(b), _ptr(got), a.size)
    with np.errstate(all="ignore"):
        assert same_bits(got, a / b)
        for k in (1, 2, 3):
            lib.fixed_divide_by_pi(_ptr(a), _ptr(got), a.size, k)
            assert same_bits(got, a / (2 ** k * np.pi))


def test_factor_digits(lib):
    """Two signed digits give the factor back; a low digit of -2^31, which has
    no negative, becomes the next one."""
    rng = np.random.default_rng(37)
    k = np.concatenate([np.arange(-6, 7), rng.integers(-(1 << 30) + 1, 1 << 30, 1000)])
    low = k * (1 << 32) - (1 << 31)
    w = np.concatenate([low, rng.integers(-(1 << 62), 1 << 62, 20000), [1 << 62, -(1 << 62), 0, (1 << 31) - 1]])
    out = np.zeros_like(w)
    lib.fixed_digits(_ptr(w), _ptr(out), w.size)
    assert np.array_equal(out, w + np.isin(w, low))


@pytest.mark.parametrize("forward", [0, 1])
def test_radix_3_rounds_to_neither_side(lib, forward):
    """Half of the sums that a radix-3 butterfly halves are odd: an error of one
    unit, up or down, whose mean stays within five standard deviations of 0."""
    n = 200000
    x = np.random.default_rng(38).integers(-(1 << 58), 1 << 58, 3 * n)
    out = np.zeros(n, dtype=np.int64)
    lib.fixed_radix3(_ptr(x), _ptr(out), n, forward)
    assert np.abs(out).max() <= 1 and abs(out.mean()) <= 5 * np.sqrt(0.5 / n)


@pytest.mark.parametrize("shift", [0, 3, 6, 7, 9, 12])
def test_alignment_rounds_to_neither_side(lib, shift):
    """A value brought to a larger one's exponent: within half a unit, with a
    mean within five standard deviations (at most 1/2 unit each) of 0."""
    n = 200000
    r = np.random.default_rng(39)
    m = r.integers(1 << 61, 1 << 62, n) * r.choice([-1, 1], n)
    out = np.zeros(n)
    lib.fixed_align(_ptr(m), _ptr(out), n, shift)
    assert np.abs(out).max() <= 0.5 and abs(out.mean()) <= 5 * 0.5 / np.sqrt(n)


@pytest.mark.parametrize("negative", [0, 1])
def test_half_products_round_to_neither_side(lib, negative):
    """Real numbers times sixth roots of unity are halves: within one unit, with
    a mean within five standard deviations (1/2 unit) of 0."""
    n = 200000
    x = np.random.default_rng(40).integers(-(1 << 56), 1 << 56, n)
    out = np.zeros(n)
    lib.fixed_half_product(_ptr(x), _ptr(out), n, negative)
    assert np.abs(out).max() <= 1 and abs(out.mean()) <= 5 * 0.5 / np.sqrt(n)


def test_partials_are_published_before_the_ticket(lib):
    """What other blocks may rely on when they see a block's ticket is what its
    thread knew at its last fence: the partials of all warps."""
    out = np.zeros(3)
    lib.published_partials(_ptr(out))
    assert np.array_equal(out, 128.0 * np.arange(1, 4))
