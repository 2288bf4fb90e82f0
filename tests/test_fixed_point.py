"""The fixed-point arithmetic of the FP64 transforms, compiled for the host and compared with exact arithmetic."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("fixed") / "fixed_host.so")
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.run(["g++", "-std=c++17", "-O2", "-fPIC", "-shared", "-I", os.path.join(cuda, "include"), "-o", so,
                    os.path.join(HERE, "fixed_host.cpp")], check=True)
    return C.CDLL(so)


def _to_fixed(host, d, k):
    d, out = np.ascontiguousarray(d, np.float64), np.zeros(len(d), np.int64)
    host.to_fixed(len(d), d.ctypes.data_as(C.c_void_p), k, out.ctypes.data_as(C.c_void_p))
    return out


@pytest.mark.parametrize("k", [-900, -3, 0, 61, 900])
def test_conversion_rounds_to_nearest(host, k):
    """Within half a unit of the value at every size, from far below a unit to the top of the range."""
    rng = np.random.default_rng(1)
    v = np.concatenate([2.0 ** np.arange(-120, 61), 0.49999 * 2.0 ** -np.arange(0, 60), [0.25, 0.49, 0.51, 0.75, 1.0, 1.49, 1.51],
                        rng.uniform(1, 2, 400) * 2.0 ** rng.integers(-70, 60, 400)])
    v = np.concatenate([v, -v])
    got = _to_fixed(host, np.ldexp(v, -k), k)
    for x, g in zip(v, got):
        a, b = float(x).as_integer_ratio()  # |g - a / b| <= 1 / 2, in exact arithmetic
        assert abs(2 * (int(g) * b - a)) <= b, (x, g)


@pytest.mark.parametrize("k", [-900, 0, 900])
def test_sum_of_65_bits(host, k):
    """The sum of two integers whose sum may not fit 64 bits, rounded to a double: within half an ulp."""
    rng = np.random.default_rng(2)
    top = int(0.91 * 2 ** 63)
    edge = [0, 1, -1, 2 ** 62, -2 ** 62, top, -top, top - 1, 1 - top]
    x = np.array([a for a in edge for _ in edge] + list(rng.integers(-top, top, 500) >> rng.integers(0, 63, 500)), np.int64)
    y = np.array([b for _ in edge for b in edge] + list(rng.integers(-top, top, 500) >> rng.integers(0, 63, 500)), np.int64)
    out = np.zeros(len(x))
    host.sum_from_fixed(len(x), x.ctypes.data_as(C.c_void_p), y.ctypes.data_as(C.c_void_p), k, out.ctypes.data_as(C.c_void_p))
    for a, b, o in zip(x, y, out):
        exact = int(a) + int(b)
        p, q = (float(o) * 2.0 ** (k // 2) * 2.0 ** (k - k // 2)).as_integer_ratio()
        assert q == 1 and abs(p - exact) * 2 ** 53 <= abs(exact), (a, b, o)


def test_tails_of_a_line_do_not_add_up(host):
    """One large value and 1023 of one sign far below a unit: none of them counts."""
    v = np.r_[2.0 ** 60, np.full(1023, 1e-5)]
    assert _to_fixed(host, v, 0).sum() == 2 ** 60


KINDS = ["noise", "uniform", "unit modulus", "profile", "flat", "decades", "spike", "tone", "comb"]


def _lines(kind, L, n, rng):
    """n lines of L points, (n, L, 2)"""
    i = np.arange(L)
    if kind == "noise":
        return rng.standard_normal((n, L, 2))
    if kind == "uniform":
        return rng.uniform(0, 1, (n, L, 2))
    if kind == "unit modulus":
        t = rng.uniform(0, 2 * np.pi, (n, L))
        return np.stack([np.cos(t), np.sin(t)], -1)
    if kind == "profile":  # two rows across a crack
        c = L / 2 + rng.uniform(-1, 1, (n, 1))
        return np.stack([np.exp(-np.abs(i - c) / 2), np.exp(-np.abs(i - c + 1) / 2)], -1)
    if kind == "flat":
        return 1 + 1e-6 * rng.standard_normal((n, L, 2))
    if kind == "decades":
        return rng.standard_normal((n, L, 2)) * 10.0 ** rng.uniform(-4, 4, (n, L, 2))
    if kind == "spike":  # one value, the others of one sign and far below a unit
        x = 1e-25 * (1 + rng.uniform(0, 1, (n, L, 2)))
        x[:, 0] = 1.0
        return x
    f = rng.integers(1, L // 2, (n, 1))
    t = 2 * np.pi * f * i / L + rng.uniform(0, 2 * np.pi, (n, 1))
    x = np.stack([np.cos(t), np.sin(t)], -1)
    if kind == "comb":  # all of the norm in one residue class: the largest operands of a twiddle multiply
        x[:, i % 8 != 7 % L] = 0.0
    return x


@pytest.mark.parametrize("lgL", range(2, 11))
@pytest.mark.parametrize("kind", KINDS)
def test_lines_are_as_accurate_as_fp64(host, kind, lgL):
    """The transform of a line is no further from long double than a radix-4 FP64 network is: mean relative
    error in the 2-norm of 16 lines, at the worst of eight scales within an octave for each side (a power-of-two
    scale makes the fixed-point error depend on where the norm lies). Below 2^-54 both sides are the rounding of the
    results alone. With twiddles rounded to doubles, as both FP64 and rve_dissipation_noalloc have them, too."""
    L, worst = 1 << lgL, np.zeros(3)
    for a in range(8):
        x = np.ascontiguousarray(_lines(kind, L, 16, np.random.default_rng(lgL)) * 2.0 ** (a / 8))
        e = np.zeros((3, 16))
        host.line_errors(16, lgL, x.ctypes.data_as(C.c_void_p), *[r.ctypes.data_as(C.c_void_p) for r in e])
        worst = np.maximum(worst, e.mean(1))
    print(kind, L, "1e-16:", *np.round(worst * 1e16, 2))
    assert worst[0] <= max(worst[2], 2.0 ** -54)
    assert worst[1] <= max(worst[2], 2.0 ** -54)


def test_multiply_at_the_limit_of_the_scale(host):
    """No partial sum overflows at |a| = 0.91 2^63, and the result is within 2.5 units: two dropped products of at
    most one unit each and the rounding."""
    host.multiply_error.restype = C.c_double
    for lgL in range(2, 11):
        assert host.multiply_error(1 << lgL) <= 2.5
