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


def test_tails_of_a_line_do_not_add_up(host):
    """One large value and 1023 of one sign far below a unit: none of them counts."""
    v = np.r_[2.0 ** 60, np.full(1023, 1e-5)]
    assert _to_fixed(host, v, 0).sum() == 2 ** 60
