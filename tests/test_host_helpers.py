"""Host-side helpers of the library, compiled on their own."""
import ctypes as C
import mmap
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("host") / "host_helpers.so")
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.run(["g++", "-std=c++17", "-O2", "-fPIC", "-shared", "-I", os.path.join(cuda, "include"), "-o", so,
                    os.path.join(HERE, "host_helpers.cpp")], check=True)
    return C.CDLL(so)


@pytest.mark.parametrize("offset,size", [(0, 1), (8, 8), (4088, 16), (3, 100001), (0, 1 << 20)])
def test_mapping_pages_keeps_what_they_hold(host, offset, size):
    a = np.random.default_rng(size).integers(0, 256, offset + size + 70000, np.uint8)
    b = a.copy()
    host.map_pages(C.c_void_p(a.ctypes.data + offset), C.c_size_t(size))
    assert (a == b).all()


def test_mapping_pages_refuses_without_harm(host):
    """No buffer, no length, memory that cannot be written, and an address that is not mapped at all."""
    host.map_pages(None, C.c_size_t(8))
    m = mmap.mmap(-1, 1 << 16, prot=mmap.PROT_READ)
    at = np.frombuffer(m, np.uint8).ctypes.data
    host.map_pages(C.c_void_p(at), C.c_size_t(0))
    host.map_pages(C.c_void_p(at), C.c_size_t(1 << 16))
    host.map_pages(C.c_void_p(1 << 44), C.c_size_t(1 << 16))
