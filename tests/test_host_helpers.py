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
    # -Bsymbolic: the stand-ins for CUDA calls are the library's own, whatever else the process has loaded
    subprocess.run(["g++", "-std=c++17", "-O2", "-fPIC", "-shared", "-Wl,-Bsymbolic", "-I", os.path.join(cuda, "include"), "-o", so,
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


def test_shared_memory_opt_in(host):
    """Only ever raised, not asked for again, an error is passed on and not remembered, and no memory for the
    table is an error code too: an exception would leave through an entry point with C linkage."""
    calls, size = C.c_int(), C.c_size_t()

    def raise_to(kernel, kb, no_memory=0):
        e = host.smem_raise(C.c_size_t(kernel), C.c_size_t(kb * 1024), no_memory, C.byref(calls), C.byref(size))
        return e, calls.value, size.value // 1024

    assert raise_to(16, 32) == (0, 0, 0)
    assert raise_to(16, 100, no_memory=1) == (2, 0, 0)  # cudaErrorMemoryAllocation
    assert raise_to(16, 100) == (0, 1, 100)
    assert raise_to(16, 60) == (0, 1, 100)
    assert raise_to(16, 100, no_memory=1) == (0, 1, 100)
    assert raise_to(32, 228) == (1, 2, 228)  # cudaErrorInvalidValue
    assert raise_to(32, 200) == (0, 3, 200)
