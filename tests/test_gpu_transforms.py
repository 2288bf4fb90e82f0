"""FP64 line transforms (64-bit fixed point) at every line length and at the shapes where a launch rule
changes: D and Gamma of a device field through rve_dissipation_noalloc (forward x, y, z, gradient, inverse)
against numpy in FP64.

Tolerance. D is a sum of squares of the field and its gradient. A transform of L <= 1024 points has a
relative error below 3.5e-16 in the 2-norm in FP64 (numpy) and below that in fixed point; a gradient takes
at most six, so the gradient is within 2 * 6 * 3.5e-16 = 4.2e-15 and its square within 8.4e-15; the sums of
up to 2^18 non-negative terms add less than 1e-15 (pairwise trees). Bound: 2e-14.
"""
import ctypes as C

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

GRIDS = [(4, 64, 1), (8, 32, 1), (16, 16, 1), (32, 32, 1), (64, 4, 1), (64, 8, 1), (64, 16, 1), (128, 256, 1),
         (256, 128, 1), (512, 32, 1), (32, 512, 1), (512, 512, 1), (1024, 64, 1), (64, 1024, 1), (16, 32, 8), (64, 32, 4),
         (16, 16, 64), (8, 16, 128), (32, 32, 32)]


def _numpy(phi, n, dim, ell):
    h = np.fft.rfftn(phi, axes=(0, 1, 2))
    e = phi * phi / (2 * ell)
    for ax in range(3 - dim, 3):
        m = phi.shape[ax]
        k = np.fft.fftfreq(m, 1.0 / m)
        k[np.abs(k) * 2 == m] = 0.0
        xi = (2 * np.pi * k / m)[: h.shape[ax]].reshape([-1 if a == ax else 1 for a in range(3)])
        e += 0.5 * ell * np.fft.irfftn(1j * xi * h, s=phi.shape, axes=(0, 1, 2)) ** 2
    return float(e.sum())


def _library(phi, n, dim, ell):
    import torch
    from paper_2508_07424_gb300 import build, capi
    build.build()
    t = torch.as_tensor(np.ascontiguousarray(phi), device="cuda")
    gid = torch.zeros(phi.size, device="cuda", dtype=torch.int32)
    gc = torch.ones(1, device="cuda", dtype=torch.float64)
    A = torch.tensor([[1.0, 1.0, 0.0 if dim == 2 else 1.0, 0.0, 0.0, 0.0]], device="cuda", dtype=torch.float64)
    out = torch.zeros(2, device="cuda", dtype=torch.float64)
    capi.check(capi.lib().rve_dissipation_noalloc(dim, (C.c_int * 3)(*n), ell, 1,
                                                  *[C.c_void_p(x.data_ptr()) for x in (gid, gc, A, t, out)], None), "D")
    torch.cuda.synchronize()
    return out.cpu().numpy()


@pytest.mark.parametrize("kind", ["uniform", "peaks", "magnitudes"])
@pytest.mark.parametrize("n", GRIDS)
def test_functional_of_random_fields(n, kind):
    rng = np.random.default_rng(n[0] * 7 + n[1] * 3 + n[2])
    dim = 2 if n[2] == 1 else 3
    shape = n[::-1]
    if kind == "uniform":
        phi = rng.uniform(0.0, 1.0, shape)
    elif kind == "peaks":  # nearly flat with a few large values, as at crack tips
        phi = 1e-3 * rng.uniform(0.0, 1.0, shape)
        phi.flat[rng.integers(0, phi.size, 3)] = 1.0
    else:  # rows of very different size, some of them zero
        phi = rng.standard_normal(shape) * 10.0 ** rng.integers(-12, 12, (shape[0], shape[1], 1))
        phi[:, ::5] = 0.0
    ref = _numpy(phi, n, dim, 2.0)
    got = _library(phi, n, dim, 2.0)
    assert abs(got[0] - ref) <= 2e-14 * ref and got[0] == got[1]


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_non_finite_values_reach_the_result(bad):
    phi = np.random.default_rng(3).uniform(0.0, 1.0, (1, 64, 64))
    phi[0, 5, 9] = bad
    assert not np.isfinite(_library(phi, (64, 64, 1), 2, 2.0)).any()


def test_zero_field():
    assert (_library(np.zeros((1, 32, 32)), (32, 32, 1), 2, 2.0) == 0.0).all()


@pytest.mark.parametrize("precision", ["fp64", "fp32r"])
def test_a_smaller_grid_does_not_take_shared_memory_from_a_larger_one(monkeypatch, precision):
    """The shared-memory opt-in belongs to the kernel, which serves every line length: a handle of 512-point
    columns (37 KB in FP64) used between two calls of one of 1024-point columns (74 KB)."""
    import synth
    from paper_2508_07424_gb300 import build
    from paper_2508_07424_gb300.rve import Rve
    build.build()
    monkeypatch.setenv("PFF_TILE_CW", "2")
    rng = np.random.default_rng(1)
    out = {}
    hs = {ny: Rve.from_workload(synth.Workload(synth.homogeneous((64, ny)), ell=2.0, precision=precision)) for ny in (1024, 512)}
    phi = {ny: rng.uniform(0.0, 1.0, (1, ny, 64)) for ny in hs}
    for ny in (1024, 512, 1024):
        got = hs[ny].dissipation(phi[ny]), hs[ny].mech_solve()
        assert out.setdefault(ny, got)[0] == got[0]
