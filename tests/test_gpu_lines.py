"""Transforms at every line length on every axis, where a value in the wrong place shows.

Each voxel has a grain of its own choice out of six with different toughness, stiffness and anisotropic cleavage
tensor, so D, Gamma and the solved fields depend on where every gradient and every strain component lands: a line
that comes back permuted, reversed or transformed the wrong way changes them by far more than the bounds
(the first test shows that on the oracle). Both entry points are used, since they make their twiddles in
different ways.

Tolerances. Functional: a gradient takes at most six transforms of 3.5e-16 each (2-norm), times pi for the
frequencies over the ratio of gradient to field (at least 0.9 for white noise in [0, 1]): 7.4e-15, twice that for
its square, 1e-15 for the sums, the same for the oracle, times the ratio of the largest to the smallest weight.
Solves: both sides stop at 1e-13 of the right-hand side, with condition numbers up to 200: 1e-10, as in the
parity tests.
"""
import ctypes as C

import numpy as np
import pytest

import synth
from oracle import solver as S
from oracle import spectral as sp
from tests.helpers import rel, sym_components

GRIDS = [(4, 128), (8, 32), (16, 16), (32, 8), (64, 4), (128, 64), (256, 32), (512, 8), (1024, 16), (16, 128), (16, 256),
         (16, 512), (8, 1024), (4, 8, 16), (16, 4, 8), (8, 16, 32), (8, 8, 64), (8, 8, 128), (8, 4, 256), (4, 8, 512),
         (8, 4, 1024), (64, 8, 4), (8, 32, 4), (128, 4, 4), (8, 256, 4)]


def _model(n):
    rng = np.random.default_rng(sum(n))
    w = synth.Workload(synth.voronoi(n, 6, 7, orientation="inplane" if len(n) == 2 else "so3", beta=1.0, sigma_Gc=0.4), ell=2.0)
    w.micro.grain_id = rng.integers(0, 6, w.micro.grain_id.shape).astype(np.int32)
    kw = dict(tol_mech=1e-13, tol_dmg=1e-13)
    return w, S.Model(w.micro, S.params_from_workload(w, **kw)), rng, kw


@pytest.mark.parametrize("n", [(16, 32), (8, 4, 16)])
def test_the_functional_depends_on_the_order_of_every_line(n, monkeypatch):
    _, model, rng, _ = _model(n)
    phi = rng.uniform(0, 1, model.grid)
    ref = model.dissipation(phi), model.crack_surface(phi)
    true = sp.ifft_real
    wrong = [lambda U, a=a: np.flip(true(U), a) for a in (-3, -2, -1) if model.grid[a] > 1]  # reversed lines
    wrong += [lambda U, a=a: np.roll(true(U), 1, a) for a in (-3, -2, -1) if model.grid[a] > 1]
    wrong.append(lambda U: true(np.conj(U)))  # the wrong direction
    for f in wrong:
        monkeypatch.setattr(sp, "ifft_real", f)
        got = model.dissipation(phi), model.crack_surface(phi)
        monkeypatch.setattr(sp, "ifft_real", true)
        assert all(abs(g - r) > 1e-6 * r for g, r in zip(got, ref))


@pytest.mark.gpu
@pytest.mark.parametrize("n", GRIDS)
def test_functional(n):
    import torch
    from paper_2508_07424_gb300 import build, capi
    from paper_2508_07424_gb300.rve import Rve
    build.build()
    w, model, rng, kw = _model(n)
    m = w.micro
    phi = rng.uniform(0, 1, model.grid)
    ref = model.dissipation(phi), model.crack_surface(phi)
    tol = 3.2e-14 * np.array([2 * m.Gc.max() / m.Gc.min(), 2.0])
    got = Rve.from_workload(w, **kw).dissipation(phi)
    assert (np.abs(np.subtract(got, ref)) <= tol * ref).all()
    # the same from device buffers
    at = [(0, 0), (1, 1), (0, 1)] if m.dim == 2 else [(0, 0), (1, 1), (2, 2), (1, 2), (0, 2), (0, 1)]
    A = np.zeros((m.n_grains, 6))
    for g in range(m.n_grains):
        v = np.argwhere(m.grain_id == g)[0]
        A[g, : len(at)] = [model.A[(*p, *v)] for p in at]
    bufs = [torch.as_tensor(np.ascontiguousarray(a), device="cuda") for a in (m.grain_id, m.Gc, A, phi, np.zeros(2))]
    capi.check(capi.lib().rve_dissipation_noalloc(m.dim, (C.c_int * 3)(*m.n), w.ell, m.n_grains,
                                                  *[C.c_void_p(b.data_ptr()) for b in bufs], None), "functional")
    torch.cuda.synchronize()
    assert (np.abs(bufs[-1].cpu().numpy() - ref) <= tol * ref).all()


@pytest.mark.gpu
@pytest.mark.parametrize("n", GRIDS)
def test_solves_voxel_by_voxel(n):
    from paper_2508_07424_gb300 import build, capi
    from paper_2508_07424_gb300.rve import Rve
    build.build()
    w, model, rng, kw = _model(n)
    g = Rve.from_workload(w, **kw)
    phi = rng.uniform(0.0, 0.9, model.grid)
    g.set(capi.RVE_FIELD_PHI, phi)
    g.mech_solve()
    F1, _ = S.mech_solve(model, phi, np.zeros((model.d, model.d) + model.grid))
    assert rel(g.get(capi.RVE_FIELD_FLUCT1), sym_components(F1, model.d)) < 1e-10
    psi1 = model.drive(model.fB + 0.5 * (F1 + np.swapaxes(F1, 0, 1)))
    assert rel(g.get(capi.RVE_FIELD_PSI1), psi1) < 1e-10
    H0, ini = rng.uniform(0, 0.5, model.grid), rng.uniform(0, 0.2, model.grid)
    g.set(capi.RVE_FIELD_H, H0)
    g.set(capi.RVE_FIELD_PSI_INI, ini)
    ref, _ = S.damage_solve(model, S.history_field(model, 0.5, psi1, ini, H0), phi)
    D, _ = g.damage_solve(0.5)
    assert rel(g.get(capi.RVE_FIELD_PHI_TRIAL), ref) < 1e-10
    assert abs(D - model.dissipation(ref)) < 1e-10 * D
