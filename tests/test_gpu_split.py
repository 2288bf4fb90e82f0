"""A strain that is not finite ends an equilibrium solve with the spectral split as a breakdown.

The positive and negative parts of a NaN eigenvalue compare as zero, so the split stress of such a voxel is
zero and the residual does not show it; the tangent has to.
"""
import ctypes as C

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("component", [0, 1, 2])
@pytest.mark.parametrize("precision", ["fp64", "fp32r"])
def test_non_finite_strain_is_a_breakdown(precision, component, bad):
    from paper_2508_07424_gb300 import build, capi
    from paper_2508_07424_gb300.rve import Rve
    build.build()
    crack = synth.Crack(synth.CRACK_CTE, row=8, x0=0, length=4, phi_M=0.8)
    w = synth.Workload(synth.homogeneous((32, 32), crack=crack), ell=2.0, split=1, precision=precision)
    g = Rve.from_workload(w)
    x = np.zeros((3, 1, 32, 32))
    x[component, 0, 5, 7] = bad
    g.set(capi.RVE_FIELD_FLUCT1, x)
    it = C.c_int()
    assert capi.lib().rve_mech_solve(g.h, C.byref(it)) == capi.RVE_EBREAKDOWN
