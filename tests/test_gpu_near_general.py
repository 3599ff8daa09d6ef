"""RADIAL plans whose near radius the fitted kernels do not cover: the general
kernel for charges at the points and, in FP64, the operator's assembly from
erfc, against the FP64 oracle; and the fitted kernels just inside their range.

The bounds are what the arithmetic and the windows reach, not the tolerance:
FP32 rounding of the potential (2e-6), and the half-width-8 window's aliasing in
FP64 (1e-12)."""
import numpy as np
import pytest

import oracle
from synthetic import fields, meshes
from tests.gpu_util import lib, rel_l2, run

pytestmark = pytest.mark.gpu

#: mesh, rule, grid, precision, tolerance, deterministic, fitted
CASES = [(meshes.icosphere(3), 3, (128, 128, 128), 32, 5e-7, 0, True),
         (meshes.icosphere(3), 3, (128, 128, 128), 32, 2e-7, 0, False),
         (meshes.cube(5), 1, (128, 128, 128), 32, 2e-7, 1, False),
         (meshes.box(4.0, 1.0, 0.2, 40, 10, 2), 3, (256, 128, 128), 32, 1e-7, 0, False),
         (meshes.icosphere(2), 3, (256, 256, 256), 64, 1e-19, 0, True),
         (meshes.icosphere(2), 3, (256, 256, 256), 64, 1e-21, 0, False),
         (meshes.cube(3), 1, (256, 256, 256), 64, 1e-21, 1, False)]


@pytest.mark.parametrize("case", CASES, ids=[f"{i}-fp{c[3]}-{c[4]:g}" for i, c in enumerate(CASES)])
def test_radius_beyond_the_fits(case):
    slp = lib()
    (V, T), q, grid, prec, tol, det, fitted = case
    o = slp.slp_default_opts()
    o.precision, o.deterministic, o.kernel_mode = prec, det, slp.SLP_KERNEL_RADIAL
    for d in range(3):
        o.grid[d] = grid[d]
    plan = slp.slp_plan(V, T, q, tol, o)
    try:
        assert slp.slp_query(plan)["kernel_mode"] == slp.SLP_KERNEL_RADIAL
        assert slp.slp_debug_near_fit(plan) == fitted
        bound = 2e-6 if prec == 32 else 1e-12
        for kind, data in ((slp.SLP_INPUT_SIGMA, fields.random_sigma(q * len(T), 11)),
                           (slp.SLP_INPUT_MAG, fields.random_mag(q * len(T), 12)),
                           (slp.SLP_INPUT_NODAL_MAG, fields.smooth_random(V, 13))):
            phi = run(slp, plan, kind, data, prec)
            err = rel_l2(phi, oracle.slp(V, T, q, kind, data))
            print(f"{case[3:]}: kind {kind} rel-L2 {err:.2e}")
            assert err <= bound
            if det:
                assert np.array_equal(phi, run(slp, plan, kind, data, prec))
    finally:
        slp.slp_destroy(plan)
