"""The near field computed per pair (charges at the quadrature points): the
fitted kernels and the general one at the sizes where their work lists, odd
last sources and fit ranges change, against the FP64 oracle's direct sum."""
import numpy as np
import pytest

import oracle
from synthetic import fields, meshes
from tests.gpu_util import lib, rel_l2, run

pytestmark = pytest.mark.gpu

#: (mesh, rule, grid, precision, tolerance, deterministic): few targets and odd
#: source counts (1-point rule), long and short items, anisotropic cells, every
#: pair inside the radius, and a tolerance whose radius the FP32 fit does not cover
CASES = [
    (meshes.icosphere(0), 1, (64, 64, 64), 32, 1e-5, 0),
    (meshes.icosphere(1), 7, (64, 64, 64), 32, 1e-5, 1),
    (meshes.cube(5), 1, (128, 128, 128), 32, 1e-5, 0),
    (meshes.cube(9), 3, (256, 256, 256), 32, 1e-5, 0),
    (meshes.box(4.0, 1.0, 0.2, 40, 10, 2), 3, (256, 128, 128), 32, 1e-5, 0),
    (meshes.icosphere(4), 7, (128, 128, 128), 32, 1e-5, 1),
    (meshes.icosphere(3), 3, (128, 128, 128), 32, 1e-6, 0),
    (meshes.icosphere(0), 1, (128, 128, 128), 64, 1e-10, 0),
    (meshes.cube(5), 3, (128, 128, 128), 64, 1e-10, 1),
    (meshes.box(4.0, 1.0, 0.2, 20, 5, 1), 3, (512, 256, 256), 64, 1e-10, 0),
    (meshes.icosphere(3), 1, (256, 256, 256), 64, 1e-10, 0),
]


@pytest.mark.parametrize("case", CASES, ids=[f"{i}-fp{c[3]}-q{c[1]}" for i, c in enumerate(CASES)])
def test_charges_at_points(case):
    slp = lib()
    (V, T), q, grid, prec, tol, det = case
    o = slp.slp_default_opts()
    o.precision, o.deterministic = prec, det
    for d in range(3):
        o.grid[d] = grid[d]
    plan = slp.slp_plan(V, T, q, tol, o)
    try:
        for kind, data in ((slp.SLP_INPUT_SIGMA, fields.random_sigma(q * len(T), 11)),
                           (slp.SLP_INPUT_MAG, fields.random_mag(q * len(T), 12))):
            phi = run(slp, plan, kind, data, prec)
            assert rel_l2(phi, oracle.slp(V, T, q, kind, data)) <= tol
            if det:
                assert np.array_equal(phi, run(slp, plan, kind, data, prec))
    finally:
        slp.slp_destroy(plan)
