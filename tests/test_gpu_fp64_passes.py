"""FP64 evaluations on either side of the line between passes launched early and
passes launched one after another (the y pass with fewer than 64, 64 to 304 and
more blocks), behind the spread kernel and behind both gridding products; at the
plan's tolerance, and deterministic plans bit for bit from call to call."""
import numpy as np
import pytest

import oracle
from synthetic import fields, meshes
from tests.gpu_util import lib, rel_l2, run

pytestmark = pytest.mark.gpu

#: mesh, grid
CASES = {"few blocks": (meshes.box(4.0, 1.0, 0.2, 20, 5, 1), (128, 128, 128)),
         "up to two per SM": (meshes.cube(7), (128, 128, 128)),
         "many blocks": (meshes.icosphere(2), (256, 256, 256))}


@pytest.mark.parametrize("deterministic", [0, 1])
@pytest.mark.parametrize("name", sorted(CASES))
def test_point_plans(name, deterministic):
    slp = lib()
    (V, T), grid = CASES[name]
    o = slp.slp_default_opts()
    o.precision, o.deterministic, o.kernel_mode = 64, deterministic, slp.SLP_KERNEL_RADIAL
    for d in range(3):
        o.grid[d] = grid[d]
    plan = slp.slp_plan(V, T, 1, 1e-10, o)
    try:
        m = fields.smooth_random(V, 5)
        phi = run(slp, plan, slp.SLP_INPUT_NODAL_MAG, m, 64)
        assert rel_l2(phi, oracle.slp_nodal(V, T, 1, m)) <= 1e-10
        for _ in range(5 if deterministic else 0):
            assert np.array_equal(phi, run(slp, plan, slp.SLP_INPUT_NODAL_MAG, m, 64))
    finally:
        slp.slp_destroy(plan)


@pytest.mark.parametrize("mesh", [meshes.icosphere(2), meshes.cube(7)], ids=["sphere", "cube"])
def test_triangle_plans(mesh):
    """The triangle products have a fixed order, so an evaluation repeats bit for bit."""
    slp = lib()
    V, T = mesh
    o = slp.slp_default_opts()
    o.precision, o.integration = 64, 1
    for d in range(3):
        o.grid[d] = 128
    plan = slp.slp_plan(V, T, 3, 1e-10, o)
    try:
        m = fields.smooth_random(V, 5)
        phi = run(slp, plan, slp.SLP_INPUT_NODAL_MAG, m, 64)
        assert rel_l2(phi, oracle.slp_p0(V, T, oracle.element_charges(V, T, m))) <= 1e-10
        for _ in range(5):
            assert np.array_equal(phi, run(slp, plan, slp.SLP_INPUT_NODAL_MAG, m, 64))
    finally:
        slp.slp_destroy(plan)
