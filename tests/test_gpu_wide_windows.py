"""Wide windows (2m > 10: one tile per block, a warp per residue of the z
planes) and gather items of fewer targets than warps, for every window width
they are compiled for, on meshes with one and with many sources per cell,
against the FP64 oracle at the plan's tolerance."""
import pytest

import oracle
from synthetic import fields, meshes
from tests.gpu_util import lib, rel_l2, run

pytestmark = pytest.mark.gpu

CASES = [(m, prec, tol, mesh, grid)
         for m, prec, tol in ((6, 32, 1e-5), (6, 64, 1e-8), (7, 64, 1e-10), (8, 64, 1e-10))
         for mesh, grid in (("octa", 64), ("cube", 128), ("sphere", 64))]


@pytest.mark.parametrize("m,prec,tol,mesh,grid", CASES)
def test_nodal_field(m, prec, tol, mesh, grid):
    slp = lib()
    V, T, q = {"octa": (*meshes.icosphere(0), 1), "cube": (*meshes.cube(5), 3), "sphere": (*meshes.icosphere(3), 7)}[mesh]
    o = slp.slp_default_opts()
    o.precision, o.m = prec, m
    for d in range(3):
        o.grid[d] = grid
    plan = slp.slp_plan(V, T, q, tol, o)
    try:
        assert slp.slp_query(plan)["m"] == m
        x = fields.smooth_random(V, 3)
        phi = run(slp, plan, slp.SLP_INPUT_NODAL_MAG, x, prec)
        assert rel_l2(phi, oracle.slp_nodal(V, T, q, x)) <= tol
    finally:
        slp.slp_destroy(plan)
