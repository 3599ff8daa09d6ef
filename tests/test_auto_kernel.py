"""What a plan without a given grid does where the grid by points (2 sqrt(points)
cells across the body) cannot carry the radial kernel: a small FP64 mesh at a
tight tolerance keeps the separable kernel on that grid, whose error does not
depend on the tolerance, unless its sum over every pair costs more than the
radial kernel's larger grid; a plan that may not raise its grid is refused."""
import numpy as np
import pytest

import oracle
from synthetic import fields, meshes
from tests.gpu_util import lib, rel_l2, run

#: mesh, rule, the grid by points
SMALL = {"sphere0": (lambda: meshes.icosphere(0), 7, (32, 32, 32)), "sphere1": (lambda: meshes.icosphere(1), 1, (32, 32, 32)),
         "cube3": (lambda: meshes.cube(3), 1, (32, 32, 32)),
         "plate9": (lambda: meshes.box(3.0, 1.0, 0.1, 9, 3, 1), 1, (32, 32, 32)),
         "torus": (lambda: meshes.torus(1.0, 0.3, 17, 7), 1, (64, 64, 32)),
         "rod": (lambda: meshes.box(0.2, 0.3, 5.0, 1, 2, 17), 1, (32, 32, 64))}


def _opts(slp, prec, **kw):
    o = slp.slp_default_opts()
    o.precision = prec
    for k, v in kw.items():
        setattr(o, k, v)
    return o


def _info(slp, V, T, q, tol, o):
    p = slp.slp_plan(V, T, q, tol, o)
    try:
        return slp.slp_query(p)
    finally:
        slp.slp_destroy(p)


def test_every_pair_against_a_larger_grid():
    """A plate of 252 vertices: charges at its points cost the separable kernel 400 us
    more than the radial one's grid saves at 1e-10, which at 1e-13 is four times as large."""
    slp = lib()
    V, T = meshes.box(4.0, 1.0, 0.2, 20, 5, 1)
    modes = [_info(slp, V, T, 1, tol, _opts(slp, 64, device=-1))["kernel_mode"] for tol in (1e-10, 1e-13)]
    assert modes == [slp.SLP_KERNEL_RADIAL, slp.SLP_KERNEL_SEPARABLE]


@pytest.mark.parametrize("raise_grid", [0, 1])
@pytest.mark.parametrize("tol", [5e-10, 1e-10, 1e-13])
@pytest.mark.parametrize("name", sorted(SMALL))
def test_small_fp64_meshes_keep_the_separable_kernel(name, tol, raise_grid):
    slp = lib()
    make, q, grid = SMALL[name]
    V, T = make()
    info = _info(slp, V, T, q, tol, _opts(slp, 64, device=-1, allow_grid_raise=raise_grid))
    assert info["kernel_mode"] == slp.SLP_KERNEL_SEPARABLE and tuple(info["grid"]) == grid
    # larger meshes, looser tolerances and a kernel that is named take the radial one
    radial = _info(slp, V, T, q, tol, _opts(slp, 64, device=-1, kernel_mode=slp.SLP_KERNEL_RADIAL))
    assert radial["kernel_mode"] == slp.SLP_KERNEL_RADIAL and max(radial["grid"]) > max(grid)
    assert _info(slp, V, T, q, 1e-8, _opts(slp, 64, device=-1))["kernel_mode"] == slp.SLP_KERNEL_RADIAL
    V, T = meshes.icosphere(3)
    assert _info(slp, V, T, 7, tol, _opts(slp, 64, device=-1))["kernel_mode"] == slp.SLP_KERNEL_RADIAL


@pytest.mark.parametrize("tol", [1e-5, 1e-6])
@pytest.mark.parametrize("mode", ["AUTO", "RADIAL"])
def test_refused_where_the_grid_may_not_be_raised(tol, mode):
    slp = lib()
    V, T = meshes.icosphere(0)
    kw = dict(device=-1, kernel_mode=getattr(slp, "SLP_KERNEL_" + mode))
    with pytest.raises(slp.SlpError) as e:
        _info(slp, V, T, 1, tol, _opts(slp, 32, allow_grid_raise=0, **kw))
    assert e.value.status == slp.SLP_ERR_TOLERANCE_INFEASIBLE
    assert _info(slp, V, T, 1, tol, _opts(slp, 32, **kw))["kernel_mode"] == slp.SLP_KERNEL_RADIAL


@pytest.mark.gpu
@pytest.mark.parametrize("name", sorted(SMALL))
def test_error_is_rounding(name):
    """The separable kernel subtracts exactly what it adds, and its smooth part is a
    tenth of the potential: the error is rounding, 1.1e-16 for each of at most a
    few hundred partial sums of one sign."""
    slp = lib()
    make, q, _ = SMALL[name]
    V, T = make()
    m = fields.smooth_random(V, 5)
    plan = slp.slp_plan(V, T, q, 1e-10, _opts(slp, 64))
    try:
        phi = run(slp, plan, slp.SLP_INPUT_NODAL_MAG, m, 64)
        err = rel_l2(phi, oracle.slp_nodal(V, T, q, m))
        print(f"{name}: rel-L2 {err:.2e}")
        assert err <= 1.6e-14
    finally:
        slp.slp_destroy(plan)
