"""Which grid a plan without a given one gets (host-only plans): the rule by
estimated cost against the same grid given explicitly, and the rule by the
number of points where that one still holds."""
import math

import numpy as np
import pytest

from synthetic import meshes
from tests.gpu_util import lib

MESHES = {
    "sphere": lambda: meshes.icosphere(2),
    "plate": lambda: meshes.box(3.0, 1.0, 0.1, 9, 3, 1),
    "rod": lambda: meshes.box(0.2, 0.3, 5.0, 1, 2, 17),
    "torus": lambda: meshes.torus(1.0, 0.3, 17, 7),
}


def _info(slp, V, T, q, tol, prec, grid=(0, 0, 0), **kw):
    o = slp.slp_default_opts()
    o.device = -1
    o.precision = prec
    for d in range(3):
        o.grid[d] = grid[d]
    for k, v in kw.items():
        setattr(o, k, v)
    p = slp.slp_plan(V, T, q, tol, o)
    try:
        return slp.slp_query(p)
    finally:
        slp.slp_destroy(p)


def _extent(V):
    ctr = (V.min(axis=0) + V.max(axis=0)) / 2
    return V.max(axis=0) - V.min(axis=0), 2 * np.linalg.norm(V - ctr, axis=1).max()


@pytest.mark.parametrize("prec,tol", [(32, 1e-3), (32, 1e-6), (64, 1e-5), (64, 1e-9)])
@pytest.mark.parametrize("q", [1, 7])
@pytest.mark.parametrize("name", sorted(MESHES))
def test_by_cost_is_a_grid_a_user_could_give(name, q, prec, tol):
    slp = lib()
    V, T = MESHES[name]()
    a = _info(slp, V, T, q, tol, prec)
    L = a["grid"]
    assert all(v & (v - 1) == 0 and 16 <= v <= 1024 for v in L)
    assert a["kernel_mode"] == slp.SLP_KERNEL_RADIAL and not a["grid_raised"]
    # equal spacing: rounding to a power of two moves an axis by sqrt(2) at most
    D, diam = _extent(V)
    h = [(D[d] + diam) / L[d] for d in range(3) if 16 < L[d] < 1024]
    assert not h or max(h) / min(h) <= 2 * (1 + 1e-9)
    # the same grid given explicitly: the same transform, and a near radius that
    # the larger share of the tolerance makes shorter
    b = _info(slp, V, T, q, tol, prec, L, kernel_mode=slp.SLP_KERNEL_RADIAL, allow_grid_raise=0)
    for key in ("grid", "modes", "m", "kernel_mode", "tolerance"):
        assert a[key] == b[key], key
    assert a["eps_near"] >= b["eps_near"]


@pytest.mark.parametrize("name", sorted(MESHES))
@pytest.mark.parametrize("case", ["integration", "one axis given", "expsum"])
def test_other_plans_keep_the_rule_by_points(name, case):
    slp = lib()
    V, T = MESHES[name]()
    q, grid, kw = 3, (0, 0, 0), {"allow_grid_raise": 1}
    if case == "integration":
        kw["integration"] = 1
    elif case == "one axis given":
        grid = (0, 128, 0)
    else:
        kw["kernel_mode"] = slp.SLP_KERNEL_EXPSUM
    info = _info(slp, V, T, q, 1e-3, 32, grid, **kw)
    D, diam = _extent(V)
    points = info["n_sources"] + info["n_targets"]
    cells = max(16.0, 2 * math.sqrt(points))
    want = []
    for d in range(3):
        v = 16
        while v < cells * (D[d] + diam) / (D.max() + diam) and v < 1024:
            v <<= 1
        want.append(grid[d] or v)
    if not info["grid_raised"]:
        assert info["grid"] == want
    else:
        assert all(g >= w for g, w in zip(info["grid"], want))
