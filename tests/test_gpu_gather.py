"""The gather at every window of the FP32 range against numpy on the plan's own
grid: tiles of 8 and of 4 cells, row lengths of three to six 16-byte vectors, so
every way the tile copy deals rows to threads.  The tolerance is the stage
tests': window polynomials in FP32 and sums over up to 1728 points."""
import numpy as np
import pytest

from synthetic import fields, meshes
from tests import stage_ref as ref
from tests.gpu_util import lib, rel_l2, run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("grid", [(32, 32, 32), (128, 64, 64)])
@pytest.mark.parametrize("m", [2, 3, 4, 5, 6])
def test_gather_windows(m, grid):
    slp = lib()
    V, T = meshes.box(1.9, 1.0, 1.3, 7, 5, 6)
    o = slp.slp_default_opts()
    o.precision = 32
    o.m = m
    for d in range(3):
        o.grid[d] = grid[d]
    plan = slp.slp_plan(V, T, 3, 1e-2, o)
    try:
        info = slp.slp_query(plan)
        L = info["grid"]
        assert tuple(L) == grid and info["m"] == m
        sigma = fields.random_sigma(T.shape[0] * 3, 11)
        phi = run(slp, plan, slp.SLP_INPUT_SIGMA, sigma, 32, slp.SLP_STAGE_GATHER)
        G = slp.slp_debug_copy(plan, slp.SLP_BUF_GRID_B, np.float32).astype(np.float64).reshape(L[2], L[1], L[0])
        tg = slp.slp_debug_host_array(plan, slp.SLP_HOST_TGT_GRID)
        perm = slp.slp_debug_host_array(plan, slp.SLP_HOST_TGT_PERM)
        want = np.zeros(V.shape[0])
        want[perm] = ref.gather(tg, G, L, m)
        assert rel_l2(phi, want) < 2e-5
    finally:
        slp.slp_destroy(plan)
