"""The near-field product's sums do not depend on how many states share a pass,
bit for bit, whether one, two or four warps share a group of rows."""
import numpy as np
import pytest

from synthetic import fields, meshes
from tests.gpu_util import lib, run, to_dev, torch_cuda

pytestmark = pytest.mark.gpu

#: groups shared by four, two and one warps, rows longer and shorter than a warp's share
CASES = [(meshes.icosphere(1), 32, None), (meshes.icosphere(4), 32, (64, 64, 64)), (meshes.icosphere(3), 64, (64, 64, 64)),
         (meshes.icosphere(5), 32, (64, 64, 64)), (meshes.torus(2.0, 0.5, 200, 149), 32, (128, 128, 64))]


@pytest.mark.parametrize("k", range(len(CASES)))
def test_states_share_a_pass(k):
    torch = torch_cuda()
    slp = lib()
    (V, T), prec, grid = CASES[k]
    dt = torch.float64 if prec == 64 else torch.float32
    o = slp.slp_default_opts()
    o.precision = prec
    for d in range(3):
        o.grid[d] = grid[d] if grid else 0
    plan = slp.slp_plan(V, T, 3, 1e-5 if prec == 32 else 1e-10, o)
    try:
        n = len(V)
        m = np.stack([fields.smooth_random(V, 20 + s) for s in range(8)])
        alone = []
        for s in range(8):
            run(slp, plan, slp.SLP_INPUT_NODAL_MAG, m[s], prec)
            alone.append(slp.slp_debug_copy(plan, slp.SLP_BUF_NEAR, np.float64 if prec == 64 else np.float32)[:n])
        for count in (1, 2, 5, 8):
            phi = torch.zeros(count, n, dtype=dt, device="cuda")
            slp.slp_eval_states(plan, slp.SLP_INPUT_NODAL_MAG, count, to_dev(m[:count], prec), phi,
                                torch.cuda.current_stream())
            torch.cuda.synchronize()
            got = slp.slp_debug_copy(plan, slp.SLP_BUF_NEAR, np.float64 if prec == 64 else np.float32)
            for s in range(count):
                assert np.any(alone[s]) and np.array_equal(got[s * n:(s + 1) * n], alone[s]), (count, s)
    finally:
        slp.slp_destroy(plan)
