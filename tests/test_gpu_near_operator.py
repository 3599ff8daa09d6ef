"""The grouped near-field operator at the sizes where its groups and the warps
that share them change: last groups of one, two and three rows, groups shared
by four, two and one warps, more states than one pass takes, both precisions;
against the FP64 oracle at the plan's tolerance, and a state of a batch against
its own evaluation to rounding (the spread's atomics have no fixed order)."""
import numpy as np
import pytest

import oracle
from synthetic import fields, meshes
from tests.gpu_util import lib, rel_l2, run, to_dev, torch_cuda

pytestmark = pytest.mark.gpu

#: 12, 42, 81, 91, 296, 7575 and 29800 vertices
CASES = [(meshes.icosphere(0), 32), (meshes.icosphere(1), 32), (meshes.torus(2.0, 0.5, 9, 9), 32),
         (meshes.torus(2.0, 0.5, 13, 7), 64), (meshes.cube(7), 64), (meshes.torus(2.0, 0.5, 101, 75), 32),
         (meshes.torus(2.0, 0.5, 200, 149), 32)]


@pytest.mark.parametrize("k", range(len(CASES)))
def test_rows_and_states(k):
    torch = torch_cuda()
    slp = lib()
    (V, T), prec = CASES[k]
    tol, dt = (1e-5, torch.float32) if prec == 32 else (1e-10, torch.float64)
    o = slp.slp_default_opts()
    o.precision = prec
    plan = slp.slp_plan(V, T, 3, tol, o)
    try:
        assert slp.slp_query(plan)["near_matrix_nnz"] > 0
        n, states = len(V), 9
        m = np.stack([fields.smooth_random(V, 20 + s) for s in range(states)])
        sel = np.random.default_rng(k).choice(n, min(n, 500), replace=False)
        y, _, _ = oracle.sources(V, T, 3)
        phi = torch.zeros(states, n, dtype=dt, device="cuda")
        slp.slp_eval_states(plan, slp.SLP_INPUT_NODAL_MAG, states, to_dev(m, prec), phi, torch.cuda.current_stream())
        torch.cuda.synchronize()
        got = phi.double().cpu().numpy()
        for s in (0, 3, 8):
            ref, _ = oracle.direct_subset(V, sel, y, oracle.charges(V, T, 3, oracle.KIND_NODAL_MAG, m[s]))
            assert rel_l2(got[s][sel], ref) <= tol
        assert rel_l2(run(slp, plan, slp.SLP_INPUT_NODAL_MAG, m[3], prec), got[3]) <= (1e-6 if prec == 32 else 1e-14)
    finally:
        slp.slp_destroy(plan)
