"""Both solvers of phi_1 over meshes of every kind: the solve graph (a launch
per inner step), which only systems too large for one launch take by
themselves, and the one-launch solve with the most rows a thread it is compiled
for, reached on a moderate mesh by capping its blocks.  phi_1 against the FP64
oracle, the iteration limit, a zero field and a NaN, each with the solver that
the call names."""
import numpy as np
import pytest

from oracle import fem
from synthetic import fields, meshes
from tests.gpu_util import lib, rel_l2, to_dev, torch_cuda
from tests.test_gpu_solve import fan

pytestmark = pytest.mark.gpu

#: mesh, its blocks at most (0: the graph), rows per thread expected (0: the graph), precision, large
CASES = [("graph, one slice of rows", lambda: meshes.cube_tets(3, 0.4), 0, 0, 32, False),
         ("graph, wide rows", lambda: fan(2, 4), 0, 0, 32, False),
         ("graph, fp64", lambda: meshes.ball_tets(8, 0.2), 0, 0, 64, False),
         ("graph, 12 cells", lambda: meshes.ball_tets(12, 0.2), 0, 0, 32, False),
         ("graph, 28 cells", lambda: meshes.ball_tets(28, 0.2), 0, 0, 32, True),
         ("too many rows for four blocks", lambda: meshes.ball_tets(28, 0.2), 4, 0, 32, True),
         ("eight rows per thread, one block", lambda: meshes.ball_tets(10, 0.2), 1, 8, 32, False),
         ("ten rows per thread", lambda: meshes.ball_tets(28, 0.2), 17, 10, 32, True),
         ("ten rows per thread, fp64", lambda: meshes.ball_tets(20, 0.2), 7, 10, 64, True)]


def _create(slp, case, **kw):
    _, make, most, rows, prec, _ = case
    X, K = make()
    o = slp.slp_default_opts()
    o.precision = prec
    pot = slp.slp_debug_potential_create(X, K, 1e-5 if prec == 32 else 1e-10, most, o, **kw)
    parts, rpt = slp.slp_debug_potential_solver(pot)
    assert rpt == rows and (parts > 0) == (rows > 0) and parts <= most
    return X, K, pot


def _phi1(slp, pot, m, prec):
    torch = torch_cuda()
    d_phi, d_phi1 = (torch.zeros(len(m), dtype=torch.float64 if prec == 64 else torch.float32, device="cuda")
                     for _ in range(2))
    slp.slp_potential_eval(pot, to_dev(m, prec), d_phi, d_phi1, torch.cuda.current_stream())
    torch.cuda.synchronize()
    return d_phi1.double().cpu().numpy()


@pytest.mark.parametrize("case", CASES, ids=[c[0] for c in CASES])
def test_phi1(case):
    slp = lib()
    prec, large = case[4], case[5]
    X, K, pot = _create(slp, case)
    try:
        m = fields.smooth_random(X, 5).astype(np.float32).astype(np.float64)
        phi1 = _phi1(slp, pot, m, prec)
        info = slp.slp_potential_query(pot)
        err = rel_l2(phi1, (fem.phi1_iterative if large else fem.phi1)(X, K, m))
        print(f"{case[0]}: {info['n_free']} unknowns, {info['cg_iterations']} steps, rel-L2 {err:.2e}")
        assert info["cg_residual"] <= info["cg_tolerance"]
        assert err <= (1e-5 if prec == 32 else 1e-9)
        assert np.array_equal(phi1, _phi1(slp, pot, m, prec))  # every sum in a fixed order
        assert not _phi1(slp, pot, np.zeros_like(X), prec).any()
        assert slp.slp_potential_query(pot)["cg_iterations"] == 0
        bad = m.copy()
        bad[len(X) // 2, 1] = np.nan
        with pytest.raises(slp.SlpError) as e:
            _phi1(slp, pot, bad, prec)
        assert e.value.status == slp.SLP_ERR_NONFINITE
        assert np.array_equal(phi1, _phi1(slp, pot, m, prec))
    finally:
        slp.slp_potential_destroy(pot)


@pytest.mark.parametrize("case", [CASES[3], CASES[7]], ids=["graph", "one launch"])
def test_iteration_limit(case):
    slp = lib()
    X, K, pot = _create(slp, case, cg_max_iterations=7)
    try:
        with pytest.raises(slp.SlpError) as e:
            _phi1(slp, pot, fields.smooth_random(X, 5), case[4])
        assert e.value.status == slp.SLP_ERR_TOLERANCE_INFEASIBLE
        assert slp.slp_potential_query(pot)["cg_iterations"] == 7
    finally:
        slp.slp_potential_destroy(pot)
