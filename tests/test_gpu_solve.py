"""The one-launch solve of phi_1 at the sizes where its variants change: one
part and several, one and two rows per thread with the matrix in registers,
rows too wide for registers, and more rows per thread; phi_1 against the FP64
oracle (direct solve, or conjugate gradients to 1e-13 on the larger meshes).
The FP32 plan's solve stops at |b - S x| <= 1e-7 |b|."""
import numpy as np
import pytest

from oracle import fem
from synthetic import fields, meshes
from tests.gpu_util import lib, rel_l2, to_dev, torch_cuda

pytestmark = pytest.mark.gpu


def fan(level, layers):
    """Ball of icosphere shells about one centre node, whose row couples to every node of the first shell."""
    V, T = meshes.icosphere(level)
    n = len(V)
    X = np.concatenate([[[0.0, 0.0, 0.0]]] + [V * (0.2 * (k + 1) / layers) for k in range(layers)])
    T = np.sort(T, 1)
    tets = [np.concatenate([np.zeros((len(T), 1), int), T + 1], 1)]
    for k in range(layers - 1):
        lo, hi = T + 1 + k * n, T + 1 + (k + 1) * n
        tets += [np.stack([lo[:, 0], lo[:, 1], lo[:, 2], hi[:, 2]], 1), np.stack([lo[:, 0], lo[:, 1], hi[:, 1], hi[:, 2]], 1),
                 np.stack([lo[:, 0], hi[:, 0], hi[:, 1], hi[:, 2]], 1)]
    return X, np.concatenate(tets).astype(np.int32)


CASES = [("one part", lambda: meshes.ball_tets(4, 0.2, layers=1), False),
         ("two parts", lambda: meshes.ball_tets(4, 0.2), False),
         ("wide rows", lambda: fan(2, 4), False),
         ("wide rows, many parts", lambda: fan(4, 8), False),
         ("one row per thread", lambda: meshes.ball_tets(12, 0.2), False),
         ("two rows per thread", lambda: meshes.ball_tets(28, 0.2), True),
         ("four rows per thread", lambda: meshes.ball_tets(36, 0.2), True),
         ("eight rows per thread", lambda: meshes.ball_tets(44, 0.2, layers=20), True)]


@pytest.mark.parametrize("case", CASES, ids=[c[0] for c in CASES])
def test_phi1(case):
    torch = torch_cuda()
    slp = lib()
    _, make, large = case
    X, K = make()
    m = fields.smooth_random(X, 5).astype(np.float32).astype(np.float64)
    pot = slp.slp_potential_create(X, K, 1e-5)
    try:
        d_phi, d_phi1 = (torch.zeros(len(X), dtype=torch.float32, device="cuda") for _ in range(2))
        first = None
        for _ in range(2):
            slp.slp_potential_eval(pot, to_dev(m, 32), d_phi, d_phi1, torch.cuda.current_stream())
            torch.cuda.synchronize()
            first = d_phi1.clone() if first is None else first
        info = slp.slp_potential_query(pot)
        ref = (fem.phi1_iterative if large else fem.phi1)(X, K, m)
        err = rel_l2(d_phi1.double().cpu().numpy(), ref)
        print(f"{case[0]}: {info['n_free']} unknowns, {info['cg_iterations']} steps, rel-L2 {err:.2e}")
        assert info["cg_residual"] <= info["cg_tolerance"]
        assert err <= 1e-5  # the plan's tolerance
        assert torch.equal(first, d_phi1)  # every sum in a fixed order
    finally:
        slp.slp_potential_destroy(pot)
