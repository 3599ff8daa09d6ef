"""Two scalar potentials alive at once whose solves run the same kernel with
different amounts of shared memory: the larger one, evaluated after the smaller
one was created (and evaluated), gives what it gave alone, bit for bit (every
sum of phi_1 has a fixed order)."""
import pytest

from synthetic import fields, meshes
from tests.gpu_util import lib, to_dev, torch_cuda

pytestmark = pytest.mark.gpu

#: one row per thread with the matrix in registers (16.8 and 10.0 KB), eight rows (over 48 KB)
PAIRS = {"one row": (lambda: meshes.ball_tets(16, 0.2), lambda: meshes.ball_tets(12, 0.2)),
         "eight rows": (lambda: meshes.ball_tets(48, 0.2, layers=20), lambda: meshes.ball_tets(44, 0.2, layers=20))}


@pytest.mark.parametrize("name", sorted(PAIRS))
def test_larger_potential_after_a_smaller_one(name):
    torch = torch_cuda()
    slp = lib()
    pots = []

    def phi1(k):
        pot, X = pots[k]
        d_phi, d_phi1 = (torch.zeros(len(X), dtype=torch.float32, device="cuda") for _ in range(2))
        slp.slp_potential_eval(pot, to_dev(fields.smooth_random(X, 5), 32), d_phi, d_phi1, torch.cuda.current_stream())
        torch.cuda.synchronize()
        return d_phi1

    try:
        for make in PAIRS[name]:
            X, K = make()
            pots.append((slp.slp_potential_create(X, K, 1e-5), X))
            if len(pots) == 1:
                first = phi1(0)
        assert torch.equal(phi1(0), first)
        small = phi1(1)
        assert torch.equal(phi1(0), first)
        assert torch.equal(phi1(1), small)
    finally:
        for pot, _ in pots:
            slp.slp_potential_destroy(pot)
