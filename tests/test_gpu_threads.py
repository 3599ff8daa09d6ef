"""Plans of different sizes that run the same kernels, evaluated by two host
threads on two streams at once: a kernel's shared-memory limit is state of the
process, so one thread's launches must not lower it under the other's."""
import threading

import numpy as np
import pytest

import oracle
from synthetic import fields, meshes
from tests.gpu_util import lib, rel_l2, to_dev, torch_cuda

pytestmark = pytest.mark.gpu


def _plan(slp, V, T, prec, grid, **kw):
    o = slp.slp_default_opts()
    o.precision = prec
    for d in range(3):
        o.grid[d] = grid[d]
    for k, v in kw.items():
        setattr(o, k, v)
    return slp.slp_plan(V, T, 3, 1e-5 if prec == 32 else 1e-10, o)


@pytest.mark.parametrize("prec,grid,kws", [(64, (64, 64, 64), ({"gather_item_targets": 32}, {"gather_item_targets": 64})),
                                           (64, (64, 64, 64), ({"gather_item_targets": 64}, {"gather_item_targets": 32})),
                                           (32, (64, 64, 64), ({"fuse_plane_passes": 1}, {"fuse_plane_passes": 1}))])
def test_two_host_threads(prec, grid, kws):
    torch = torch_cuda()
    slp = lib()
    bodies = [meshes.icosphere(3), meshes.box(3.0, 1.0, 0.4, 24, 8, 3)]
    plans, fails = [], []
    try:
        for (V, T), kw in zip(bodies, kws):
            plans.append(_plan(slp, V, T, prec, grid, **kw))

        def work(k):
            V, T = bodies[k]
            try:
                m = fields.smooth_random(V, 5)
                s = torch.cuda.Stream()
                with torch.cuda.stream(s):
                    d_in = to_dev(m, prec)
                    d_phi = torch.zeros(len(V), dtype=d_in.dtype, device="cuda")
                    for _ in range(3000):
                        slp.slp_eval(plans[k], slp.SLP_INPUT_NODAL_MAG, d_in, d_phi, s)
                    s.synchronize()
                err = rel_l2(d_phi.double().cpu().numpy(), oracle.slp_nodal(V, T, 3, m))
                assert err <= (1e-5 if prec == 32 else 1e-10), err
            except BaseException as e:  # noqa: BLE001 - reported by the main thread
                fails.append(e)

        threads = [threading.Thread(target=work, args=(k,)) for k in range(2)]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
        assert not fails, fails
    finally:
        for p in plans:
            slp.slp_destroy(p)
