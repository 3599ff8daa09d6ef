"""The separate FFT passes at every transform length with its own compiled
kernel, along each axis, against numpy's transforms of the same buffers.

Tolerance: a radix-8 stage is three additions and one twiddle product on the
way of each element, a relative error of at most 6 u in the l2 norm, and a
length has at most four stages, so one direction stays below 32 u (with the
split of a row pair) and the z pass, both directions and the multiply, below
64 u; twice that covers numpy's own rounding and the order in which the spread
adds up in two runs."""
import numpy as np
import pytest

from synthetic import fields, meshes
from tests import stage_ref as ref
from tests.gpu_util import lib, rel_l2, run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [32, 64])
@pytest.mark.parametrize("axis", [0, 1, 2])
@pytest.mark.parametrize("length", [64, 128, 256, 512, 1024])
def test_passes_along_axis(length, axis, prec):
    slp = lib()
    dims, div, grid = [0.25] * 3, [2] * 3, [32] * 3
    dims[axis], div[axis], grid[axis] = 2.0, 12, length
    V, T = meshes.box(*dims, *div)
    o = slp.slp_default_opts()
    o.precision = prec
    o.fuse_plane_passes = 0
    for d in range(3):
        o.grid[d] = grid[d]
    plan = slp.slp_plan(V, T, 3, 1e-3, o)
    try:
        info = slp.slp_query(plan)
        L, n = info["grid"], info["modes"]
        assert L == grid
        Kx = n[0] // 2
        fdt, cdt = (np.float64, np.complex128) if prec == 64 else (np.float32, np.complex64)
        u = np.finfo(fdt).eps / 2
        sigma = fields.random_sigma(T.shape[0] * 3, 5)
        iv = slp.slp_debug_host_array(plan, slp.SLP_HOST_PLANE_ROWS).reshape(L[2], 2)
        z0, nz = slp.slp_debug_host_array(plan, slp.SLP_HOST_ACTIVE_Z)
        zact = ((np.arange(L[2]) - z0) % L[2]) < nz
        ract = ((np.arange(L[1])[None, :] - iv[:, :1]) % L[1]) < iv[:, 1:]

        def stage(last, buf, dt, shape):
            run(slp, plan, slp.SLP_INPUT_SIGMA, sigma, prec, last)
            wide = np.complex128 if dt is cdt else np.float64
            return slp.slp_debug_copy(plan, buf, dt).astype(wide).reshape(shape)

        A = stage(slp.SLP_STAGE_SPREAD, slp.SLP_BUF_GRID_A, fdt, (L[2], L[1], L[0]))
        S1 = stage(slp.SLP_STAGE_FFT_X, slp.SLP_BUF_S1, cdt, (L[2], L[1], Kx))
        assert rel_l2(S1, ref.fft_x(A, Kx)) < 64 * u, "fft x"
        assert not np.any(slp.slp_debug_copy(plan, slp.SLP_BUF_GRID_A, fdt)), "grid A is left zero"
        S2 = stage(slp.SLP_STAGE_FFT_Y, slp.SLP_BUF_S2, cdt, (L[2], n[1], Kx))
        assert rel_l2(S2, ref.fft_y(S1, n[1])) < 64 * u, "fft y"
        S2b = stage(slp.SLP_STAGE_FFT_Z, slp.SLP_BUF_S2, cdt, (L[2], n[1], Kx))
        dtab = slp.slp_debug_copy(plan, slp.SLP_BUF_DTAB, fdt).astype(np.float64)
        assert rel_l2(S2b[zact], ref.fft_z_multiply(S2, dtab, n, L[2])[zact]) < 128 * u, "fft z"
        S1b = stage(slp.SLP_STAGE_IFFT_Y, slp.SLP_BUF_S1, cdt, (L[2], L[1], Kx))
        assert rel_l2(S1b[ract], ref.ifft_y(S2b, L[1])[ract]) < 64 * u, "ifft y"
        G = stage(slp.SLP_STAGE_IFFT_X, slp.SLP_BUF_GRID_B, fdt, (L[2], L[1], L[0]))
        assert rel_l2(G[ract], ref.ifft_x(S1b, L[0])[ract]) < 64 * u, "ifft x"
        assert not np.any(G[~ract])
    finally:
        slp.slp_destroy(plan)
