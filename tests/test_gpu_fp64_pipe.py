"""The FP64-pipe kernels that serve plans whose weights do not fit fixed point (csrc/diffusion.cu,
csrc/xcorr.cu, csrc/xcorr_wide.cu): heat steps of a negative dt, correlations of weights outside the
exponent range, against the oracle, with the periodic images and as z-slabs."""
import numpy as np
import pytest
import torch

import oracle
from gpu_util import assert_close
from paper_2406_08923_gb300 import _lib as L
from paper_2406_08923_gb300 import synth

pytestmark = pytest.mark.gpu


# one tile and several, extents no tile divides, the least extent
@pytest.mark.parametrize("r,shape", [(1, (3, 3, 3)), (1, (9, 17, 129)), (2, (5, 8, 66)), (3, (7, 7, 7)), (3, (20, 33, 65)),
                                     (4, (9, 9, 9)), (4, (13, 21, 130))])
def test_heat_backward_steps(cuda_lib, r, shape):
    nz, ny, nx = shape
    par = L.heat_params(shape)
    par.dt = -0.02 * min(par.dx[0], par.dx[1], par.dx[2]) ** 2
    p = L.Plan(3, (nx, ny, nz), r, 1, L.STENCIL_BC_PERIODIC, L.STENCIL_DIFFUSION, L.STENCIL_F64, L.STENCIL_F64, params=par)
    assert "vx2" in p.variant()[2]
    f = synth.uniform(5, 1, nx * ny * nz, -1.0, 1.0).reshape(shape)
    a, b = p.alloc(), p.alloc()
    p.upload(a, [f])
    p.step(a, b, 3)
    p.sync()
    assert_close(p.download(b)[0], oracle.diffusion_r(f, r, par.dt, par.alpha, tuple(par.dx), 3), 1e-12, f"r {r} {shape}")
    ox, oy, oz = p.origin
    box = p.view3(b[0])[oz - r:oz + nz + r, oy - r:oy + ny + r, ox - r:ox + nx + r].cpu().numpy()
    np.testing.assert_array_equal(box, np.pad(box[r:-r, r:-r, r:-r], r, mode="wrap"))


def test_heat_backward_slabs_equal_the_whole(cuda_lib):
    shape, r = (22, 19, 70), 3
    par = L.heat_params(shape)
    par.dt = -0.02 * min(par.dx[0], par.dx[1], par.dx[2]) ** 2
    f = synth.uniform(6, 1, int(np.prod(shape)), -1.0, 1.0).reshape(shape)
    p = L.Plan(3, shape[::-1], r, 1, L.STENCIL_BC_PERIODIC, L.STENCIL_DIFFUSION, L.STENCIL_F64, L.STENCIL_F64, params=par)
    a, b = p.alloc(), p.alloc()
    p.upload(a, [f])
    p.step(a, b, 1)
    p.sync()
    whole = p.download(b)[0]
    for z0, z1 in ((0, 8), (8, 13), (13, 22)):
        q = L.Plan(3, (shape[2], shape[1], z1 - z0), r, 1, L.STENCIL_BC_PERIODIC_XY, L.STENCIL_DIFFUSION, L.STENCIL_F64,
                   L.STENCIL_F64, params=par)
        c, d = q.alloc(), q.alloc()
        ox, oy, oz = q.origin
        q.view3(c[0])[oz - r:oz + z1 - z0 + r, oy:oy + shape[1], ox:ox + shape[2]] = torch.from_numpy(
            f[np.arange(z0 - r, z1 + r) % shape[0]]).cuda()
        q.step(c, d, 1)
        q.sync()
        np.testing.assert_array_equal(q.download(d)[0], whole[z0:z1])


@pytest.mark.parametrize("scale", [2.0 ** -120, 2.0 ** 120])
@pytest.mark.parametrize("r,n,sweeps", [(1, 3, 2), (1, 70001, 3), (2, 4099, 8), (3, 2305, 7), (4, 9001, 2), (5, 3001, 1),
                                        (22, 4999, 2), (100, 20001, 1), (1024, 5000, 1)])
def test_correlation_of_weights_out_of_range(cuda_lib, r, n, sweeps, scale):
    w = synth.uniform(7, 100 + r, 2 * r + 1, -1.0, 1.0)
    w = w / np.abs(w).sum()
    f = synth.uniform(7, r, n, -1.0, 1.0)
    p = L.Plan(1, (n,), r, 1, L.STENCIL_BC_PERIODIC, L.STENCIL_XCORR, L.STENCIL_F64, L.STENCIL_F64, coeffs=w * scale)
    assert p.variant()[2] in ("wide_register_blocked", "runtime_chunk_scalar_temporal_blocking")
    a, b = p.alloc(), p.alloc()
    p.upload(a, [f])
    p.step(a, b, sweeps)
    p.sync()
    got = p.download(b)[0] / scale ** sweeps  # powers of two: exact
    assert_close(got, oracle.xcorr1d(f, w, sweeps), 1e-12, f"r {r}")
    whole, o = p.view3(b[0])[0, 0].cpu().numpy(), p.origin[0]
    np.testing.assert_array_equal(whole[o - r:o + n + r], np.pad(whole[o:o + n], r, mode="wrap"))


@pytest.mark.parametrize("r,n", [(1, 5000), (3, 2304), (4, 301), (9, 5000), (64, 20001)])
def test_correlation_of_weights_out_of_range_with_the_callers_halo(cuda_lib, r, n):
    scale = 2.0 ** 120
    w = synth.uniform(8, r, 2 * r + 1, -1.0, 1.0)
    f = synth.uniform(8, 50 + r, n + 2 * r, -1.0, 1.0)
    p = L.Plan(1, (n,), r, 1, L.STENCIL_BC_CALLER, L.STENCIL_XCORR, L.STENCIL_F64, L.STENCIL_F64, coeffs=w * scale)
    a, b = p.alloc(), p.alloc()
    o = p.origin[0]
    p.view3(a[0])[0, 0, o - r:o + n + r] = torch.from_numpy(f).cuda()
    p.step(a, b, 1)
    p.sync()
    ref = sum(w[j] * f[j:j + n] for j in range(2 * r + 1))
    assert_close(p.download(b)[0] / scale, ref, 1e-12, f"r {r}")
