"""Every tile shape of the FP32 3D heat step, 64 and 128 cells wide, gives the same bits on
extents that no tile divides, periodic images included, and the oracle's step within 1e-5."""
import numpy as np
import pytest

import oracle
from gpu_util import assert_close
from paper_2406_08923_gb300 import _lib as L
from paper_2406_08923_gb300 import synth

pytestmark = pytest.mark.gpu


# one cell past and short of a tile, rows of one group, the least extent, images on both faces
# of one vector (nx = 2 r + 2 at r = 1, 2 r + 1 at r = 2)
@pytest.mark.parametrize("r,shape", [(1, (3, 3, 4)), (1, (9, 17, 129)), (2, (5, 5, 5)), (2, (11, 8, 66)), (3, (7, 7, 7)),
                                     (3, (20, 9, 65)), (3, (33, 12, 127)), (3, (18, 31, 192)), (4, (9, 10, 63)), (4, (13, 21, 130))])
def test_shapes_agree(cuda_lib, r, shape):
    nz, ny, nx = shape
    par = L.heat_params(shape)
    p = L.Plan(3, (nx, ny, nz), r, 1, L.STENCIL_BC_PERIODIC, L.STENCIL_DIFFUSION, L.STENCIL_F32, L.STENCIL_F32, params=par)
    f = synth.uniform(5, 1, nx * ny * nz, -1.0, 1.0).reshape(shape).astype(np.float32).astype(np.float64)
    ref = oracle.diffusion_r(f, r, par.dt, par.alpha, (par.dx[0], par.dx[1], par.dx[2]), 3)
    ox, oy, oz = p.origin
    first = None
    for v in range(p.variant()[1]):
        p.set_variant(v)
        a, b = p.alloc(), p.alloc()
        p.upload(a, [f])
        p.step(a, b, 3)
        p.sync()
        box = p.view3(b[0])[oz - r:oz + nz + r, oy - r:oy + ny + r, ox - r:ox + nx + r].cpu().numpy()
        if first is None:
            first = box
            assert_close(p.download(b)[0], ref, 1e-5, f"r {r} {shape}")
            np.testing.assert_array_equal(box, np.pad(box[r:-r, r:-r, r:-r], r, mode="wrap"))
        np.testing.assert_array_equal(box, first, err_msg=p.variant()[2])
