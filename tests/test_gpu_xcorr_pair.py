"""The packed FP32 cross-correlation of radius 33..1024 (csrc/xcorr_pair.cu): bit-identical to one
fused multiply-add per weight in ascending order, which the caller-halo path (csrc/xcorr_wide.cu)
computes, at sizes around half chunks, chunks and whole register blocks."""
import numpy as np
import pytest
import torch

from paper_2406_08923_gb300 import _lib as L

pytestmark = pytest.mark.gpu


def _plan(n, r, g, bc):
    return L.Plan(1, (n,), r, 1, bc, L.STENCIL_XCORR, L.STENCIL_F32, L.STENCIL_F32, coeffs=g)


# n and r that pick V = 3, 5, 7, 9, 13; n of one half chunk, a chunk and one cell more; wrapped halos
@pytest.mark.parametrize("r,n", [(33, 67), (33, 768), (33, 1537), (64, 65536), (500, 300001), (64, 1 << 20), (1024, 1 << 21),
                                 (100, 3000001), (1024, 2049), (49, 4608), (65, 3000003)])
def test_periodic_equals_the_caller_halo_path(cuda_lib, r, n):
    rng = np.random.default_rng(r + n)
    g = rng.uniform(-1.0, 1.0, 2 * r + 1)
    f = rng.standard_normal(n).astype(np.float32)
    p, q = _plan(n, r, g, L.STENCIL_BC_PERIODIC), _plan(n, r, g, L.STENCIL_BC_CALLER)
    o = p.origin[0]
    a, b = p.alloc(), p.alloc()
    p.upload(a, [f])
    p.step(a, b, 1)
    p.sync()
    c, d = q.alloc(), q.alloc()
    q.view3(c[0])[0, 0, o - r:o + n + r] = torch.from_numpy(np.pad(f, r, mode="wrap")).cuda()
    q.step(c, d, 1)
    q.sync()
    got = p.view3(b[0])[0, 0, o - r:o + n + r].cpu().numpy()
    np.testing.assert_array_equal(got, np.pad(q.interior(d[0]).cpu().numpy(), r, mode="wrap"))


# radii whose 2 r + 1 weights fill whole blocks of V, or all but one to V - 1 of the last; both paths
@pytest.mark.parametrize("r,n", [(33, 1537), (37, 65536), (52, 3000000), (52, 70001), (64, 1 << 20), (100, 300001),
                                 (100, 3000001), (250, 20011)])
@pytest.mark.parametrize("bc", [L.STENCIL_BC_PERIODIC, L.STENCIL_BC_CALLER])
def test_special_values_reach_the_outputs_that_read_them(cuda_lib, r, n, bc):
    rng = np.random.default_rng(r)
    g = rng.uniform(0.5, 1.0, 2 * r + 1)
    f = rng.standard_normal(n).astype(np.float32)
    p = _plan(n, r, g, bc)
    o = p.origin[0]

    def run(v):
        a, b = p.alloc(), p.alloc()
        p.view3(a[0])[0, 0, o - r:o + n + r] = torch.from_numpy(np.pad(v, r, mode="wrap")).cuda()
        p.step(a, b, 1)
        p.sync()
        return p.interior(b[0]).cpu().numpy()

    plain = run(f)
    for at, value in ((5, np.nan), (n // 3, np.inf), (n // 2 + 1, -np.inf), (n - 3, np.nan)):
        v = f.copy()
        v[at] = value
        got = run(v)
        reads = np.zeros(n, bool)
        reads[(np.arange(-r, r + 1) + at) % n] = True
        assert not np.isfinite(got[reads]).any(), (at, value)
        np.testing.assert_array_equal(got[~reads], plain[~reads], err_msg=f"{at} {value}")
