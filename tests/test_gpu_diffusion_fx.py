"""The FP64 3D heat step in 64-bit fixed point (csrc/diffusion_fx.cu, csrc/fixed.cuh): every output,
also where a field spans hundreds of binary orders, is as close to the exact step as a chain of
FP64 multiply-adds is, infinities and NaN spread as they do in FP64, and the launch shapes agree
bit for bit."""
import numpy as np
import pytest
import torch

from paper_2406_08923_gb300 import _lib as L

pytestmark = pytest.mark.gpu

C = {1: (-2.0, 1.0), 2: (-5 / 2, 4 / 3, -1 / 12), 3: (-49 / 18, 3 / 2, -3 / 20, 1 / 90),
     4: (-205 / 72, 8 / 5, -1 / 5, 8 / 315, -1 / 560)}


def _plan(shape, r, h, dt=0.02):
    par = L.heat_params(shape)
    par.dx[0], par.dx[1], par.dx[2] = h
    par.dt, par.alpha = dt, 1.0
    return L.Plan(3, shape[::-1], r, 1, L.STENCIL_BC_PERIODIC, L.STENCIL_DIFFUSION, L.STENCIL_F64, L.STENCIL_F64,
                  params=par)


def _step(p, f, variant=0):
    p.set_variant(variant)
    a, b = p.alloc(), p.alloc()
    p.upload(a, [f])
    p.step(a, b, 1)
    p.sync()
    return p.download(b)[0], b[0].cpu().numpy()


def _reference(f, r, h, dt=0.02):
    """The folded step and sum |w| |f| per cell, in extended precision."""
    q = f.astype(np.longdouble)
    g0 = np.longdouble(1.0 + sum(dt * C[r][0] / (x * x) for x in h))
    out, mag = g0 * q, abs(g0) * abs(q)
    for a in range(3):
        for k in range(1, r + 1):
            w = np.longdouble(dt * C[r][k] / (h[a] * h[a]))
            s, t = np.roll(q, k, 2 - a), np.roll(q, -k, 2 - a)
            out = out + w * (s + t)
            mag = mag + abs(w) * (abs(s) + abs(t))
    return out, mag


def _fields(shape, seed):
    rng = np.random.default_rng(seed)
    z, y, x = np.meshgrid(*[np.arange(n) for n in shape], indexing="ij")
    smooth = np.sin(0.3 * x + 0.2 * y + 0.25 * z)
    yield "random", rng.standard_normal(shape)
    yield "smooth", smooth
    yield "decay", np.exp(-2.0 * (x + y + z)) * (1 + 0.1 * rng.standard_normal(shape))
    yield "orders", rng.standard_normal(shape) * 2.0 ** rng.integers(-300, 300, shape)
    yield "blocks", np.where((x // 5 + y // 4 + z // 3) % 2, 0.0, smooth * 1e-30)
    yield "edges of the range", smooth * 2.0 ** np.where(z % 7 < 3, -1015.0, 900.0)


@pytest.mark.parametrize("r,h", [(1, (0.5, 0.5, 0.5)), (2, (0.4, 0.5, 0.6)), (3, (0.5, 0.5, 0.5)), (3, (0.5, 0.4, 0.7)),
                                 (4, (0.5, 0.5, 0.5)), (4, (0.45, 0.5, 0.6))])
@pytest.mark.parametrize("shape", [(9, 17, 65), (21, 33, 130), (40, 16, 64)])
def test_every_output_is_as_close_as_fp64(cuda_lib, r, h, shape):
    p = _plan(shape, r, h)
    for name, f in _fields(shape, 5):
        got, _ = _step(p, f)
        ref, mag = _reference(f, r, h)
        # the weights' own roundings and one rounding per multiply-add of the 1 + 6 r terms
        bound = (1 + 6 * r + 2) * 2.0 ** -53 * mag + 2.0 ** -1074
        worst = float(np.max(np.abs(got - ref) / bound))
        assert worst <= 1.0, (name, worst)


def _cold_fields(shape):
    z, y, x = np.meshgrid(*[np.arange(n) for n in shape], indexing="ij")
    hot = np.zeros(shape)
    hot[4, 6, 20], hot[-3, -1, -2], hot[7, 9, 40:44] = 1.0, -0.7, 1.3
    yield "hot cells in a cold field", hot
    yield "hot cells in a faint field", hot + 1e-9 * np.sin(0.7 * x + 0.4 * y + 0.9 * z)
    yield "hot spot", np.exp(-((x - 30.3) ** 2 + (y - 8.1) ** 2 + (z - 9.2) ** 2) / 18.0)
    yield "front", np.where(x < 33, 1.0 + 0.1 * np.sin(0.5 * y), 1e-12 * np.cos(0.3 * z + y))
    yield "large mean", 1.0 + 1e-8 * np.sin(0.3 * x + 0.2 * y + 0.25 * z)


# small steps, and axes whose weights are far below the others': terms of small weight times a
# large value, or of a large weight times a small value, carry the output
@pytest.mark.parametrize("r,h", [(1, (0.5, 0.5, 0.5)), (2, (0.4, 0.5, 0.6)), (3, (0.5, 0.5, 0.5)), (3, (50.0, 0.5, 0.5)),
                                 (3, (0.5, 0.5, 50.0)), (4, (0.5, 0.5, 0.5)), (4, (0.5, 60.0, 0.45))])
@pytest.mark.parametrize("dt", [0.02, 1e-3, 1e-4, 1e-6, 1e-9])
def test_every_output_is_as_close_as_fp64_at_small_steps(cuda_lib, r, h, dt):
    shape = (21, 18, 70)
    p = _plan(shape, r, h, dt)
    for name, f in list(_cold_fields(shape)) + list(_fields(shape, 6)):
        got, _ = _step(p, f)
        ref, mag = _reference(f, r, h, dt)
        bound = (1 + 6 * r + 2) * 2.0 ** -53 * mag + 2.0 ** -1074  # as above
        worst = float(np.max(np.abs(got - ref) / bound))
        assert worst <= 1.0, (name, worst)


def test_infinities_and_nan_spread_as_in_fp64(cuda_lib):
    shape, r, h = (20, 20, 70), 3, (0.5, 0.5, 0.5)
    f = np.random.default_rng(3).standard_normal(shape)
    f[4, 5, 6], f[15, 3, 66], f[10, 12, 30] = np.inf, -np.inf, np.nan
    p = _plan(shape, r, h)
    got, _ = _step(p, f)
    ref, mag = _reference(f, r, h)
    fine = np.isfinite(ref)
    assert np.array_equal(np.isnan(got), np.isnan(ref)) and np.array_equal(np.isfinite(got), fine)
    inf = np.isinf(ref.astype(np.float64))
    assert np.array_equal(got[inf], ref[inf].astype(np.float64))
    assert np.all(np.abs(got - ref)[fine] <= 21 * 2.0 ** -53 * mag[fine])


@pytest.mark.parametrize("shape", [(7, 7, 7), (37, 40, 66), (50, 33, 131)])
def test_launch_shapes_agree_bit_for_bit(cuda_lib, shape):
    p = _plan(shape, 3, (0.5, 0.5, 0.5))
    f = np.random.default_rng(7).standard_normal(shape) * 2.0 ** np.random.default_rng(8).integers(-6, 3, (shape[0], 1, 1))
    first = _step(p, f)[0]
    for v in range(1, p.variant()[1]):
        assert np.array_equal(_step(p, f, v)[0], first), v


# fields whose rows are evaluated in FP64 as a whole, or list up to 16 outputs each, thousands per
# block of threads (the columns of small values), in every launch shape
@pytest.mark.parametrize("r", [1, 3, 4])
@pytest.mark.parametrize("kind", ["columns", "spot"])
def test_localised_fields(cuda_lib, r, kind):
    shape, h = (33, 200, 500), (0.5, 0.5, 0.5)
    z, y, x = np.meshgrid(*[np.arange(n) for n in shape], indexing="ij")
    rng = np.random.default_rng(4)
    f = (np.where((x // 8 + y // 8) % 2, 1e-12, 1.0) * rng.uniform(0.5, 1.0, shape) if kind == "columns" else
         np.exp(-((x - 250.3) ** 2 + (y - 99.5) ** 2 + (z - 15.7) ** 2) / 288.0))
    p = _plan(shape, r, h)
    ref, mag = _reference(f, r, h)
    ox, oy, oz = p.origin
    first = None
    for v in range(p.variant()[1]):
        p.set_variant(v)
        a, b = p.alloc(), p.alloc()
        p.upload(a, [f])
        p.step(a, b, 1)
        p.sync()
        box = p.view3(b[0])[oz - r:oz + 33 + r, oy - r:oy + 200 + r, ox - r:ox + 500 + r].cpu().numpy()
        if first is None:
            first, got = box, box[r:-r, r:-r, r:-r]
            bound = (1 + 6 * r + 2) * 2.0 ** -53 * mag + 2.0 ** -1074
            assert float(np.max(np.abs(got - ref) / bound)) <= 1.0
            assert np.array_equal(box, np.pad(got, r, mode="wrap"))
        assert np.array_equal(box, first), v


def test_weights_of_a_backward_step_run_on_the_fp64_pipe(cuda_lib):
    shape, r, h = (12, 18, 40), 3, (0.5, 0.5, 0.5)  # dt < 0: the signs the fixed-point kernel has not compiled in
    p = _plan(shape, r, h, dt=-0.01)
    assert p.variant()[2].startswith("vx2") and _plan(shape, r, h).variant()[2].startswith("fx64")
    f = np.random.default_rng(9).standard_normal(shape)
    ref, mag = _reference(f, r, h, dt=-0.01)
    assert np.all(np.abs(_step(p, f)[0] - ref) <= 21 * 2.0 ** -53 * mag)
