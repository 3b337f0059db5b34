"""The FP64 cross-correlation in fixed point and the sweeps composed into one launch
(csrc/xcorr_fx.cu): every output, also where the data span hundreds of binary orders or cancel, is
as close to the exact sum as a chain of FP64 multiply-adds is, and infinities and NaN spread as
they do in FP64."""
import numpy as np
import pytest
import torch

from paper_2406_08923_gb300 import _lib as L

pytestmark = pytest.mark.gpu


def _run(data, g, bc=L.STENCIL_BC_PERIODIC, halo=None, sweeps=1):
    n, r = data.size, g.size // 2
    p = L.Plan(1, (n,), r, 1, bc, L.STENCIL_XCORR, L.STENCIL_F64, L.STENCIL_F64, coeffs=g)
    a, b = p.alloc(), p.alloc()
    p.upload(a, [data])
    if halo is not None:
        o = p.origin[0]
        v = p.view3(a[0])[0, 0]
        v[o - r:o], v[o + n:o + n + r] = torch.from_numpy(halo[0]).cuda(), torch.from_numpy(halo[1]).cuda()
    p.step(a, b, sweeps)
    p.sync()
    whole = p.view3(b[0])[0, 0].cpu().numpy()
    o = p.origin[0]
    return whole[o:o + n], (whole[o - r:o], whole[o + n:o + n + r])


def _reference(fhat, g):
    """sum_j g_j f_{i+j} and sum_j |g_j f_{i+j}| of the augmented array, in extended precision."""
    q, w = fhat.astype(np.longdouble), g.astype(np.longdouble)
    n = q.size - g.size + 1
    out, mag = np.zeros(n, np.longdouble), np.zeros(n, np.longdouble)
    for j in range(g.size):
        t = w[j] * q[j:j + n]
        out += t
        mag += np.abs(t)
    return out, mag


def _data(n, seed):
    rng = np.random.default_rng(seed)
    i = np.arange(n)
    yield "random", rng.standard_normal(n)
    yield "positive", rng.random(n)
    yield "decay", np.exp(-i / 3.0)
    yield "orders", rng.standard_normal(n) * 2.0 ** rng.integers(-200, 200, n)
    yield "cancel", np.where(i % 2, 1.0, -1.0) + 1e-13 * rng.standard_normal(n)
    yield "spikes", np.where(i % 97 == 5, 1e200, rng.standard_normal(n) * 1e-100) * (i % 1000 < 700)
    yield "tiny", rng.standard_normal(n) * 2.0 ** -1030


def _weights(r, kind):
    rng = np.random.default_rng(1000 + r)
    j = np.arange(-r, r + 1)
    return {"average": lambda: np.full(2 * r + 1, 1.0 / (2 * r + 1)), "signed": lambda: rng.uniform(-1.0, 1.0, 2 * r + 1),
            "gauss": lambda: np.exp(-12.0 * (j / r) ** 2), "orders": lambda: rng.standard_normal(2 * r + 1) *
            2.0 ** rng.integers(-70, 5, 2 * r + 1)}[kind]()


# radii around whole register blocks of 3, 7 and 9 weights, and the ends of the range
@pytest.mark.parametrize("r,n", [(5, 11), (5, 3001), (6, 2305), (7, 2304), (8, 1793), (13, 5001), (22, 4999), (100, 4096),
                                 (333, 2777), (1024, 2049), (1024, 7001),
                                 (10, 400001), (40, 300001)])
@pytest.mark.parametrize("kind", ["average", "signed", "gauss", "orders"])
def test_every_output_is_as_close_as_fp64(cuda_lib, r, n, kind):
    g = _weights(r, kind)
    for name, f in _data(n, r):
        got, (lo, hi) = _run(f, g)
        ref, mag = _reference(np.pad(f, r, mode="wrap"), g)
        bound = (2 * r + 1) * 2.0 ** -53 * mag + (2 * r + 1) * 2.0 ** -1074  # one rounding per multiply-add
        worst = float(np.max(np.abs(got - ref) / bound))
        assert worst <= 1.0, (name, worst)
        assert np.array_equal(lo, got[-r:]) and np.array_equal(hi, got[:r])


def test_caller_halo_and_special_values(cuda_lib):
    r, n = 9, 5000
    rng = np.random.default_rng(4)
    g = rng.uniform(-1.0, 1.0, 2 * r + 1)
    f, halo = rng.standard_normal(n), (rng.standard_normal(r) * 1e3, rng.standard_normal(r) * 1e-3)
    got, _ = _run(f, g, L.STENCIL_BC_CALLER, halo)
    ref, mag = _reference(np.concatenate([halo[0], f, halo[1]]), g)
    assert np.all(np.abs(got - ref) <= (2 * r + 1) * 2.0 ** -53 * mag)
    f[100], f[3000], f[4990] = np.inf, np.nan, -np.inf
    got, _ = _run(f, g)
    with np.errstate(invalid="ignore"):
        ref, mag = _reference(np.pad(f, r, mode="wrap"), g)
        fine = np.isfinite(ref)
        assert np.array_equal(np.isnan(got), np.isnan(ref)) and np.array_equal(np.isfinite(got), fine)
        assert np.all(np.abs(got - ref)[fine] <= (2 * r + 1) * 2.0 ** -53 * mag[fine])


def _pulses(n, r):
    rng = np.random.default_rng(r)
    i = np.arange(n)
    yield "spikes on zeros", np.where(i % 997 == 5, 1.0 + rng.random(n), 0.0)
    yield "a spike and zeros", np.where(i == n // 2, -3.0, 0.0)
    yield "pulses", np.exp(-((i % 4096) - 2048.0) ** 2 / 2e4)
    yield "many orders", rng.standard_normal(n) * 2.0 ** -rng.integers(0, 60, n)
    yield "faint half", np.where((i // 300) % 2, 1.0, 1e-30) * rng.random(n)
    yield "signed zeros", np.where(i % 2, 0.0, -0.0)


# chunks of which most outputs lie far below the scale, windows and chunks of zeros; radii of each block size
@pytest.mark.parametrize("r,n,sweeps", [(5, 9001, 1), (13, 5001, 1), (100, 30011, 1), (1000, 20001, 1), (1, 20011, 16),
                                        (3, 20011, 10), (4, 7001, 3)])
@pytest.mark.parametrize("kind", ["average", "gauss", "orders"])
def test_pulses_and_zeros(cuda_lib, r, n, sweeps, kind):
    g = _weights(r, kind)
    for name, f in _pulses(n, r):
        got, (lo, hi) = _run(f, g, sweeps=sweeps)
        ref, mag = f.astype(np.longdouble), np.abs(f).astype(np.longdouble)
        for _ in range(sweeps):
            ref, mag = _reference(np.pad(ref, r, mode="wrap"), g)[0], _reference(np.pad(mag, r, mode="wrap"), np.abs(g))[0]
        tiny = sweeps * (2 * r + 1) * max(1.0, float(np.abs(g).sum())) ** sweeps * 2.0 ** -1074
        worst = float(np.max(np.abs(got - ref) / (sweeps * (2 * r + 1) * 2.0 ** -53 * mag + tiny)))
        assert worst <= 1.0, (name, worst)
        assert np.all(got[mag == 0] == 0) and np.array_equal(lo, got[-r:]) and np.array_equal(hi, got[:r]), name


# one launch, one launch and a remainder, and radii that fill register blocks or not; n below the
# composed halo wraps more than once
@pytest.mark.parametrize("r,n,sweeps", [(1, 3, 1), (1, 2305, 16), (2, 5, 16), (2, 4000, 7), (3, 4099, 10), (3, 2304, 17),
                                        (4, 9, 16), (4, 1793, 5)])
@pytest.mark.parametrize("kind", ["average", "signed", "orders"])
def test_composed_sweeps_are_as_close_as_fp64(cuda_lib, r, n, sweeps, kind):
    g = _weights(r, kind)
    for name, f in _data(n, 50 + r):
        got, (lo, hi) = _run(f, g, sweeps=sweeps)
        ref, mag = f.astype(np.longdouble), np.abs(f).astype(np.longdouble)
        for _ in range(sweeps):
            ref, mag = _reference(np.pad(ref, r, mode="wrap"), g)[0], _reference(np.pad(mag, r, mode="wrap"), np.abs(g))[0]
        # one rounding per multiply-add of every sweep, each worth a denormal at least
        tiny = sweeps * (2 * r + 1) * max(1.0, float(np.abs(g).sum())) ** sweeps * 2.0 ** -1074
        worst = float(np.max(np.abs(got - ref) / (sweeps * (2 * r + 1) * 2.0 ** -53 * mag + tiny)))
        assert worst <= 1.0, (name, worst)
        assert np.array_equal(lo, got[-r:]) and np.array_equal(hi, got[:r])


def test_composed_sweeps_spread_special_values_as_sweeps_do(cuda_lib):
    r, n, sweeps = 3, 9001, 6
    g = np.array([0.1, -0.2, 0.0, 0.5, 0.3, -0.1, 0.2])
    f = np.random.default_rng(6).standard_normal(n)
    f[100], f[3000], f[n - 2] = np.inf, np.nan, -np.inf
    got, _ = _run(f, g, sweeps=sweeps)
    ref = f.copy()
    with np.errstate(invalid="ignore"):
        for _ in range(sweeps):
            q = np.pad(ref, r, mode="wrap")
            ref = sum(g[j] * q[j:j + n] for j in range(7))
    assert np.array_equal(np.isnan(got), np.isnan(ref)) and np.array_equal(np.isinf(got), np.isinf(ref))
    fine = np.isfinite(ref)
    np.testing.assert_allclose(got[fine], ref[fine], rtol=0, atol=1e-14)


@pytest.mark.parametrize("r,n,sweeps", [(1, 3, 16), (2, 2305, 2), (3, 4099, 10), (3, 7, 33), (4, 9, 16), (4, 2304, 17),
                                        (4, 70001, 16)])
def test_composed_int32_sweeps_are_exact(cuda_lib, r, n, sweeps):
    rng = np.random.default_rng(r + n)
    f = rng.integers(-2 ** 31, 2 ** 31, n).astype(np.int32)
    g = rng.integers(-2 ** 31, 2 ** 31, 2 * r + 1).astype(np.int32)
    p = L.Plan(1, (n,), r, 1, L.STENCIL_BC_PERIODIC, L.STENCIL_XCORR, L.STENCIL_I32, L.STENCIL_I32, coeffs=g)
    a, b = p.alloc(), p.alloc()
    p.upload(a, [f])
    p.step(a, b, sweeps)
    p.sync()
    ref = f.astype(np.uint32)
    for _ in range(sweeps):
        q = np.pad(ref, r, mode="wrap")
        ref = sum(g.astype(np.uint32)[j] * q[j:j + n] for j in range(2 * r + 1))
    whole = p.view3(b[0])[0, 0].cpu().numpy().astype(np.uint32)
    o = p.origin[0]
    assert np.array_equal(whole[o - r:o + n + r], np.pad(ref, r, mode="wrap"))


# weights whose sum is far from 1 leave the range of fixed point after some sweeps (11, 16 and 15 at
# r = 3): fewer sweeps still compose, and calls of more take several launches
@pytest.mark.parametrize("total", [1000.0, 100.0, 0.01])
@pytest.mark.parametrize("r,sweeps", [(3, 1), (3, 10), (3, 16), (3, 25), (4, 16)])
def test_weights_that_compose_for_some_sweeps(cuda_lib, total, r, sweeps):
    n, g = 4099, np.full(2 * r + 1, total / (2 * r + 1))
    p = L.Plan(1, (n,), r, 1, L.STENCIL_BC_PERIODIC, L.STENCIL_XCORR, L.STENCIL_F64, L.STENCIL_F64, coeffs=g)
    assert p.variant()[2] == "composed_fixed_point"
    f = np.random.default_rng(8).standard_normal(n)
    got, (lo, hi) = _run(f, g, sweeps=sweeps)
    ref, mag = f.astype(np.longdouble), np.abs(f).astype(np.longdouble)
    for _ in range(sweeps):
        ref, mag = _reference(np.pad(ref, r, mode="wrap"), g)[0], _reference(np.pad(mag, r, mode="wrap"), np.abs(g))[0]
    assert float(np.max(np.abs(got - ref) / (sweeps * (2 * r + 1) * 2.0 ** -53 * mag))) <= 1.0
    assert np.array_equal(lo, got[-r:]) and np.array_equal(hi, got[:r])


@pytest.mark.parametrize("r,storage,g,bc,name", [
    (3, L.STENCIL_F64, [0.1] * 7, L.STENCIL_BC_PERIODIC, "composed_fixed_point"),
    (1, L.STENCIL_F64, [0.3] * 3, L.STENCIL_BC_PERIODIC, "composed_fixed_point"),
    (3, L.STENCIL_F64, [0.1] * 7, L.STENCIL_BC_CALLER, "composed_fixed_point"),
    (1, L.STENCIL_F64, [0.3] * 3, L.STENCIL_BC_CALLER, "runtime_chunk_scalar_temporal_blocking"),
    (3, L.STENCIL_F64, [2.0 ** -120] * 7, L.STENCIL_BC_PERIODIC, "runtime_chunk_scalar_temporal_blocking"),
    (3, L.STENCIL_F64, [np.nan] * 7, L.STENCIL_BC_PERIODIC, "runtime_chunk_scalar_temporal_blocking"),
    (2, L.STENCIL_I32, [1, -2, 3, 1, 1], L.STENCIL_BC_PERIODIC, "composed_v9"),
    (2, L.STENCIL_I32, [1, -2, 3, 1, 1], L.STENCIL_BC_CALLER, "chunk2184_v9_temporal_blocking"),
    (3, L.STENCIL_F32, [0.1] * 7, L.STENCIL_BC_PERIODIC, "chunk2184_v9_temporal_blocking")])
def test_variant_name_tells_the_kernel(cuda_lib, r, storage, g, bc, name):
    g = np.array(g, dtype=np.int32 if storage == L.STENCIL_I32 else np.float64)
    assert L.Plan(1, (5000,), r, 1, bc, L.STENCIL_XCORR, storage, storage, coeffs=g).variant()[2] == name
