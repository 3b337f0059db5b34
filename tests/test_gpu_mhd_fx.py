"""The FP64 MHD substep with its differences in 64-bit fixed point (csrc/mhd_fx.cu): the right-hand
side is as close to the exact one as an FP64 evaluation is, also where a component is tiny beside
the others or a field is a small wave on a large mean; planes of different scales, fields of
zeros, infinities and scales at the ends of the range; the lengths of the z-chunks agree bit for
bit."""
import numpy as np
import pytest
import torch

from paper_2406_08923_gb300 import _lib as L

pytestmark = pytest.mark.gpu

W1 = (3 / 4, -3 / 20, 1 / 60)
W2 = (-49 / 18, 3 / 2, -3 / 20, 1 / 90)
WM = (270 / 720, -27 / 720, 2 / 720)


def _plan(shape, K=0.0):
    nz, ny, nx = shape
    par = L.mhd_params(shape)
    par.K = K
    par.dx[0], par.dx[1], par.dx[2] = 0.05, 0.06, 0.07
    par.dt = 1e-4
    p = L.Plan(3, (nx, ny, nz), 3, 8, L.STENCIL_BC_PERIODIC, L.STENCIL_MHD8, L.STENCIL_F64, L.STENCIL_F64, params=par)
    assert p.variant()[2].startswith("fx"), p.variant()
    return p, par


def _rhs(f8, par, t):
    """Eqs. A1-A4 in the type t, with the weights as FP64 has them."""
    f = f8.astype(t)
    h = [np.float64(x) for x in (par.dx[0], par.dx[1], par.dx[2])]

    def at(v, *moves):
        for a, s in moves:
            v = np.roll(v, -s, axis=2 - a)
        return v

    def d(v, a):
        return sum(t(np.float64(w) / h[a]) * (at(v, (a, k + 1)) - at(v, (a, -k - 1))) for k, w in enumerate(W1))

    def dd(v, a, b):
        if a == b:
            return t(W2[0] / (h[a] * h[a])) * v + sum(
                t(W2[k] / (h[a] * h[a])) * (at(v, (a, k)) + at(v, (a, -k))) for k in (1, 2, 3))
        return sum(t(np.float64(w) * 720 / (720.0 * h[a] * h[b])) *
                   ((at(v, (a, k + 1), (b, k + 1)) + at(v, (a, -k - 1), (b, -k - 1))) -
                    (at(v, (a, k + 1), (b, -k - 1)) + at(v, (a, -k - 1), (b, k + 1)))) for k, w in enumerate(WM))

    lr, u, av, s = f[0], f[1:4], f[4:7], f[7]
    glr, gs = [d(lr, a) for a in range(3)], [d(s, a) for a in range(3)]
    gu = [[d(u[c], a) for a in range(3)] for c in range(3)]
    div = gu[0][0] + gu[1][1] + gu[2][2]
    lap = lambda v: dd(v, 0, 0) + dd(v, 1, 1) + dd(v, 2, 2)
    gdiv = lambda w, a: dd(w[0], a, 0) + dd(w[1], a, 1) + dd(w[2], a, 2)
    b = [d(av[2], 1) - d(av[1], 2), d(av[0], 2) - d(av[2], 0), d(av[1], 0) - d(av[0], 1)]
    j = [(gdiv(av, a) - lap(av[a])) * t(1.0 / par.mu0) for a in range(3)]
    cross = lambda p, q: [p[1] * q[2] - p[2] * q[1], p[2] * q[0] - p[0] * q[2], p[0] * q[1] - p[1] * q[0]]
    S = [[t(0.5) * (gu[a][c] + gu[c][a]) - (div / t(3) if a == c else t(0)) for c in range(3)] for a in range(3)]
    rho = np.exp(lr)
    icp = t(1.0 / par.cp)
    cs2 = t(par.cs0 ** 2) * np.exp(t(par.gamma) * icp * s + t(par.gamma - 1.0) * (lr - t(par.lnrho0)))
    temp = cs2 / t(par.cp * (par.gamma - 1.0))
    dot = lambda p, q: p[0] * q[0] + p[1] * q[1] + p[2] * q[2]
    jb, ub = cross(j, b), cross(u, b)
    out = [-dot(u, glr) - div]
    for c in range(3):
        gd = gdiv(u, c)
        out.append(-dot(u, gu[c]) - cs2 * (gs[c] * icp + glr[c]) + jb[c] / rho +
                   t(par.nu) * (lap(u[c]) + gd / t(3) + t(2) * dot(S[c], glr)) + t(par.zeta) * gd)
    out += [ub[c] + t(par.eta) * lap(av[c]) for c in range(3)]
    s2 = sum(S[a][c] ** 2 for a in range(3) for c in range(3))
    heat = t(par.eta * par.mu0) * dot(j, j) + t(2 * par.nu) * rho * s2 + t(par.zeta) * rho * div * div
    out.append(-dot(u, gs) + heat / (rho * temp))
    if par.K:
        gcp, gm1 = t(par.gamma) * icp, t(par.gamma - 1.0)
        gphi = [gcp * gs[a] + gm1 * glr[a] for a in range(3)]
        out[7] = out[7] + t(par.K) / rho * (gcp * lap(s) + gm1 * lap(lr) + dot(gphi, gphi))
    return out


def _fields(kind, shape):
    rng = np.random.default_rng(11)
    z, y, x = np.meshgrid(*(np.arange(n) * (2 * np.pi / n) for n in shape), indexing="ij")
    f = np.stack([np.sin(x + 0.3 * q) * np.cos(y - q) + 0.5 * np.sin(z + y + q) for q in range(8)])
    if kind == "waves":
        return f
    if kind == "random":
        return rng.uniform(-1, 1, (8,) + shape)
    if kind == "means":  # small waves on large means
        return 1e-7 * f + np.array([1, 2, -1, 3, 0.5, 1, 2, -0.7])[:, None, None, None]
    if kind == "tiny":  # components far below their companions
        return f * np.array([1, 1, 1e-7, 1e-12, 1, 1e-9, 1e-4, 1e-3])[:, None, None, None]
    if kind == "planes":  # planes of all scales, and a field of zeros
        f = rng.uniform(0.5, 1, (8,) + shape) * np.exp2(-rng.integers(0, 40, (8, shape[0], 1, 1)))
        f[5] = 0.0
        return f
    if kind == "specks":  # cells far below the scale of their plane
        return f * np.exp2(-rng.integers(0, 60, (8,) + shape))
    if kind == "vortex":  # localised: most cells lie far below the scale of their tile
        d = [np.arange(n) - c for n, c in zip(shape, (3.2, 30.7, 60.4))]
        e = np.exp(-(d[0][:, None, None] ** 2 + d[1][:, None] ** 2 + d[2] ** 2) / 50.0)
        return np.stack([(1.0 - 0.2 * q + 0.05 * d[1][:, None] - 0.03 * q * d[2]) * e for q in range(8)])
    if kind == "shear":  # a perturbation of a layer in y, on a flow that changes sign there
        dy = (np.arange(shape[1]) - 29.5)[:, None]
        f = f * np.exp(-dy ** 2 / 32.0)
        f[1] = 0.3 * np.tanh(dy / 4.0) * np.ones(shape)
        return f
    raise ValueError(kind)


# The kernel's sums round less often than FP64 chains of multiply-adds, the rest is the same
# arithmetic: its rms error may be that of a NumPy FP64 evaluation, whose order of operations
# differs (the kernel that works in FP64 throughout reaches 1.03 of it on these fields, 1.28 where
# cells go to FP64), plus one rounding of the result.
@pytest.mark.parametrize("kind,K", [("waves", 0.0), ("random", 0.0), ("means", 0.0), ("tiny", 0.0), ("planes", 0.0),
                                    ("specks", 0.0), ("waves", 0.7), ("vortex", 0.0), ("vortex", 0.7), ("shear", 0.0)])
def test_rhs_as_accurate_as_fp64(cuda_lib, kind, K):
    shape = (7, 59, 115)
    f8 = _fields(kind, shape)
    p, par = _plan(shape, K)
    a = p.alloc()
    p.upload(a, f8)
    rhs = [torch.zeros(shape, dtype=torch.float64, device="cuda") for _ in range(8)]
    p.mhd_rhs(a, rhs)
    p.sync()
    exact, plain = _rhs(f8, par, np.longdouble), _rhs(f8, par, np.float64)
    for q in range(8):
        got = rhs[q].cpu().numpy()
        rms = lambda v: float(np.sqrt(np.mean(np.square(v))))
        err, ref = rms(got - exact[q]), rms(plain[q] - exact[q])
        print(kind, q, err, ref)
        assert err <= (1.3 if kind in ("planes", "specks", "vortex", "shear") else 1.05) * ref + 2.0 ** -53 * rms(exact[q]), (kind, q)


def _step(p, f8, steps):
    a, b = p.alloc(), p.alloc()
    p.upload(a, f8)
    p.step(a, b, steps)
    p.sync()
    return np.stack([np.asarray(v) for v in p.download(b)])


@pytest.mark.parametrize("kind", ("waves", "planes", "specks", "vortex"))
def test_slabs_of_z_are_bit_identical(cuda_lib, kind):
    # the same planes in a deeper periodic field start other z-chunks
    shape = (24, 50, 130)
    f8 = 1e-3 * _fields(kind, shape)
    p, _ = _plan(shape)
    deep, _ = _plan((48,) + shape[1:])
    got = _step(p, f8, 2)
    twice = _step(deep, np.concatenate([f8, f8], axis=1), 2)
    assert np.array_equal(twice[:, :24], got) and np.array_equal(twice[:, 24:], got)


@pytest.mark.parametrize("K", (0.0, 0.7))
def test_variants_and_chunk_lengths_are_bit_identical(cuda_lib, K):
    shape = (40, 50, 130)  # ragged tiles; chunks of 5 to 40 planes
    f8 = 1e-3 * _fields("waves", shape)
    p, _ = _plan(shape, K)
    ref = _step(p, f8, 2)
    for v in range(p.variant()[1]):
        for zmode in range(3):
            p.set_variant(v)
            p.set_zmode(zmode)
            assert np.array_equal(_step(p, f8, 2), ref), (v, zmode)


def test_more_listed_cells_than_the_list_holds(cuda_lib):
    # s at the end of the exponent range: the two columns of the last tiles list every cell, 16 per
    # plane, in chunks of up to 128 planes (tiles for two per SM); elsewhere whole warps take the field in FP64
    shape = (132, 272, 130)
    f8 = 1e-3 * _fields("waves", shape)
    f8[7] *= 1e-305
    p, _ = _plan(shape)
    ref = _step(p, f8, 1)
    for zmode in (1, 2):
        p.set_zmode(zmode)
        assert np.array_equal(_step(p, f8, 1), ref), zmode


@pytest.mark.parametrize("value", (np.inf, np.nan, 1e300, 1e-310))
def test_extreme_values_go_to_fp64(cuda_lib, value):
    # an extreme value of s: its gradient reaches the cells within 3 along the axes alone
    shape = (12, 50, 130)
    f8 = 1e-3 * _fields("waves", shape)
    if value < 1:
        f8[7] = value * np.sign(f8[7])
    else:
        f8[7, 6, 5, 9] = value
    p, par = _plan(shape)
    a = p.alloc()
    p.upload(a, f8)
    rhs = [torch.zeros(shape, dtype=torch.float64, device="cuda") for _ in range(8)]
    p.mhd_rhs(a, rhs)
    p.sync()
    with np.errstate(all="ignore"):
        plain = _rhs(f8, par, np.float64)
    for q in range(8):
        got = rhs[q].cpu().numpy()
        finite = np.isfinite(plain[q])
        assert np.array_equal(finite, np.isfinite(got)), q
        assert np.array_equal(np.isnan(plain[q]), np.isnan(got)), q
        scale = np.abs(np.where(finite & (np.abs(plain[q]) < 1e200), plain[q], 0)).max()
        err = np.abs(np.where(finite, got, 0) - np.where(finite, plain[q], 0))
        assert np.all(err <= 1e-13 * np.maximum(np.where(finite, np.abs(plain[q]), 0), scale)), q
