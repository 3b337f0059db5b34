"""Performance cases of the stencil engine: what its users run, timed through the public binding.

Every case is one call (or one served batch) of paper_2406_08923_gb300._lib on data that is
already where a user has it.  Sizes come from the benchmark's configurations (256^3 and 384^3
grids, 2^20 and 2^24 cells, 4096^2) and the tests' ragged shapes; plans are used as created,
without autotuning, as most callers do.

A case is a dict of plain values; "op" is what it runs:
  sweep      1D cross-correlation, radius <= 4 (FP32 <= 32), several sweeps per call
  wide       1D cross-correlation of a large radius, one sweep
  maxfilter  1D max filter, one sweep
  heat       forward-Euler heat steps in 1, 2 or 3 dimensions
  mhd        RK3 steps of the 8-field MHD system
  rhs        the MHD right-hand side alone (diagnostics)
  norms      per-field norms of an MHD state, with the mass (diagnostics between steps)
  serve      a batch of mixed requests through the continuous-batching server, host to host
"""
import math

import numpy as np
import torch

from paper_2406_08923_gb300 import _lib as L
from paper_2406_08923_gb300 import serving

_DT = {"i32": L.STENCIL_I32, "f64": L.STENCIL_F64, "f32": L.STENCIL_F32, "bf16": L.STENCIL_BF16}
_TORCH = {"i32": torch.int32, "f64": torch.float64, "f32": torch.float32, "bf16": torch.bfloat16}
_SIZE = {"i32": 4, "f64": 8, "f32": 4, "bf16": 2}


def listed():
    return [
        # one step of a small grid: an interactive or coupled caller that steps one call at a time
        {"name": "heat3d_f32_32", "op": "heat", "ndim": 3, "nx": 32, "ny": 32, "nz": 32, "r": 3, "type": "f32", "steps": 1},
        # the 2^20-cell, 10-sweep cross-correlation job in int32 and FP64
        {"name": "sweep_i32_1m", "op": "sweep", "n": 1 << 20, "r": 3, "type": "i32", "steps": 10},
        {"name": "sweep_f64_1m", "op": "sweep", "n": 1 << 20, "r": 3, "type": "f64", "steps": 10},
        # the radius sweep: a large-radius filter over 2^24 cells, and a ragged one in FP64
        {"name": "wide_f32_16m", "op": "wide", "n": 1 << 24, "r": 64, "type": "f32"},
        {"name": "wide_f64_3m", "op": "wide", "n": 3000001, "r": 100, "type": "f64"},
        # 2D heat equation at the radius sweep's size
        {"name": "heat2d_f32_4096", "op": "heat", "ndim": 2, "nx": 4096, "ny": 4096, "nz": 1, "r": 2, "type": "f32", "steps": 16},
        # the headline: 3D heat equation, 256^3 FP64, sixth order
        {"name": "heat3d_f64_256", "op": "heat", "ndim": 3, "nx": 256, "ny": 256, "nz": 256, "r": 3, "type": "f64", "steps": 10},
        # a grid whose extents no tile divides
        {"name": "heat3d_f32_ragged", "op": "heat", "ndim": 3, "nx": 301, "ny": 187, "nz": 250, "r": 3, "type": "f32", "steps": 20},
        # one RK3 step of the MHD system at the sizes of the benchmark, and a ragged one in BF16
        {"name": "mhd_f64_256", "op": "mhd", "nx": 256, "ny": 256, "nz": 256, "type": "f64", "steps": 1},
        {"name": "mhd_f32_384", "op": "mhd", "nx": 384, "ny": 384, "nz": 384, "type": "f32", "steps": 1},
        {"name": "mhd_bf16_ragged", "op": "mhd", "nx": 200, "ny": 150, "nz": 171, "type": "bf16", "steps": 1},
        # a burst of mixed requests on a running server
        {"name": "serve_mix_12", "op": "serve", "count": 12, "nmin": 32, "nmax": 96, "smin": 10, "smax": 20, "mix": 1},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["sweep", "sweep", "wide", "wide", "maxfilter", "heat", "heat", "heat", "heat", "mhd", "mhd", "mhd",
                     "rhs", "norms", "serve"])
    if op == "sweep":
        t = rng.choice(["i32", "f32", "f64"])
        r = rng.choice([1, 2, 3, 3, 4]) if t != "f32" else rng.choice([1, 2, 3, 4, 8, 16])
        return {"op": op, "n": _log(rng, 4099, (1 << 24) - 5), "r": r, "type": t, "steps": rng.randint(1, 16)}
    if op == "wide":
        t = rng.choice(["f32", "f64"])
        r = _log(rng, 5 if t == "f64" else 33, 1024)
        most = min(1 << 24, (2 << 30) // r if t == "f32" else (400 << 20) // r)
        return {"op": op, "n": _log(rng, 1 << 16, most), "r": r, "type": t}
    if op == "maxfilter":
        return {"op": op, "n": _log(rng, 1 << 14, 1 << 24), "r": _log(rng, 1, 1024), "type": rng.choice(["i32", "f32", "f64"])}
    if op == "heat":
        t, d = rng.choice(["f32", "f64"]), rng.choice([1, 2, 2, 3, 3, 3, 3])
        r = rng.choice([1, 2, 3, 3, 3, 4])
        hi = {1: 1 << 24, 2: 4096, 3: 420 if t == "f32" else 256}[d]
        lo = {1: 4099, 2: 61, 3: 17}[d]
        ext = [_log(rng, lo, hi) if i < d else 1 for i in range(3)]
        return {"op": op, "ndim": d, "nx": ext[0], "ny": ext[1], "nz": ext[2], "r": r, "type": t, "steps": rng.randint(1, 20)}
    if op == "serve":
        return {"op": op, "count": rng.randint(3, 12), "nmin": 32, "nmax": rng.choice([48, 64, 96]), "smin": 10, "smax": 20,
                "mix": rng.randint(2, 1 << 20)}
    t = rng.choice(["f32", "f64", "bf16"])
    hi = 256 if t != "f64" else 160
    e = [_log(rng, 17, hi) for _ in range(3)]
    return {"op": op, "nx": e[0], "ny": e[1], "nz": e[2], "type": t, "steps": 1}


# ------------------------------------------------------------------ inputs


def _gen(seed, salt=0):
    g = torch.Generator(device="cuda")
    g.manual_seed((int(seed) * 1000003 + salt * 7919) & 0x7FFFFFFF)
    return g


def _uniform(g, n, lo, hi):
    return torch.rand(n, generator=g, device="cuda", dtype=torch.float64) * (hi - lo) + lo


def _modes(g, shape, count, amps, kmax):
    """A periodic sum of sine modes with random wave vectors and phases, of shape (nz, ny, nx)."""
    out = torch.zeros(shape, device="cuda", dtype=torch.float64)
    k = torch.randint(1, kmax + 1, (count, 3), generator=g, device="cuda").double()
    ph = torch.rand(count, generator=g, device="cuda", dtype=torch.float64) * (2 * math.pi)
    ax = [torch.arange(n, device="cuda", dtype=torch.float64) * (2 * math.pi / n) for n in shape]
    for m in range(count):
        z = (k[m, 2] * ax[0] + ph[m]).view(-1, 1, 1) if shape[0] > 1 else ph[m].view(1, 1, 1)
        y = (k[m, 1] * ax[1]).view(1, -1, 1) if shape[1] > 1 else torch.zeros(1, 1, 1, device="cuda", dtype=torch.float64)
        out += amps[m] * torch.sin(z + y + (k[m, 0] * ax[2]).view(1, 1, -1))
    return out


def _weights(case, seed):
    rng = np.random.default_rng([int(seed), 11])
    r = case["r"]
    if case["op"] == "wide":  # a normalised averaging kernel
        w = rng.random(2 * r + 1)
        return w / w.sum()
    if case["type"] == "i32":
        return rng.integers(-8, 9, 2 * r + 1).astype(np.int32)
    w = rng.random(2 * r + 1) + 0.1  # a smoothing kernel, stable over any number of sweeps
    return w / w.sum()


def _shape(case):
    return (case["nz"], case["ny"], case["nx"])


def _heat_params(case):
    shape = _shape(case)[3 - case["ndim"]:]
    return L.heat_params(shape, dt=0.1 * min(2 * math.pi / n for n in shape) ** 2 / case["ndim"])


def _input(case, seed):
    """The case's interior input fields as device tensors of the storage type."""
    g, t = _gen(seed, 1), _TORCH[case["type"]]
    op = case["op"]
    if op == "sweep" and case["type"] == "i32":
        return [torch.randint(-1000, 1001, (case["n"],), generator=g, device="cuda", dtype=torch.int32)]
    if op == "sweep":
        return [_uniform(g, case["n"], -1.0, 1.0).to(t)]
    if op == "wide":
        return [_uniform(g, case["n"], 0.0, 1.0).to(t)]
    if op == "maxfilter":
        v = _uniform(g, case["n"], -1.0, 1.0)
        return [(v * 1e6).to(t) if case["type"] == "i32" else v.to(t)]
    if op == "heat":
        shape = _shape(case)
        f = _modes(g, shape, 4, [1.0] * 4, 8)
        f += 1e-3 * torch.randn(shape, generator=g, device="cuda", dtype=torch.float64)
        return [f.to(t)]
    out = []  # an MHD state: every field a few smooth modes of small amplitude
    for _ in range(8):
        amps = (torch.rand(4, generator=g, device="cuda", dtype=torch.float64) * 2 - 1) * 2e-2
        out.append(_modes(g, _shape(case), 4, amps, 4).to(t))
    return out


# ------------------------------------------------------------------ serving


def _requests(case):
    return serving.make_requests(case["count"], seed=int(case["mix"]), nmin=case["nmin"], nmax=case["nmax"],
                                 smin=case["smin"], smax=case["smax"])


def _request_inputs(case, seed):
    out = []
    for r in _requests(case):
        g = _gen(seed, 100 + r.index)
        if r.kind == L.STENCIL_XCORR:
            f = [_uniform(g, r.cells, -1.0, 1.0)]
        elif r.kind == L.STENCIL_DIFFUSION:
            f = [_modes(g, (r.n,) * 3, 4, [1.0] * 4, 8)]
        else:
            f = [_modes(g, (r.n,) * 3, 4, (torch.rand(4, generator=g, device="cuda", dtype=torch.float64) * 2 - 1) * 2e-2, 4)
                 for _ in range(8)]
        out.append((r, [x.float().reshape(-1) for x in f]))
    return out


def _prepare_serve(case, seed):
    jobs, outs = [], []
    for r, fields in _request_inputs(case, seed):
        ins = [f.cpu().pin_memory() for f in fields]
        res = [torch.empty(r.cells, dtype=torch.float32).pin_memory() for _ in fields]
        outs.append(res)
        jobs.append((serving.request_params(r.kind, r.n, r.nsteps), ins, [t.data_ptr() for t in ins],
                     [t.data_ptr() for t in res]))
    return {"op": "serve", "server": _Server(), "jobs": jobs, "out": outs}


class _Server:
    """A running server, released with the state that holds it."""

    def __init__(self):
        self.h = L.stencil_server_create(20 * 10 ** 9, 64)

    def __del__(self):
        try:
            L.stencil_server_destroy(self.h)
        except Exception:  # noqa: BLE001 -- interpreter shutdown
            pass


def _run_serve(state):
    h = state["server"].h
    todo = [L.stencil_server_submit(h, q, pin, pout) for q, _, pin, pout in state["jobs"]]
    while todo:
        L.stencil_server_progress(h)
        todo = [t for t in todo if L.stencil_server_poll(h, t) != L.STENCIL_REQ_DONE]
    return state["out"]


# ------------------------------------------------------------------ prepare / run


def _plan(case, seed):
    t = _DT[case["type"]]
    op = case["op"]
    if op in ("sweep", "wide"):
        return L.Plan(1, (case["n"],), case["r"], 1, L.STENCIL_BC_PERIODIC, L.STENCIL_XCORR, t, t, coeffs=_weights(case, seed))
    if op == "maxfilter":
        return L.Plan(1, (case["n"],), case["r"], 1, L.STENCIL_BC_PERIODIC, L.STENCIL_MAXFILTER, t, t)
    if op == "heat":
        d = case["ndim"]
        return L.Plan(d, (case["nx"], case["ny"], case["nz"])[:d], case["r"], 1, L.STENCIL_BC_PERIODIC, L.STENCIL_DIFFUSION,
                      t, t, params=_heat_params(case))
    c = L.STENCIL_F64 if case["type"] == "f64" else L.STENCIL_F32
    return L.Plan(3, (case["nx"], case["ny"], case["nz"]), 3, 8, L.STENCIL_BC_PERIODIC, L.STENCIL_MHD8, t, c,
                  params=L.mhd_params(_shape(case)))


def prepare(case, seed):
    if case["op"] == "serve":
        return _prepare_serve(case, seed)
    p = _plan(case, seed)
    a, b = p.alloc(), p.alloc()
    for t, f in zip(a, _input(case, seed)):
        p.interior(t).copy_(f.view(p.interior(t).shape))
    state = {"op": case["op"], "plan": p, "in": a, "out": b, "steps": case.get("steps", 1),
             "views": [p.interior(t) for t in b]}
    if case["op"] == "rhs":
        c = torch.float64 if case["type"] == "f64" else torch.float32
        state["views"] = [torch.empty(_shape(case), dtype=c, device="cuda") for _ in range(8)]
    return state


def run(state):
    op = state["op"]
    if op == "serve":
        return _run_serve(state)
    p = state["plan"]
    if op == "norms":
        return p.norms(state["in"])
    if op == "rhs":
        p.mhd_rhs(state["in"], state["views"])
    else:
        p.step(state["in"], state["out"], state["steps"])
    return state["views"]


# ------------------------------------------------------------------ work


def work(case):
    op = case["op"]
    if op == "serve":
        b = f = 0
        for r in _requests(case):
            b += 2 * 4 * r.cells * r.nfields
            per = {L.STENCIL_XCORR: 14, L.STENCIL_DIFFUSION: 38, L.STENCIL_MHD8: 822}[r.kind]
            f += per * r.work()
        return {"bytes": b, "flops": f}
    e = _SIZE[case["type"]]
    if op in ("sweep", "wide", "maxfilter"):
        per = 2 * (2 * case["r"] + 1) if op != "maxfilter" else 2 * max(1, math.ceil(math.log2(2 * case["r"] + 1)))
        return {"bytes": 2 * e * case["n"], "flops": per * case["n"] * case.get("steps", 1)}
    cells = case["nx"] * case["ny"] * case["nz"]
    if op == "heat":
        return {"bytes": 2 * e * cells, "flops": 2 * (2 * case["r"] * case["ndim"] + 1) * cells * case["steps"]}
    if op == "norms":
        return {"bytes": 8 * e * cells, "flops": (8 * 4 + 20) * cells}
    if op == "rhs":
        return {"bytes": 8 * (e + (8 if e == 8 else 4)) * cells, "flops": 795 * cells}
    return {"bytes": 16 * e * cells, "flops": 2465 * cells * case["steps"]}


# ------------------------------------------------------------------ tolerance


def tolerance(case):
    """About four times the distance from a plain 64-bit evaluation, per storage type: one RK3
    step changes a state little, and sums of up to 2049 terms may be taken in any order."""
    op, t = case["op"], case.get("type", "f32")
    if (t == "i32" and op != "norms") or op == "maxfilter":
        return "exact"
    if op == "norms":  # the sums of a few signed modes nearly cancel
        return {"rel": 1e-9}
    if op == "rhs":
        return {"rel": 2e-13, "max": 1e-11} if t == "f64" else {"rel": 2e-5, "max": 2e-3}
    if t == "f64":
        return {"rel": {"heat": 6e-15, "sweep": 3e-15, "wide": 3e-15, "mhd": 2e-15}[op], "max": 3e-13}
    if t == "bf16":  # one rounding of the stored value
        return {"rel": 7e-3, "max": 4e-2}
    return {"rel": 1e-6 if op == "mhd" else 4e-6, "max": 1e-4}


# ------------------------------------------------------------------ plain 64-bit evaluation


def _corr(f, w, steps):
    r = len(w) // 2
    for _ in range(steps):
        acc = torch.zeros_like(f)
        for j in range(-r, r + 1):
            acc += w[j + r] * torch.roll(f, -j)
        f = acc
    return f


def _lap_weights(r):
    fact = math.factorial
    c = [0.0] * (r + 1)
    for k in range(1, r + 1):
        c[k] = 2.0 * (-1) ** (k + 1) * fact(r) ** 2 / (k * k * fact(r - k) * fact(r + k))
        c[0] -= 2.0 / (k * k)
    return c


def _heat64(f, r, dt, alpha, h, ndim, steps):
    c = _lap_weights(r)
    for _ in range(steps):
        lap = torch.zeros_like(f)
        for a in range(ndim):
            d = 2 - a  # axis 0 is x, the last dimension
            s = c[0] * f
            for k in range(1, r + 1):
                s += c[k] * (torch.roll(f, -k, d) + torch.roll(f, k, d))
            lap += s / (h[a] * h[a])
        f = f + dt * alpha * lap
    return f


def _mhd_rhs64(f, p):
    """Right-hand sides of the 8-field system (continuity, momentum, entropy, induction; constant
    viscosity and diffusivity, ideal gas) from sixth-order central differences."""
    h = (p.dx[0], p.dx[1], p.dx[2])
    w1 = (3 / 4, -3 / 20, 1 / 60)
    w2c, w2 = -49 / 18, (3 / 2, -3 / 20, 1 / 90)
    wm = (270.0, -27.0, 2.0)

    def sh(q, *moves):
        for axis, s in moves:
            q = torch.roll(q, -s, 2 - axis)
        return q

    def d1(q, a):
        return sum(w1[k - 1] * (sh(q, (a, k)) - sh(q, (a, -k))) for k in (1, 2, 3)) / h[a]

    def d2(q, a):
        return (w2c * q + sum(w2[k - 1] * (sh(q, (a, k)) + sh(q, (a, -k))) for k in (1, 2, 3))) / h[a] ** 2

    def dd(q, a, b):
        if a == b:
            return d2(q, a)
        s = sum(wm[k - 1] * (sh(q, (a, k), (b, k)) + sh(q, (a, -k), (b, -k)) - sh(q, (a, k), (b, -k)) - sh(q, (a, -k), (b, k)))
                for k in (1, 2, 3))
        return s / (720.0 * h[a] * h[b])

    lnrho, u, A, ss = f[0], f[1:4], f[4:7], f[7]
    glr, gs = [d1(lnrho, a) for a in range(3)], [d1(ss, a) for a in range(3)]
    gu = [[d1(u[c], a) for a in range(3)] for c in range(3)]
    divu = gu[0][0] + gu[1][1] + gu[2][2]
    bx, by, bz = d1(A[2], 1) - d1(A[1], 2), d1(A[0], 2) - d1(A[2], 0), d1(A[1], 0) - d1(A[0], 1)
    B = (bx, by, bz)
    lapa = [d2(A[c], 0) + d2(A[c], 1) + d2(A[c], 2) for c in range(3)]
    J = [(sum(dd(A[c], a, c) for c in range(3)) - lapa[a]) / p.mu0 for a in range(3)]

    def cross(v, w, a):
        b, c = (a + 1) % 3, (a + 2) % 3
        return v[b] * w[c] - v[c] * w[b]

    def adv(g):
        return u[0] * g[0] + u[1] * g[1] + u[2] * g[2]

    S = [[0.5 * (gu[i][j] + gu[j][i]) - (divu / 3 if i == j else 0.0) for j in range(3)] for i in range(3)]
    s2 = sum(S[i][j] * S[i][j] for i in range(3) for j in range(3))
    rho = torch.exp(lnrho)
    cs2 = p.cs0 ** 2 * torch.exp(p.gamma * ss / p.cp + (p.gamma - 1) * (lnrho - p.lnrho0))
    out = [-adv(glr) - divu]
    for a in range(3):
        lapu = d2(u[a], 0) + d2(u[a], 1) + d2(u[a], 2)
        gdiv = sum(dd(u[c], a, c) for c in range(3))
        sg = sum(S[a][j] * glr[j] for j in range(3))
        out.append(-adv(gu[a]) - cs2 * (gs[a] / p.cp + glr[a]) + cross(J, B, a) / rho
                   + p.nu * (lapu + gdiv / 3 + 2 * sg) + p.zeta * gdiv)
    for a in range(3):
        out.append(cross(u, B, a) + p.eta * lapa[a])
    heat = p.eta * p.mu0 * (J[0] ** 2 + J[1] ** 2 + J[2] ** 2) + 2 * rho * p.nu * s2 + p.zeta * rho * divu ** 2
    out.append(-adv(gs) + heat * p.cp * (p.gamma - 1) / (rho * cs2))
    return out


def _mhd64(f, p, steps):
    alpha, beta = (0.0, -5 / 9, -153 / 128), (1 / 3, 15 / 16, 8 / 15)
    for _ in range(steps):
        w = [torch.zeros_like(q) for q in f]
        for s in range(3):
            rhs = _mhd_rhs64(f, p)
            w = [alpha[s] * a + p.dt * b for a, b in zip(w, rhs)]
            f = [q + beta[s] * a for q, a in zip(f, w)]
    return f


def exact(case, seed):
    op = case["op"]
    if op == "serve":
        out = []
        for r, fields in _request_inputs(case, seed):
            if r.kind == L.STENCIL_XCORR:
                out.append([_corr(fields[0].double(), [float(np.float32(w)) for w in serving.XC_WEIGHTS], r.nsteps)])
                continue
            q = serving.request_params(r.kind, r.n, r.nsteps).params
            f = [x.double().view((r.n,) * 3) for x in fields]
            if r.kind == L.STENCIL_DIFFUSION:
                res = [_heat64(f[0], 3, q.dt, q.alpha, tuple(q.dx), 3, r.nsteps)]
            else:
                res = _mhd64(f, q, r.nsteps)
            out.append([x.reshape(-1) for x in res])
        return out
    fields = _input(case, seed)
    if op == "maxfilter":
        f = fields[0]
        m = torch.cat([f[-case["r"]:], f, f[:case["r"]]])  # windows by doubling
        width, left = 1, 2 * case["r"] + 1
        while 2 * width <= left:
            m = torch.maximum(m[:-width], m[width:])
            width *= 2
        return [torch.maximum(m[:case["n"]], m[left - width:left - width + case["n"]])]
    if op in ("sweep", "wide"):
        if case["type"] == "i32":
            return [_corr(fields[0], [int(w) for w in _weights(case, seed)], case["steps"])]
        w = _weights(case, seed)
        if case["type"] == "f32":
            w = w.astype(np.float32)
        return [_corr(fields[0].double(), [float(x) for x in w], case.get("steps", 1))]
    if op == "heat":
        p = _heat_params(case)
        f = _heat64(fields[0].double(), case["r"], p.dt, p.alpha, tuple(p.dx), case["ndim"], case["steps"])
        return [f.view(f.shape[3 - case["ndim"]:])]
    p = L.mhd_params(_shape(case))
    f = [q.double() for q in fields]
    if op == "rhs":
        return _mhd_rhs64(f, p)
    if op == "norms":
        vals = []
        for q in f:
            vals += [float(q.sum()), float((q * q).sum()), float(q.abs().max())]
        return np.array(vals + [float(torch.exp(f[0]).sum() * p.dx[0] * p.dx[1] * p.dx[2])])
    return _mhd64(f, p, case["steps"])
