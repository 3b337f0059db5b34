#!/usr/bin/env python3
"""Benchmark of the GB300 stencil engine.

Headline workload: the 3D heat equation with the 6th-order 19-point Laplacian, 256^3 cells,
FP64, periodic halos, forward Euler dt = 0.1 dx^2, 100 steps (Sec. 3.2, Eqs. 4-7).  One bench
step is one whole job: stencil_step(plan, in, out, 100) -- the input halo fill and 100 fused
Euler passes, each writing its output's periodic halo.  The metric is Mcell-updates/s
(cells x Euler steps / time).  The two 145 MB padded FP64 fields the passes stream between
exceed the 126 MB L2, so no flush is needed between iterations.

The JSON line also carries, per the other stencil workloads (1D cross-correlation, FP32 heat,
fused 8-field MHD in FP64 and in FP32/BF16 storage), their own throughput and roofline.

  python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference] [--no-extras] [--zslab]

Under torchrun (N > 1) every rank solves its own independent grid (weak scaling, no
data-path collective); the time is the max over ranks.  --zslab instead decomposes the one
256^3 grid along z over the ranks (strong scaling, a 3-plane halo exchange per Euler step).  --impl reference times the FP64 CPU
oracle on the host cores on a bounded sample of the same workload.
"""
from __future__ import annotations

import argparse
import json
import os
import statistics
import subprocess
import sys
import tempfile
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

import numpy as np  # noqa: E402

HEAT_N, HEAT_STEPS = 256, 100
HEADLINE_VARIANT = 0
MHD_N, MHD_N_LOWP, MHD_STEPS = 256, 384, 20
XC_N, XC_SWEEPS = 1 << 20, 10


def _peaks():
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(p):
        d = json.load(open(p))
        return float(d["hbm_gbs"]), "measured"
    return 6800.0, "fallback"


# DRAM traffic per launch of the dominant kernel from one ncu capture (profiles/), valid only
# while the kernel source is unchanged (first 16 hex digits of sha256 of each file).
SRC_MHD = {"mhd.cu": "7247c6ba8525b938", "mhd_win.cuh": "a8287b7e01d5801c", "mhd_rhs.cuh": "be5b445fecd5703b", "common.cuh": "3f7458d1c75ca5f9"}
SRC_HEAT32 = {"diffusion_f32.cu": "2cacbf4617d874ff", "common.cuh": "3f7458d1c75ca5f9"}
NCU_TRAFFIC = {
    # dram__bytes_read.sum + dram__bytes_write.sum per launch, mean of 3 launches of a 1-pass capture at
    # the bench sizes (profiles/dram_traffic_full_size.md); MHD: the mean over the 3 RK substeps
    "heat_f64": {"variant": "fx64x16", "zmode": 0, "bytes": 147750229 + 102371072,
                 "src": {"diffusion_fx.cu": "2b4f7cb8238067a7", "fixed.cuh": "84e7b11e6dde86ee", "common.cuh": "3f7458d1c75ca5f9"}},
    "heat_f32": {"variant": "f32_by4_ry2_zb2_s8_m3", "zmode": 0, "bytes": 82052181 + 21760939, "src": SRC_HEAT32},
    "heat_f32_512": {"variant": "f32_by8_ry2_zb2_s8_m2", "zmode": 0, "bytes": 586154069 + 507398315,
                     "src": SRC_HEAT32},
    "mhd_f32": {"variant": "tx32_ty12_s8_b1", "zmode": 1, "bytes": 5369747115 + 4896249685, "src": SRC_MHD},
    "mhd_bf16": [
        {"variant": "tx32_ty8_s8_b2", "zmode": 1, "bytes": 3312621312 + 2566468779, "src": SRC_MHD},
        {"variant": "tx32_ty4_s8_b3", "zmode": 1, "bytes": 2714962944 + 2446886229, "src": SRC_MHD},
    ],
}


def _traffic_records(case):
    """The capture records of a case: one record, or a list (one per captured variant / z-chunk mode)."""
    rec = NCU_TRAFFIC.get(case)
    return [] if rec is None else (rec if isinstance(rec, list) else [rec])


def _traffic(case, variant_name, zmode=0):
    import hashlib
    for rec in _traffic_records(case):
        if rec["variant"] != variant_name or rec.get("zmode", 0) != zmode:
            continue
        for f, h in rec["src"].items():
            path = os.path.join(ROOT, "paper_2406_08923_gb300", "csrc", f)
            if hashlib.sha256(open(path, "rb").read()).hexdigest()[:16] != h:
                return None
        return rec["bytes"]
    return None


# FP64 vector FMA rate of GB300 (nominal 1.25 TFLOP/s dense, recipe table); FP32 from the
# unit count: 152 SMs x 128 FP32 lanes x 2 flop x 2.07 GHz boost.
FP64_PEAK_TFLOPS = 1.25
FP64_PIPE_TINSTR = 2 * 152 * 2.07e9 / 1e12  # FP64 instructions (DFMA, DADD, DMUL alike) per s
# Algorithmic FP64 work of one MHD cell-substep (mean over the 3 RK substeps): the pruned
# 6th-order derivatives (600 flop), the right-hand side of Eqs. A1-A4 and the 2N-storage RK
# update, counted by tests/mhd_flops.py (checked against the oracle in test_mhd_flops.py).
MHD_FLOPS_PER_CELL_SUBSTEP = 2465 / 3
MHD_F64_INSTR = 200  # FP64 instructions per cell-substep the kernel executes (ncu sass counts)
# 32 x 32 + 64-bit multiply-adds of the integer pipe, which the FP64 linear stencils run on: 32
# lanes per clock and SM (28 to 30 measured with distinct operands).
INT_PIPE_TINSTR = 32 * 152 * 2.07e9 / 1e12
FP32_PEAK_TFLOPS = 152 * 128 * 2 * 2.07e9 / 1e12


class Clocks:
    """nvidia-smi sampling of SM clocks and throttle reasons during a timed region."""

    Q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
         "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
         "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index: int):
        self.idx = gpu_index
        self.proc = None
        self.path = None

    def __enter__(self):
        fd, self.path = tempfile.mkstemp(prefix="clocks", suffix=".csv")
        os.close(fd)
        try:
            self.proc = subprocess.Popen(["nvidia-smi", "-i", str(self.idx), f"--query-gpu={self.Q}",
                                          "--format=csv,noheader,nounits", "-lms", "200"],
                                         stdout=open(self.path, "w"), stderr=subprocess.DEVNULL)
        except OSError:
            self.proc = None
        time.sleep(0.3)
        return self

    def __exit__(self, *exc):
        if self.proc is not None:
            self.proc.terminate()
            try:
                self.proc.wait(timeout=5)
            except subprocess.TimeoutExpired:
                self.proc.kill()

    def summary(self):
        sm, smax, reasons = [], None, set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        try:
            for line in open(self.path):
                f = [x.strip() for x in line.split(",")]
                if len(f) < 9:
                    continue
                try:
                    sm.append(float(f[1]))
                    smax = float(f[2])
                except ValueError:
                    continue
                for n, v in zip(names, f[5:9]):
                    if v.lower().startswith("active"):
                        reasons.add(n)
            os.unlink(self.path)
        except OSError:
            pass
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": smax,
                "samples": len(sm), "reasons": sorted(reasons)}


# ----------------------------------------------------------------------------- helpers


def _dist(backend=None):
    """(rank, world, torch.distributed or None) from the torchrun environment.  The data path
    has no collective: ranks only meet in barriers and the max-over-ranks timing reduction."""
    ws = int(os.environ.get("WORLD_SIZE", "1"))
    if ws <= 1:
        return 0, 1, None
    import torch
    import torch.distributed as dist
    rank = int(os.environ["RANK"])
    local = int(os.environ.get("LOCAL_RANK", rank))
    if backend is None:
        backend = "nccl" if torch.cuda.is_available() else "gloo"
    if backend == "nccl":
        torch.cuda.set_device(local)
    dist.init_process_group(backend)
    return rank, ws, dist


def _barrier(dist):
    if dist is not None:
        dist.barrier()


def _max_over_ranks(v, dist):
    if dist is None:
        return v
    import torch
    dev = "cuda" if dist.get_backend() == "nccl" else "cpu"
    t = torch.tensor([v], dtype=torch.float64, device=dev)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def weak_scaling_value(world, units_per_rank, seconds):
    """Whole-job throughput in millions of units per second: every rank processed
    units_per_rank in the same (max-over-ranks) time."""
    return world * units_per_rank / seconds / 1e6


def _timed(fn, reps, stream):
    """Average ms of fn() over reps, CUDA events on `stream`, synchronised on both sides."""
    import torch
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    torch.cuda.synchronize()
    e0.record(stream)
    for _ in range(reps):
        fn()
    e1.record(stream)
    torch.cuda.synchronize()
    return e0.elapsed_time(e1) / reps


def _roof(bound, achieved, peak, unit, traffic=None, note=""):
    return {"bound": bound, "achieved": round(achieved, 4), "peak": round(peak, 4), "unit": unit,
            "frac": round(achieved / peak, 4), "traffic": traffic, "peak_source": note}


# ----------------------------------------------------------------------------- workloads


def heat_job(L, synth, dtype, n, steps, warmup, reps, stream, with_e2e=False, variant=None):
    """Time stencil_step(n^3 heat, `steps` Euler steps) and its per-kernel average.
    variant=None runs the autotuner (Sec. 5.1); an int pins the kernel variant."""
    import torch
    par = L.heat_params(n)
    p = L.Plan(3, (n, n, n), 3, 1, L.STENCIL_BC_PERIODIC, L.STENCIL_DIFFUSION, dtype, dtype, params=par)
    a, b = p.alloc(), p.alloc()
    p.upload(a, [synth.heat_field(n)])
    p.halo_fill(a)
    torch.cuda.synchronize()
    if variant is None:  # tuned on the job itself: the schedules differ in per-call costs
        p.autotune(a, b, nsteps=steps, reps=2, stream=stream)
    else:
        p.set_variant(variant)
    for _ in range(warmup):
        p.step(a, b, steps, stream)
    res = {"plan": p, "fields": (a, b), "variant": p.variant()[2]}
    res["ms_job"] = _timed(lambda: p.step(a, b, steps, stream), reps, stream)
    ms_halo = _timed(lambda: p.halo_fill(a, stream), max(reps, 10), stream)
    res["ms_kernel"] = (res["ms_job"] - ms_halo) / steps
    res["ms_halo"] = ms_halo
    # halo fill + one launch per step, or halo fill + one persistent launch for all steps
    res["persistent"] = res["variant"].endswith("_persist")
    res["launches_per_job"] = 2 if res["persistent"] else steps + 1
    if with_e2e:
        nbytes = p.bytes_per_field
        h_in = torch.empty(nbytes // a[0].element_size(), dtype=a[0].dtype, pin_memory=True)
        h_out = torch.empty_like(h_in, pin_memory=True)
        h_in.copy_(a[0].cpu())
        d_in = p.alloc()

        def e2e():
            d_in[0].copy_(h_in, non_blocking=True)
            p.step(d_in, b, steps, stream)
            h_out.copy_(b[0], non_blocking=True)

        for _ in range(max(1, warmup // 2)):
            e2e()
        res["ms_e2e"] = _timed(e2e, reps, stream)
        res["e2e_bytes"] = (nbytes, nbytes)
    return res


def mhd_job(L, synth, storage, n, steps, warmup, reps, stream):
    import torch
    par = L.mhd_params(n)
    compute = L.STENCIL_F64 if storage == L.STENCIL_F64 else L.STENCIL_F32
    p = L.Plan(3, (n, n, n), 3, 8, L.STENCIL_BC_PERIODIC, L.STENCIL_MHD8, storage, compute, params=par)
    a, b = p.alloc(), p.alloc()
    seed = synth.SEED_MHD if storage == L.STENCIL_F64 else synth.SEED_MHD_LOWP
    p.upload(a, synth.mhd_fields(n, seed=seed))
    torch.cuda.synchronize()
    p.autotune(a, b, nsteps=1, reps=1, stream=stream)
    for _ in range(warmup):
        p.step(a, b, steps, stream)
    ms_job = _timed(lambda: p.step(a, b, steps, stream), reps, stream)
    ms_halo = _timed(lambda: p.halo_fill(a, stream), 5, stream)
    ms_sub = (ms_job - ms_halo) / (3 * steps)
    norms = p.norms(b)
    return {"plan": p, "fields": b, "ms_job": ms_job, "ms_substep": ms_sub, "variant": p.variant()[2],
            "mass": float(norms[-1]), "finite": bool(np.all(np.isfinite(norms)))}


def xcorr_job(L, synth, dtype, warmup, reps, stream):
    import torch
    n = XC_N
    if dtype == L.STENCIL_I32:
        data, g = synth.xcorr_int32(n)
    else:
        data = synth.xcorr_f64(n)
        g = np.array([1 / 90, -3 / 20, 3 / 2, -49 / 18, 3 / 2, -3 / 20, 1 / 90])
    p = L.Plan(1, (n,), 3, 1, L.STENCIL_BC_PERIODIC, L.STENCIL_XCORR, dtype, dtype, coeffs=g)
    a, b = p.alloc(), p.alloc()
    p.upload(a, [data])
    torch.cuda.synchronize()
    for _ in range(warmup):
        p.step(a, b, XC_SWEEPS, stream)
    ms_eager = _timed(lambda: p.step(a, b, XC_SWEEPS, stream), reps, stream)
    # a job is one launch of ~10-200 us, so the host's launch path can dominate: also replay
    # the job as a CUDA graph (stencil_step neither allocates nor synchronises)
    graph = torch.cuda.CUDAGraph()
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        p.step(a, b, XC_SWEEPS, side)
    torch.cuda.current_stream().wait_stream(side)
    with torch.cuda.graph(graph):
        p.step(a, b, XC_SWEEPS, torch.cuda.current_stream())
    graph.replay()
    ms = _timed(graph.replay, reps, torch.cuda.current_stream())
    return {"ms_job": ms, "ms_job_eager": ms_eager}


def run_radius_sweep(L, synth, stream, hbm_peak):
    """Diffusion equation at radius 1..4 (order-2r Laplacian) in 1D, 2D and 3D, FP32 and FP64
    (Sec. 5.3, Figs. 10-11): 2^24 cells per problem (64 MiB FP32 / 128 MiB FP64, the paper's
    sizes): 2^24 in 1D, 4096^2 in 2D, 256^3 in 3D.  Time per Euler step and its fraction of
    HBM bandwidth at one read and one write per cell-step (1D runs up to 16 steps per launch in
    shared memory and 2D FP32 up to 4 when the autotuner picks temporal blocking, so their
    traffic is lower than that)."""
    out = {}
    shapes = {1: (1 << 24,), 2: (4096, 4096), 3: (256, 256, 256)}
    steps = {1: 64, 2: 20, 3: 20}
    for ndim, shape in shapes.items():
        n = int(np.prod(shape))
        base = synth.uniform(2406089237, ndim, n, -1.0, 1.0).reshape(shape)
        for st, name, esize in ((L.STENCIL_F32, "fp32", 4), (L.STENCIL_F64, "fp64", 8)):
            for r in (1, 2, 3, 4):
                p = L.Plan(ndim, tuple(reversed(shape)), r, 1, L.STENCIL_BC_PERIODIC, L.STENCIL_DIFFUSION, st, st,
                           params=L.heat_params(shape))
                a, b = p.alloc(), p.alloc()
                p.upload(a, [base])
                if (ndim == 3 and r == 3) or (ndim == 2 and st == L.STENCIL_F32):
                    # 2D FP32: the tile kernel or temporal blocking (2 or 4 steps per pass)
                    p.autotune(a, b, nsteps=4, reps=2, stream=stream)
                k = steps[ndim]
                p.step(a, b, k, stream)
                ms = _timed(lambda: p.step(a, b, k, stream), 3, stream) / k
                gbs = n * 2.0 * esize / (ms / 1e3) / 1e9
                ent = {"ms_per_step": round(ms, 5), "gcell_updates_per_s": round(n / (ms / 1e3) / 1e9, 2),
                       "hbm_gbs_at_1r1w": round(gbs, 1), "frac_of_hbm": round(gbs / hbm_peak, 4),
                       "variant": p.variant()[2]}
                if st == L.STENCIL_F64:
                    # 1 + 2 d r multiply-adds per cell (1D: 2r + 1 of the folded cross-correlation).
                    # 2D runs them on the FP64 pipe, 1D and 3D in fixed point on the integer
                    # pipe, several times the FP64 peak
                    inst = (2 * r + 1) if ndim == 1 else (1 + 2 * ndim * r)
                    tf = n * inst * 2.0 / (ms / 1e3) / 1e12
                    ent["fp64_tflops"] = round(tf, 3)
                    ent["times_fp64_peak"] = round(tf / FP64_PEAK_TFLOPS, 4)
                out[f"{ndim}d_{name}_r{r}"] = ent
                p.close()
                del a, b
    return out


FP32_MEASURED_TFLOPS = 74.3  # FP32 FMA probe on GB300 (152 SMs x 128 lanes at ~1.9 GHz under load)


def run_xcorr_radius_sweep(L, synth, stream, hbm_peak):
    """1D cross-correlation (Eq. 3) and max filter (Sec. 2.1) over the radius sweep of Sec. 5.2
    (Fig. 8): 2^24 cells (64 MiB FP32, 128 MiB FP64), r = 0 .. 1024.  Radius <= 4 runs the
    temporally blocked kernel (16 sweeps per launch); larger radii one sweep per launch.
    Cross-correlation at large radius is FMA bound: 2 (2r+1) flop per output."""
    out = {}
    n = 1 << 24
    radii = (0, 1, 2, 4, 8, 16, 32, 64, 128, 256, 512, 1024)
    base = synth.uniform(2406089239, 1, n, 0.0, 1.0)
    for st, name, esize, peak in ((L.STENCIL_F32, "fp32", 4, FP32_MEASURED_TFLOPS), (L.STENCIL_F64, "fp64", 8, FP64_PEAK_TFLOPS)):
        for kind, kname in ((L.STENCIL_XCORR, "xcorr"), (L.STENCIL_MAXFILTER, "maxfilter")):
            for r in radii:
                g = None
                if kind == L.STENCIL_XCORR:
                    g = synth.uniform(2406089239, 10 + r, 2 * r + 1, 0.0, 1.0)
                    g = g / g.sum()
                p = L.Plan(1, (n,), r, 1, L.STENCIL_BC_PERIODIC, kind, st, st, coeffs=g)
                a, b = p.alloc(), p.alloc()
                p.upload(a, [base])
                k = 16 if (kind == L.STENCIL_XCORR and r <= 4) else (1 if (st == L.STENCIL_F64 and r >= 256) else 4)
                p.step(a, b, k, stream)
                ms = _timed(lambda: p.step(a, b, k, stream), 2, stream) / k
                gbs = n * 2.0 * esize / (ms / 1e3) / 1e9
                ent = {"ms_per_sweep": round(ms, 5), "gcell_per_s": round(n / (ms / 1e3) / 1e9, 2),
                       "hbm_gbs_at_1r1w": round(gbs, 1), "frac_of_hbm": round(gbs / hbm_peak, 4)}
                if kind == L.STENCIL_XCORR:
                    tf = n * 2.0 * (2 * r + 1) / (ms / 1e3) / 1e12
                    ent["tflops"] = round(tf, 3)
                    if st == L.STENCIL_F32:
                        ent["frac_of_fma_peak"] = round(tf / peak, 4)
                    else:
                        ent["times_fp64_peak"] = round(tf / peak, 4)
                    if st == L.STENCIL_F64 and r > 4:  # three integer multiply-adds per tap
                        ent["frac_of_int_pipe"] = round(tf / 2 * 3 / INT_PIPE_TINSTR, 4)
                out[f"{kname}_{name}_r{r}"] = ent
                p.close()
                del a, b
    return out


def run_serving_leg(n_requests=1024, load=0.7, fp64_subset=96, sweep=(0.5, 1.2)):
    """Serving configuration: 1024 requests (log-uniform 32^3..192^3, mixed kinds, 10-50
    steps, FP32) through the continuous-batching server under a 120 GB budget.

    1. saturation: every request arrives at t = 0; capacity = requests / wall time;
    2. open loop: Poisson arrivals at `load` x capacity; p50/p99 arrival-to-result latency
       and aggregate throughput;
    3. the plain per-grid FP64 path (one plan per request, in arrival order) on the first
       `fp64_subset` requests: service times measured, FIFO latencies under the same arrival
       process computed from them; speedup = batched / per-grid throughput at equal work."""
    import torch

    from paper_2406_08923_gb300 import _lib as L
    from paper_2406_08923_gb300 import serving
    t_gen = time.perf_counter()
    templates = serving.Templates(pinned=True)
    reqs = serving.make_requests(n_requests)
    for r in reqs:
        templates.get(r.kind, r.n)
    t_gen = time.perf_counter() - t_gen
    work = sum(r.work() for r in reqs)
    # the batched kernels' tile shapes: the autotuner's choice for FP32 plans of each kind (the
    # FP32 heat and MHD legs above tuned them in this process)
    probe = L.stencil_server_create(10 ** 9, 4)
    tiles = {serving.KIND_NAMES[k]: L.stencil_server_variant(probe, k) for k in serving.KINDS}
    L.stencil_server_destroy(probe)
    # warm-up: a few small requests (module load, graph instantiation, pool growth)
    warm = [serving.Request(i, k, 32, 2) for i, k in enumerate(serving.KINDS)]
    serving.serve(warm, templates)
    # 1. saturation
    for r in reqs:
        r.arrival = 0.0
    wall_sat, peak_sat, _ = serving.serve(reqs, templates)
    cap_rps = n_requests / wall_sat
    # 2. open loop at load x capacity
    serving.poisson_arrivals(reqs, load * cap_rps)
    wall, peak, updates = serving.serve(reqs, templates)
    lat = serving.latency_stats(reqs)
    # the same mix at other offered loads (below and above capacity)
    sweep_out = []
    for ld in sweep:
        serving.poisson_arrivals(reqs, ld * cap_rps)
        w2, p2, u2 = serving.serve(reqs, templates)
        l2 = serving.latency_stats(reqs)
        sweep_out.append({"load": ld, "rate_rps": round(ld * cap_rps, 1), "wall_s": round(w2, 3),
                          "mcell_updates_per_s": round(u2 / w2 / 1e6, 1), "p50_ms": round(l2["p50_ms"], 2),
                          "p99_ms": round(l2["p99_ms"], 2), "peak_gb": round(p2 / 1e9, 2)})
    serving.poisson_arrivals(reqs, load * cap_rps)
    # ragged sizes: 128 requests with n not rounded (most edges not a multiple of 4 or 8, so
    # the batched kernels take their element-wise edge paths), saturation and open loop
    rag = serving.make_requests(128, seed=serving.SEED_SERVE + 1, round_to=1)
    for r in rag:
        templates.get(r.kind, r.n)
    for r in rag:
        r.arrival = 0.0
    wall_r, peak_r, _ = serving.serve(rag, templates)
    cap_r = len(rag) / wall_r
    serving.poisson_arrivals(rag, load * cap_r)
    wall_ro, _, upd_ro = serving.serve(rag, templates)
    lat_r = serving.latency_stats(rag)
    ragged = {"requests": len(rag), "n_not_multiple_of_8": sum(r.n % 8 != 0 for r in rag),
              "work_gcell_updates": round(sum(r.work() for r in rag) / 1e9, 2),
              "saturation": {"wall_s": round(wall_r, 3), "requests_per_s": round(cap_r, 1),
                             "mcell_updates_per_s": round(sum(r.work() for r in rag) / wall_r / 1e6, 1)},
              "open_loop": {"load": load, "rate_rps": round(load * cap_r, 1), "p50_ms": round(lat_r["p50_ms"], 2),
                            "p99_ms": round(lat_r["p99_ms"], 2),
                            "mcell_updates_per_s": round(upd_ro / wall_ro / 1e6, 1)}}
    # 3. per-grid FP64 path on a subset, FIFO latencies under the same arrivals
    sub = sorted(reqs, key=lambda r: r.arrival)[:fp64_subset]
    arr = [r.arrival for r in sub]
    serving.serve_per_grid(sub[:2], templates, storage=L.STENCIL_F64)  # warm-up
    t0 = time.perf_counter()
    service = []
    for r in sub:
        t1 = time.perf_counter()
        serving.serve_per_grid([r], templates, storage=L.STENCIL_F64)
        service.append(time.perf_counter() - t1)
    wall64 = time.perf_counter() - t0
    done, lat64 = 0.0, []
    for a, sv in zip(arr, service):
        start = max(a, done)
        done = start + sv
        lat64.append(done - a)
    work_sub = sum(r.work() for r in sub)
    thr = updates / wall / 1e6
    thr64 = work_sub / wall64 / 1e6
    torch.cuda.synchronize()
    return {
        "requests": n_requests, "mix": "n log-uniform 32..192 (rounded to multiples of 8, so that one pinned input "
                                        "template per kind and size is kept; ragged_sizes runs unrounded n), kinds "
                                        "uniform {xcorr1d n^3, heat3d, mhd8}, 10-50 steps, FP32, Poisson arrivals",
        "budget_gb": 120, "template_gen_s": round(t_gen, 1), "batched_tiles": tiles,
        "work_gcell_updates": round(work / 1e9, 2),
        "saturation": {"wall_s": round(wall_sat, 3), "requests_per_s": round(cap_rps, 1),
                       "mcell_updates_per_s": round(work / wall_sat / 1e6, 1), "peak_gb": round(peak_sat / 1e9, 2)},
        "open_loop": {"load": load, "rate_rps": round(load * cap_rps, 1), "wall_s": round(wall, 3),
                      "mcell_updates_per_s": round(thr, 1), "p50_ms": round(lat["p50_ms"], 2),
                      "p99_ms": round(lat["p99_ms"], 2), "peak_gb": round(peak / 1e9, 2)},
        "load_sweep": sweep_out,
        "ragged_sizes": ragged,
        "per_grid_fp64_subset": {"requests": len(sub), "wall_s": round(wall64, 3),
                                 "mcell_updates_per_s": round(thr64, 1),
                                 "p50_ms": round(float(np.percentile(lat64, 50) * 1e3), 2),
                                 "p99_ms": round(float(np.percentile(lat64, 99) * 1e3), 2)},
        # capacity ratio: saturated batched throughput vs back-to-back per-grid FP64 throughput
        "speedup_vs_per_grid_fp64": round(work / wall_sat / 1e6 / thr64, 2),
        "speedup_open_loop_throughput": round(thr / thr64, 2),
        "accuracy": "FP32 results within 1e-5 of the FP64 oracle and bit-identical alone vs in the mix "
                    "(tests/test_gpu_serving.py)",
    }


def run_accuracy_leg(L, synth, stream, n=MHD_N_LOWP, nsteps=MHD_STEPS):
    """Accuracy of the FP32 and BF16 storage paths of the 8-field system at 384^3 over 20 RK3
    steps, against the FP64 path of the same library (which matches the FP64 oracle within
    1e-12 at 256^3 over 20 steps, tests/test_gpu_full_size.py): after every step, per field,
    relative L2 and L-infinity error over the interior, and the drift of the mass
    sum exp(lnrho) dV.  Each low-precision state after k steps is one stencil_step(k) call from
    the initial state, as the benchmark runs it; the FP64 reference steps one RK3 step at a
    time (it carries no Kahan terms, so that is the same arithmetic)."""
    import torch
    f8 = synth.mhd_fields(n, seed=synth.SEED_MHD_LOWP)

    def plan(storage):
        par = L.mhd_params(n)
        compute = L.STENCIL_F64 if storage == L.STENCIL_F64 else L.STENCIL_F32
        p = L.Plan(3, (n, n, n), 3, 8, L.STENCIL_BC_PERIODIC, L.STENCIL_MHD8, storage, compute, params=par)
        a, b = p.alloc(), p.alloc()
        p.upload(a, f8)
        p.halo_fill(a)
        return p, a, b, par

    ref, ra, rb, par = plan(L.STENCIL_F64)
    vol = par.dx[0] * par.dx[1] * par.dx[2]
    low = {name: plan(st)[:3] for name, st in (("fp32", L.STENCIL_F32), ("bf16", L.STENCIL_BF16))}
    m0 = float(ref.norms(ra)[-1])
    out = {name: {"worst_rel_l2": [0.0] * 8, "worst_rel_linf": [0.0] * 8, "per_step_worst": []} for name in low}
    for k in range(1, nsteps + 1):
        ref.step(ra, rb, 1, stream)
        ra, rb = rb, ra
        rint = [ref.interior(t) for t in ra]
        for name, (p, a, b) in low.items():
            p.step(a, b, k, stream)
            worst = 0.0
            for q in range(8):
                got = p.interior(b[q]).double()
                d = got - rint[q]
                e2 = float(torch.linalg.vector_norm(d) / torch.linalg.vector_norm(rint[q]))
                ei = float(d.abs().max() / rint[q].abs().max())
                out[name]["worst_rel_l2"][q] = max(out[name]["worst_rel_l2"][q], e2)
                out[name]["worst_rel_linf"][q] = max(out[name]["worst_rel_linf"][q], ei)
                worst = max(worst, e2, ei)
            out[name]["per_step_worst"].append(round(worst, 8))
            if k == nsteps:
                m = float(p.norms(b)[-1])
                out[name]["mass_drift_after_20_steps"] = (m - m0) / m0
    out["fp64_mass_drift_after_20_steps"] = (float(ref.norms(ra)[-1]) - m0) / m0
    names = synth.MHD_FIELDS
    for name in low:
        for key in ("worst_rel_l2", "worst_rel_linf"):
            out[name][key] = {f: float(f"{v:.3e}") for f, v in zip(names, out[name][key])}
        out[name]["bound"] = 1e-5 if name == "fp32" else 1e-2
    for p, *_ in [(ref,)] + list(low.values()):
        p.close()
    del ra, rb, low
    torch.cuda.empty_cache()
    out["reference"] = ("the library's FP64 path at the same size (FP64 oracle parity within 1e-12 "
                        "in tests/test_gpu_full_size.py); mass = sum exp(lnrho) dV, drift relative to the "
                        "initial FP64 state; mass_volume = %.6e" % vol)
    return out


def cpu_baseline(seconds_target=10.0):
    """The FP64 oracle, as it stands, on the host cores: a bounded sample of the headline
    workload (256^3 heat field, a number of Euler steps chosen to take ~10 s)."""
    import oracle
    from paper_2406_08923_gb300 import synth
    n = HEAT_N
    f = synth.heat_field(n)
    h = 2 * np.pi / n
    t0 = time.perf_counter()
    oracle.diffusion(f, 0.1 * h * h, 1.0, (h, h, h), 1)
    t1 = time.perf_counter() - t0
    k = max(1, min(HEAT_STEPS, int(seconds_target / max(t1, 1e-3))))
    t0 = time.perf_counter()
    oracle.diffusion(f, 0.1 * h * h, 1.0, (h, h, h), k)
    dt = time.perf_counter() - t0
    cores = len(os.sched_getaffinity(0)) if hasattr(os, "sched_getaffinity") else os.cpu_count()
    threads = int(os.environ.get("OMP_NUM_THREADS", cores))
    return {"value": round(n ** 3 * k / dt / 1e6, 3), "unit": "Mcell-updates/s", "cores": threads,
            "kind": "oracle", "sample": f"256^3 FP64 heat field, {k} forward-Euler steps (of 100), "
                                        f"{dt:.1f} s wall on {threads} OpenMP threads"}


# ----------------------------------------------------------------------------- arms


def run_reference(args):
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return 0
    import oracle
    from paper_2406_08923_gb300 import synth
    n = HEAT_N
    f = synth.heat_field(n)
    h = 2 * np.pi / n
    per_step = 4  # Euler steps of the oracle per bench step (bounded sample of the 100-step job)
    for _ in range(args.warmup):
        oracle.diffusion(f, 0.1 * h * h, 1.0, (h, h, h), 1)
    t0 = time.perf_counter()
    for _ in range(args.steps):
        oracle.diffusion(f, 0.1 * h * h, 1.0, (h, h, h), per_step)
    dt = (time.perf_counter() - t0) / args.steps
    value = n ** 3 * per_step / dt / 1e6
    cores = len(os.sched_getaffinity(0)) if hasattr(os, "sched_getaffinity") else os.cpu_count()
    threads = int(os.environ.get("OMP_NUM_THREADS", cores))
    line = {
        "impl": "reference", "metric": "heat3d_256_fp64_mcell_updates_per_s", "value": round(value, 3),
        "unit": "Mcell-updates/s", "n_gpus": args.gpus, "steps": args.steps, "warmup": args.warmup,
        "ms_per_step": round(dt * 1e3, 3), "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "config": {"workload": "heat3d_r3_256^3_fp64_periodic_euler_dt0.1dx2_100steps",
                   "sample": f"{per_step} of the 100 Euler steps per bench step"},
        "cpu_baseline": {"value": round(value, 3), "unit": "Mcell-updates/s", "cores": threads, "kind": "oracle",
                         "sample": f"256^3 FP64 heat field, {per_step} Euler steps per bench step"},
        "e2e": {"value": round(value, 3), "unit": "Mcell-updates/s", "h2d_bytes_per_step": 0,
                "d2h_bytes_per_step": 0},
    }
    print(json.dumps(line), flush=True)
    return 0


def run_ours(args):
    import torch

    from paper_2406_08923_gb300 import _lib as L
    from paper_2406_08923_gb300 import synth

    rank, world, dist = _dist()
    L.load()
    dev = torch.cuda.current_device()
    stream = torch.cuda.current_stream()
    hbm_peak, hbm_src = _peaks()

    # ---- headline: 256^3 FP64 heat, 100 steps per bench step
    n = HEAT_N
    cells = n ** 3
    # the headline pins the variant its ncu capture was taken on (the autotuner's variants
    # are within ~2 % of each other for FP64, which is FP64-pipe bound)
    head = heat_job(L, synth, L.STENCIL_F64, n, HEAT_STEPS, args.warmup, 1, stream, with_e2e=False,
                    variant=HEADLINE_VARIANT)
    p = head["plan"]
    a, b = head["fields"]
    _barrier(dist)
    torch.cuda.synchronize()
    with Clocks(dev) as clk:
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        for _ in range(args.steps):
            p.step(a, b, HEAT_STEPS, stream)
        e1.record(stream)
        torch.cuda.synchronize()
    _barrier(dist)
    ms = e0.elapsed_time(e1) / args.steps
    ms = _max_over_ranks(ms, dist)
    clocks = clk.summary()
    value = weak_scaling_value(world, cells * HEAT_STEPS, ms / 1e3)

    # per-kernel average: job time minus the one input halo fill, over 100 passes
    ms_halo = _timed(lambda: p.halo_fill(a, stream), 20, stream)
    ms_kernel = (ms - ms_halo) / HEAT_STEPS
    flops_cell, bytes_cell = 38.0, 16.0
    achieved_tf = cells * flops_cell / (ms_kernel / 1e3) / 1e12
    achieved_gbs = cells * bytes_cell / (ms_kernel / 1e3) / 1e9

    # e2e through the public API with host buffers: pinned H2D of the padded input,
    # the 100-step job, D2H of the padded result, every step.
    nbytes = p.bytes_per_field
    h_in = torch.empty(a[0].numel(), dtype=a[0].dtype, pin_memory=True)
    h_out = torch.empty_like(h_in, pin_memory=True)
    h_in.copy_(a[0].cpu())
    d_in = p.alloc()

    def e2e():  # one C-ABI call: H2D of the input, the 100-step job, D2H of the result, sync
        p.step_host([h_in], [h_out], d_in, b, HEAT_STEPS, stream)

    e2e()
    ms_e2e = _max_over_ranks(_timed(e2e, max(3, args.steps // 2), stream), dist)

    extras = {}
    if not args.no_extras:
        extras = run_extras(L, synth, stream, hbm_peak, args)
        extras["diffusion_radius_sweep"] = run_radius_sweep(L, synth, stream, hbm_peak)
        extras["xcorr_maxfilter_radius_sweep"] = run_xcorr_radius_sweep(L, synth, stream, hbm_peak)
        if world == 1:
            extras["serving"] = run_serving_leg()

    line = {
        "metric": "heat3d_256_fp64_mcell_updates_per_s",
        "value": round(value, 3), "unit": "Mcell-updates/s", "n_gpus": world, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": round(ms, 4), "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "config": {"workload": "heat3d_r3_256^3_fp64_periodic_euler_dt0.1dx2_100steps",
                   "cells": cells, "euler_steps_per_bench_step": HEAT_STEPS,
                   "kernel_variant": head["variant"],
                   "l2": "inputs larger than L2 (2 x 145 MB padded FP64 fields streamed per pass)",
                   "parallelism": f"{world} independent grids (one per GPU)"},
        "roofline": _roof("hbm", achieved_gbs, hbm_peak, "GB/s",
                          traffic=_traffic("heat_f64", head["variant"]),
                          note=f"{hbm_src} copy bandwidth; 16 B per cell-update; the kernel is bound by issue "
                               "and latency of the integer pipe (64-bit fixed point), at "
                               f"{achieved_tf / FP64_PEAK_TFLOPS:.2f} times the FP64 pipe's 1.25 TFLOP/s "
                               "(38 flop per cell-update)"),
        "roofline_hbm": {"achieved": round(achieved_gbs, 1), "peak": hbm_peak, "unit": "GB/s",
                         "frac": round(achieved_gbs / hbm_peak, 4), "peak_source": hbm_src,
                         "bytes_per_cell": bytes_cell},
        "kernel_ms_avg": round(ms_kernel, 5), "halo_fill_ms": round(ms_halo, 5),
        "e2e": {"value": round(world * cells * HEAT_STEPS / (ms_e2e / 1e3) / 1e6, 3), "unit": "Mcell-updates/s",
                "h2d_bytes_per_step": nbytes, "d2h_bytes_per_step": nbytes,
                "call": "stencil_step_host (pinned host buffers in, 100-step job, host buffers out, stream sync)"},
        "gpu_launches": args.steps * (HEAT_STEPS + 1),
        "clocks": clocks,
        "per_stencil": extras,
    }
    if rank == 0 and world == 1 and not args.no_cpu:
        line["cpu_baseline"] = cpu_baseline()
    if rank == 0:
        print(json.dumps(line), flush=True)
    if dist is not None:
        dist.destroy_process_group()
    return 0


def run_zslab(args):
    """The headline job on one grid decomposed along z over the N ranks (strong scaling): each
    rank owns 256/N planes as a STENCIL_BC_PERIODIC_XY plan, and every Euler step first
    exchanges the 3-plane z halos with the neighbouring ranks (NCCL point-to-point; with one
    rank the slab wraps onto itself by a device copy).  Prints the same metric as the default
    run, with "scaling": "strong"."""
    import torch

    from paper_2406_08923_gb300 import _lib as L
    from paper_2406_08923_gb300 import synth
    from paper_2406_08923_gb300.zslab import ZSlabPlan
    rank, world, dist = _dist()
    L.load()
    stream = torch.cuda.current_stream()
    n = HEAT_N
    sp = ZSlabPlan(L.STENCIL_DIFFUSION, (n, n, n), L.STENCIL_F64, L.heat_params(n), rank, world)
    sp.plan.set_variant(HEADLINE_VARIANT)
    a, b = sp.alloc(), sp.alloc()
    sp.upload(a, [synth.heat_field(n)])
    for _ in range(args.warmup):
        sp.step(a, b, HEAT_STEPS, stream)
    _barrier(dist)
    torch.cuda.synchronize()
    dev = torch.cuda.current_device()
    with Clocks(dev) as clk:
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        for _ in range(args.steps):
            sp.step(a, b, HEAT_STEPS, stream)
        e1.record(stream)
        torch.cuda.synchronize()
    _barrier(dist)
    ms = _max_over_ranks(e0.elapsed_time(e1) / args.steps, dist)
    line = {"metric": "heat3d_256_fp64_mcell_updates_per_s", "value": round(n ** 3 * HEAT_STEPS / (ms / 1e3) / 1e6, 3),
            "unit": "Mcell-updates/s", "n_gpus": world, "steps": args.steps, "warmup": args.warmup,
            "ms_per_step": round(ms, 4), "higher_is_better": True, "scaling": "strong", "vs_baseline": None,
            "dtype": "f64", "data": "synthetic",
            "config": {"workload": "heat3d_r3_256^3_fp64_periodic_euler_dt0.1dx2_100steps",
                       "parallelism": f"z-slab decomposition of one grid over {world} rank(s), "
                                      f"{sp.z1 - sp.z0} planes on rank {rank}, 3-plane halo exchange per step",
                       "kernel_variant": sp.plan.variant()[2]},
            "gpu_launches": args.steps * HEAT_STEPS * 2, "clocks": clk.summary()}
    if rank == 0:
        print(json.dumps(line), flush=True)
    if dist is not None:
        dist.destroy_process_group()
    return 0


def run_extras(L, synth, stream, hbm_peak, args):
    out = {}
    w, r = 1, 3
    # 1D cross-correlation, 2^20 cells, 10 sweeps (L2-resident: no HBM claim)
    for name, dt in (("xcorr1d_int32_2^20_10sweeps", L.STENCIL_I32), ("xcorr1d_fp64_2^20_10sweeps", L.STENCIL_F64)):
        res = xcorr_job(L, synth, dt, w, 20, stream)
        out[name] = {"ms_per_job": round(res["ms_job"], 4), "ms_per_job_eager": round(res["ms_job_eager"], 4),
                     "timing": "CUDA-graph replay of stencil_step (eager: one ctypes call per job)",
                     "mcell_updates_per_s": round(XC_N * XC_SWEEPS / (res["ms_job"] / 1e3) / 1e6, 1),
                     "launches_per_job": 1, "bound": "l2 + launch latency (4-8 MiB working set)"}
        if dt == L.STENCIL_F64:
            # the 10 sweeps composed into one correlation of 61 weights: three integer
            # multiply-adds per tap, which bound this case
            ti = XC_N * (2 * XC_SWEEPS * 3 + 1) * 3 / (res["ms_job"] / 1e3) / 1e12
            out[name]["bound"] = "integer pipe (64-bit fixed point; 8 MiB working set, L2-resident)"
            out[name]["roofline"] = _roof("alu", ti, INT_PIPE_TINSTR, "Tinstr/s",
                                          note="183 multiply-adds of 32 x 32 + 64 bits per cell and job; 32 per "
                                               "clock and SM")
    # 3D heat, 256^3, 100 steps, FP32
    res = heat_job(L, synth, L.STENCIL_F32, HEAT_N, HEAT_STEPS, w, r, stream)
    cells = HEAT_N ** 3
    gbs = cells * 8.0 / (res["ms_kernel"] / 1e3) / 1e9
    out["heat3d_256_fp32_100steps"] = {
        "ms_per_job": round(res["ms_job"], 4), "kernel_ms_avg": round(res["ms_kernel"], 5),
        "mcell_updates_per_s": round(cells * HEAT_STEPS / (res["ms_job"] / 1e3) / 1e6, 1),
        "variant": res["variant"], "launches_per_job": res["launches_per_job"],
        "zchunk_mode": res["plan"].autotune_status()[1],
        "roofline": _roof("hbm", gbs, hbm_peak, "GB/s",
                          traffic=_traffic("heat_f32", res["variant"], res["plan"].autotune_status()[1]),
                          note="8 B/cell-update algorithmic; traffic = ncu dram bytes/launch")}
    res["plan"].close()
    # 3D heat FP32 at 512^3: the two 540 MB fields far exceed the 126 MB L2
    n5 = 2 * HEAT_N
    res = heat_job(L, synth, L.STENCIL_F32, n5, HEAT_STEPS // 4, w, r, stream)
    cells5 = n5 ** 3
    gbs = cells5 * 8.0 / (res["ms_kernel"] / 1e3) / 1e9
    out["heat3d_512_fp32_25steps"] = {
        "ms_per_job": round(res["ms_job"], 4), "kernel_ms_avg": round(res["ms_kernel"], 5),
        "mcell_updates_per_s": round(cells5 * (HEAT_STEPS // 4) / (res["ms_job"] / 1e3) / 1e6, 1),
        "variant": res["variant"], "launches_per_job": res["launches_per_job"],
        "zchunk_mode": res["plan"].autotune_status()[1],
        "roofline": _roof("hbm", gbs, hbm_peak, "GB/s",
                          traffic=_traffic("heat_f32_512", res["variant"], res["plan"].autotune_status()[1]),
                          note="8 B/cell-update algorithmic; traffic = ncu dram bytes/launch")}
    res["plan"].close()
    # fused 8-field MHD, 256^3 FP64, 20 RK3 steps
    cells = MHD_N ** 3
    res = mhd_job(L, synth, L.STENCIL_F64, MHD_N, MHD_STEPS, w, 1, stream)
    # algorithmic flops per cell-substep (Eqs. A1-A4 + RK3) against the FP64 FMA peak; the
    # FP64 pipe's utilisation (instructions the kernel executes, ncu) beside it
    tf = cells * MHD_FLOPS_PER_CELL_SUBSTEP / (res["ms_substep"] / 1e3) / 1e12
    ips = cells * MHD_F64_INSTR / (res["ms_substep"] / 1e3)
    out["mhd8_256_fp64_20steps"] = {
        "ms_per_job": round(res["ms_job"], 3), "ms_per_substep": round(res["ms_substep"], 4),
        "mcell_substep_updates_per_s": round(cells / (res["ms_substep"] / 1e3) / 1e6, 1),
        "variant": res["variant"], "finite": res["finite"], "mass": res["mass"],
        "roofline": _roof("alu", tf, FP64_PEAK_TFLOPS, "TFLOP/s",
                          note=f"{MHD_FLOPS_PER_CELL_SUBSTEP:.2f} algorithmic flop per cell-substep "
                               "(tests/mhd_flops.py; an FMA is 2 flop) against the FP64 FMA peak "
                               "2 x 2 flop/clk/SM x 152 SMs x 2.07 GHz; the linear differences, 600 "
                               "of the flop, run in fixed point on the integer pipe"),
        "fp64_pipe": {"instr_per_cell_substep": MHD_F64_INSTR, "achieved_tinstr_s": round(ips / 1e12, 4),
                      "peak_tinstr_s": round(FP64_PIPE_TINSTR, 4),
                      "utilisation": round(ips / 1e12 / FP64_PIPE_TINSTR, 4)},
        "paper_ideal_hbm_frac": round(cells * 128.0 / (res["ms_substep"] / 1e3) / 1e9 / hbm_peak, 4)}
    # norms (a7): the two-pass FP64 reduction over the 8 fields of the 256^3 state, one read of
    # each interior (8 B per cell and field), through the allocation-free entry point so that a
    # call is one device-side job (stencil_field_norms also copies to the host and synchronises)
    import torch
    mp, fields = res["plan"], res["fields"]
    nout = torch.empty(3 * 8 + 1, dtype=torch.float64, device="cuda")
    vol = mp.params.dx[0] * mp.params.dx[1] * mp.params.dx[2]
    norm_call = lambda: L.stencil_field_norms_noalloc(fields, mp.storage, mp.dims, mp.padded, mp.origin, vol, nout,
                                                      stream)
    norm_call()
    ms_norm = _timed(norm_call, 20, stream)
    gbs = cells * 8 * 8 / (ms_norm / 1e3) / 1e9
    out["norms_8x256_fp64"] = {
        "ms_per_call": round(ms_norm, 4), "launches_per_call": 2,
        "roofline": _roof("hbm", gbs, hbm_peak, "GB/s",
                          note="one read of 8 fields x 256^3 interior cells x 8 B per call (sum, sum f^2, "
                               "max |f|, mass sum exp(lnrho)); 2 launches")}
    res["plan"].close()
    # fused 8-field MHD, 384^3 FP32 / BF16 storage, Kahan-compensated RK
    cells = MHD_N_LOWP ** 3
    for name, st, bpc in (("mhd8_384_fp32_20steps", L.STENCIL_F32, 4), ("mhd8_384_bf16_20steps", L.STENCIL_BF16, 2)):
        res = mhd_job(L, synth, st, MHD_N_LOWP, MHD_STEPS, w, 1, stream)
        # per cell-substep: f_in, f_out, w r/w, c r/w over 8 fields (avg over the 3 substeps)
        avg_vals = 8 * (1 + 1 + (1 + 2 + 1) / 3.0 + 2)
        gbs = cells * avg_vals * bpc / (res["ms_substep"] / 1e3) / 1e9
        zm = res["plan"].autotune_status()[1]
        out[name] = {"ms_per_job": round(res["ms_job"], 3), "ms_per_substep": round(res["ms_substep"], 4),
                     "mcell_substep_updates_per_s": round(cells / (res["ms_substep"] / 1e3) / 1e6, 1),
                     "variant": res["variant"], "zchunk_mode": zm, "finite": res["finite"], "mass": res["mass"],
                     "roofline": _roof("hbm", gbs, hbm_peak, "GB/s",
                                       traffic=_traffic("mhd_f32" if st == L.STENCIL_F32 else "mhd_bf16",
                                                        res["variant"], zm),
                                       note=f"{avg_vals:.1f} values x {bpc} B per cell-substep (mean of the 3 "
                                            "RK substeps); traffic = ncu dram bytes per launch, mean of the 3 "
                                            "substeps")}
        res["plan"].close()
    # MHD 384^3 accuracy: FP32 / BF16 storage against the FP64 path, every step of 20
    out["mhd8_384_accuracy_20steps"] = run_accuracy_leg(L, synth, stream)
    return out


CASES = {
    # name: (kind, storage, default n, steps per job)
    "heat_f64": ("heat", 1, HEAT_N, HEAT_STEPS),
    "heat_f32": ("heat", 2, HEAT_N, HEAT_STEPS),
    "mhd_f64": ("mhd", 1, MHD_N, 1),
    "mhd_f32": ("mhd", 2, MHD_N_LOWP, 1),
    "mhd_bf16": ("mhd", 3, MHD_N_LOWP, 1),
    "xcorr_i32": ("xcorr", 0, XC_N, XC_SWEEPS),
    # radius sweep workloads (2^24 cells; --radius picks r)
    "xcorr1d_f32": ("xcorr_r", 2, 1 << 24, 1),
    "xcorr1d_f64": ("xcorr_r", 1, 1 << 24, 1),
    "maxfilter_f32": ("maxfilter", 2, 1 << 24, 1),
    "heat2d_f32": ("heat2d", 2, 4096, 4),
    # the norms of the 8-field state (with the mass), through the allocation-free entry point
    "norms_f64": ("norms", 1, MHD_N, 1),
}


def run_case(args):
    """One workload, fixed kernel variant, `warmup` + `steps` jobs; prints one short JSON line."""
    import torch

    from paper_2406_08923_gb300 import _lib as L
    from paper_2406_08923_gb300 import synth
    kind, storage, n0, steps = CASES[args.case]
    n = args.n or n0
    steps = args.job_steps or steps
    stream = torch.cuda.current_stream()
    job = None
    if kind == "heat":
        par = L.heat_params(n)
        p = L.Plan(3, (n, n, n), 3, 1, L.STENCIL_BC_PERIODIC, L.STENCIL_DIFFUSION, storage, storage, params=par)
        a, b = p.alloc(), p.alloc()
        p.upload(a, [synth.heat_field(n)])
    elif kind == "norms":
        par = L.mhd_params(n)
        p = L.Plan(3, (n, n, n), 3, 8, L.STENCIL_BC_PERIODIC, L.STENCIL_MHD8, storage, storage, params=par)
        a = p.alloc()
        p.upload(a, synth.mhd_fields(n))
        nout = torch.empty(3 * 8 + 1, dtype=torch.float64, device="cuda")
        vol = par.dx[0] * par.dx[1] * par.dx[2]
        job = lambda: L.stencil_field_norms_noalloc(a, p.storage, p.dims, p.padded, p.origin, vol, nout, stream)
    elif kind == "mhd":
        par = L.mhd_params(n)
        compute = L.STENCIL_F64 if storage == L.STENCIL_F64 else L.STENCIL_F32
        p = L.Plan(3, (n, n, n), 3, 8, L.STENCIL_BC_PERIODIC, L.STENCIL_MHD8, storage, compute, params=par)
        a, b = p.alloc(), p.alloc()
        p.upload(a, synth.mhd_fields(n))
    elif kind == "heat2d":
        r = args.radius or 3
        shape = (n, n)
        p = L.Plan(2, shape, r, 1, L.STENCIL_BC_PERIODIC, L.STENCIL_DIFFUSION, storage, storage,
                   params=L.heat_params(shape))
        a, b = p.alloc(), p.alloc()
        p.upload(a, [synth.uniform(2406089237, 2, n * n, -1.0, 1.0).reshape(shape)])
    elif kind in ("xcorr_r", "maxfilter"):
        r = args.radius if args.radius is not None else 64
        g = None
        if kind == "xcorr_r":
            g = synth.uniform(2406089239, 10 + r, 2 * r + 1, 0.0, 1.0)
            g = g / g.sum()
        p = L.Plan(1, (n,), r, 1, L.STENCIL_BC_PERIODIC,
                   L.STENCIL_XCORR if kind == "xcorr_r" else L.STENCIL_MAXFILTER, storage, storage, coeffs=g)
        a, b = p.alloc(), p.alloc()
        p.upload(a, [synth.uniform(2406089239, 1, n, 0.0, 1.0)])
    else:
        data, g = synth.xcorr_int32(n)
        p = L.Plan(1, (n,), 3, 1, L.STENCIL_BC_PERIODIC, L.STENCIL_XCORR, storage, storage, coeffs=g)
        a, b = p.alloc(), p.alloc()
        p.upload(a, [data])
    if job is None:
        p.set_variant(args.variant)
        if args.zmode:
            p.set_zmode(args.zmode)
        job = lambda: p.step(a, b, steps, stream)
    for _ in range(args.warmup):
        job()
    ms = _timed(job, args.steps, stream)
    p.sync()
    print(json.dumps({"case": args.case, "n": n, "radius": args.radius, "steps_per_job": steps,
                      "variant": p.variant()[2], "zmode": args.zmode, "ms_per_job": round(ms, 4)}), flush=True)
    return 0


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=10)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=("ours", "reference"))
    ap.add_argument("--no-extras", action="store_true", help="headline workload only")
    ap.add_argument("--no-cpu", action="store_true", help="skip the cpu_baseline leg")
    ap.add_argument("--case", default=None, choices=sorted(CASES),
                    help="run one workload only (no autotune), e.g. for an ncu capture")
    ap.add_argument("--n", type=int, default=None, help="grid size for --case")
    ap.add_argument("--zmode", type=int, default=0, help="z-chunk mode for --case (3D streaming kernels)")
    ap.add_argument("--variant", type=int, default=0, help="kernel variant for --case")
    ap.add_argument("--job-steps", type=int, default=None, help="steps per job for --case")
    ap.add_argument("--radius", type=int, default=None, help="stencil radius for the 1D / 2D --case workloads")
    ap.add_argument("--serving", action="store_true", help="serving configuration only (one JSON line)")
    ap.add_argument("--radius-sweep", action="store_true", help="diffusion radius sweep only (one JSON line)")
    ap.add_argument("--zslab", action="store_true",
                    help="the headline job on one grid decomposed along z over the ranks (strong scaling)")
    args = ap.parse_args()
    if args.warmup < 3:
        args.warmup = 3
    if args.impl == "reference":
        return run_reference(args)
    if args.case:
        return run_case(args)
    if args.zslab:
        return run_zslab(args)
    if args.radius_sweep:
        import torch

        from paper_2406_08923_gb300 import _lib as L
        from paper_2406_08923_gb300 import synth
        L.load()
        st, hbm = torch.cuda.current_stream(), _peaks()[0]
        res = run_radius_sweep(L, synth, st, hbm)
        res1 = run_xcorr_radius_sweep(L, synth, st, hbm)
        print(json.dumps({"metric": "radius_sweep_ms_per_step", "diffusion": res, "xcorr_maxfilter_1d": res1}),
              flush=True)
        return 0
    if args.serving:
        print(json.dumps({"metric": "serving_p50_p99_latency_and_mcell_updates_per_s", "serving": run_serving_leg()}),
              flush=True)
        return 0
    return run_ours(args)


if __name__ == "__main__":
    sys.exit(main())
