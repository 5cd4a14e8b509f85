#!/usr/bin/env python
"""Benchmark of the matrix-free diffusion action (paper Section 2, A_L u_L) on one GB300.

Workload (default): 64^3-element hexahedral mesh of the unit cube, interior vertices perturbed by up
to 0.1h (seed 0), p = 7 on GLL nodes with collocated GLL quadrature, six stored symmetric geometric
factors with k = 1 + 0.5 sin(2 pi x) sin(2 pi y) sin(2 pi z), x ~ U[-1, 1]: 90,518,849 DOFs.
A step is one FP64 application y = A x of the whole fused path (gather, contractions, pointwise
quadrature operator, transposed contractions, atomic-free scatter); inputs are resident in HBM and
far larger than L2 (x 0.72 GB, quadrature data 6.4 GB), so no L2 flush is needed.

Beside the headline it measures the FP32-arithmetic operator (FP32 and BF16 quadrature data), the
double-float FP64-accurate operator, the end-to-end host-buffer call (ceed_apply_host), 100
Jacobi-PCG iterations, CG time to a relative residual of 1e-10 in FP64, with mixed-precision
refinement and with reliable updates, p-multigrid CG, the batched mixed-order apply, the adjoint,
the tetrahedral and hp operators, and the CPU oracle on a bounded sample; --cg-c4 1 adds CG on
80^3 elements (176.6M DOFs).

--impl reference times the CPU oracle (dense per-element quadrature, no sum factorization) on the
host cores, on a bounded sample of the same workload per step.
"""
from __future__ import annotations

import argparse
import json
import os
import subprocess
import sys
import threading
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

import numpy as np  # noqa: E402

import synthetic  # noqa: E402

METRIC = "diffusion apply GDOF/s at p=7 (FP64 vs mixed), % HBM roofline, CG time-to-1e-10"
FP64_NOMINAL_TFLOPS = 1.25      # GB300 dense FP64 (nominal table), reported beside the measured peak
# DRAM bytes (read + write) per launch of each apply kernel variant, from ncu captures of the current
# kernels on the 48^3 mesh, scaled by elements to a 64^3 colour launch; keyed by kernel and variant
# (a variant without a capture reports null).
PROFILED_TRAFFIC_PER_LAUNCH = {
    # DRAM bytes (read + write) of one colour launch at 48^3 (13,824 elements), scaled by elements to
    # a 64^3 launch (32,768): profiles/apply_kernel_variants_traffic_p7_48cube.md
    "apply_kernel<8,8,DIFFUSION,double,double,stage=0>[ne=1]": 622.10e6 * 32768 / 13824,
    "apply_kernel<8,8,DIFFUSION,double,double,stage=0>[ne=2]": 618.94e6 * 32768 / 13824,
    "apply_kernel<8,8,DIFFUSION,double,double,stage=0>[ne=4]": 614.67e6 * 32768 / 13824,
    "apply_kernel<8,8,DIFFUSION,double,double,stage=1>[ne=1]": 570.23e6 * 32768 / 13824,
    "apply_kernel<8,8,DIFFUSION,double,double,stage=1>[ne=2]": 570.97e6 * 32768 / 13824,
    "apply_kernel<8,8,DIFFUSION,double,double,stage=1>[ne=4]": 571.53e6 * 32768 / 13824,
    "apply_kernel<8,8,DIFFUSION,DF,DF,stage=0>[ne=1]": 570.61e6 * 32768 / 13824,
    "apply_kernel<8,8,DIFFUSION,DF,DF,stage=0>[ne=2]": 570.52e6 * 32768 / 13824,
    # profiles/df_apply_kernel_p7_48cube_ncu.md: 504.33 MB read + 68.59 MB written
    "apply_kernel<8,8,DIFFUSION,DF,DF,stage=0>[ne=4]": 572.92e6 * 32768 / 13824,
    # profiles/brick_kernel_p7_48cube_ncu.md: 279.28 MB read + 43.38 MB written per 3,456-brick launch
    "brick_kernel<8,8,DIFFUSION,float,float,stage=0>": 322.66e6 * 32768 / 13824,
    # same file, BF16 quadrature data: 193.56 MB read + 38.23 MB written
    "brick_kernel<8,8,DIFFUSION,float,bf16,stage=0>": 231.79e6 * 32768 / 13824,
}
# DRAM bytes (read + write) of one launch of the tensor-core tetrahedral kernel on the 48^3 x 6
# degree-4 workload (profiles/nt_tc_kernel_p4_tet48_ncu.md): 2143.84 MB read + 90.39 MB written
NT_TC_TRAFFIC_PER_LAUNCH = 2234.23e6
WORKLOADS = {
    "c2": dict(N=64, p=7),      # the diffusion workload named by element count
    "c2a": dict(N=40, p=7),     # 22.19M DOFs: the DOF count quoted for the same workload
    "c4": dict(N=80, p=7),      # the mixed-precision CG workload
    "w48": dict(N=48, p=7),     # profiling size: one colour launch moves more than L2, a few GB on the device
    "w32": dict(N=32, p=7),     # profiling size of the fused CG iteration (11.4M DOFs, about 2 GB on the device)
}


def cost_per_element(p):
    """Section 2: 7 (p+1)^3 reads and 12 (p+1)^4 + 15 (p+1)^3 flops per element (collocated)."""
    P = p + 1
    return 7 * P ** 3, 12 * P ** 4 + 15 * P ** 3


def algorithmic_bytes(m, qbytes, geo=False):
    """x read + y write once per L-node (8 B each), the quadrature data, the int32 restriction.

    Stored geometry: 6 factors per point.  On-the-fly geometry (geo): 24 FP32 map coefficients per
    element and one w k value per point."""
    nd = (m.p + 1) ** 3
    qd = (24 * 4 + qbytes * nd) * m.n_elem if geo else 6 * qbytes * m.n_elem * nd
    return 16 * m.n_ldof + qd + 4 * m.n_elem * nd


def fp64_pipe_flops(p, gauss=False):
    """Flops per element (2 per instruction) that the FP64 diffusion operator leaves on the FP64 pipe.

    Lines of 6 to 8 points (7 or 8 with Gauss quadrature) run their 1D passes as integer slices on the tensor cores:
    the 3 x 3 product at a point (9 instructions) and the sum of the three directions (3) stay.  Other lines:
    the paper's cost model (the even-odd operators execute about 0.8 of it)."""
    q = p + 2 if gauss else p + 1
    if (7 if gauss else 6) <= q <= 8:
        return 24 * q ** 3
    return 24 * (p + 1) ** 4 + 15 * q ** 3 if gauss else cost_per_element(p)[1]


def load_peaks():
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as f:
            d = json.load(f)
        return float(d["hbm_gbs"]), "measured"
    except Exception:
        return 6800.0, "fallback"


class ClockSampler:
    """nvidia-smi samples of SM clock and throttle reasons while the timed region runs."""

    Q = ("clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.hw_slowdown,"
         "clocks_event_reasons.hw_thermal_slowdown,clocks_event_reasons.sw_thermal_slowdown,"
         "clocks_event_reasons.sw_power_cap")

    def __init__(self, index=0, period_ms=100, first_sample_s=5.0):
        self.index, self.samples, self.proc = index, [], None
        self.period_ms, self.first_sample_s = period_ms, first_sample_s

    def __enter__(self):
        try:
            self.proc = subprocess.Popen(["nvidia-smi", "-i", str(self.index), f"--query-gpu={self.Q}",
                                          "--format=csv,noheader,nounits", "-lms", str(self.period_ms)],
                                         stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.thread = threading.Thread(target=self._read, daemon=True)
            self.thread.start()
            # nvidia-smi takes a while to start: wait for its first line, so that the region that
            # follows (warm-up and timed steps, all under load) is sampled from its start
            t0 = time.perf_counter()
            while not self.samples and self.proc.poll() is None and time.perf_counter() - t0 < self.first_sample_s:
                time.sleep(0.01)
            self.samples.clear()
        except Exception:
            self.proc = None
        return self

    def _read(self):
        for line in self.proc.stdout:
            parts = [s.strip() for s in line.split(",")]
            if len(parts) >= 7:
                self.samples.append(parts)

    def __exit__(self, *exc):
        if self.proc:
            self.proc.terminate()
            try:
                self.proc.wait(timeout=5)
            except Exception:
                self.proc.kill()

    def summary(self):
        if not self.samples:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["unavailable"]}
        sm = [float(s[0]) for s in self.samples if s[0].replace(".", "").isdigit()]
        mx = [float(s[1]) for s in self.samples if s[1].replace(".", "").isdigit()]
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        reasons = sorted({names[k] for s in self.samples for k in range(4) if s[3 + k].lower() == "active"})
        return {"sm_mhz": float(np.median(sm)) if sm else None, "sm_max_mhz": max(mx) if mx else None,
                "reasons": reasons, "samples": len(self.samples)}


def oracle_sample_rate(m, n_elem_sample, seed=1):
    """CPU oracle: dense FP64 diffusion action on the first n elements; returns (DOF/s, seconds, threads)."""
    from oracle import fem
    sp_ = fem.Space(m.p, "gll")
    sel = np.arange(n_elem_sample)
    G = fem.qdata_diffusion(sp_, m.vertices[sel], "sine")
    x = synthetic.uniform(m.n_ldof, seed=seed)
    t0 = time.perf_counter()
    fem.apply(sp_, m.elem_dofs[sel], G, x, fem.DIFFUSION)
    dt = time.perf_counter() - t0
    dof_per_elem = m.n_ldof / m.n_elem
    return n_elem_sample * dof_per_elem / dt, dt


def blas_threads():
    try:
        from threadpoolctl import threadpool_info
        n = [i.get("num_threads", 0) for i in threadpool_info() if i.get("user_api") == "blas"]
        if n:
            return max(n)
    except Exception:
        pass
    return os.cpu_count()


def dist_env():
    ws = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return ws, rank, local


def max_over_ranks(value: float, ws: int, device) -> float:
    """The largest of the ranks' values (the job's time is its slowest replica's); identity at N = 1."""
    if ws <= 1:
        return value
    import torch
    import torch.distributed as dist
    t = torch.tensor([value], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def whole_job_rate(units_per_rank: float, ws: int, ms: float, scale: float = 1e-6) -> float:
    """Units all ranks processed per millisecond x scale (GDOF/s for DOFs with the default scale):
    every replica processes the same units, and ms is the max over ranks."""
    return ws * units_per_rank / ms * scale


def run_reference(args):
    ws, rank, _ = dist_env()
    if rank != 0:
        return
    wl = WORKLOADS[args.workload]
    m = synthetic.cube_mesh(wl["N"], wl["p"], seed=0)
    n_sample = args.ref_sample
    times = []
    for it in range(args.warmup + args.steps):
        rate, dt = oracle_sample_rate(m, n_sample, seed=1 + it)
        if it >= args.warmup:
            times.append(dt)
    dof = n_sample * m.n_ldof / m.n_elem
    value = dof * len(times) / sum(times) / 1e9
    line = {
        "impl": "reference", "metric": METRIC, "value": value, "unit": "GDOF/s", "n_gpus": ws,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1e3 * sum(times) / len(times),
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "config": {"workload": f"diffusion apply, {wl['N']}^3 perturbed hexes, p={wl['p']}, GLL collocated",
                   "n_ldof": m.n_ldof, "sample_elements_per_step": n_sample},
        "cpu_baseline": {"value": value, "unit": "GDOF/s", "cores": blas_threads(), "kind": "oracle",
                         "sample": f"{n_sample} of {m.n_elem} elements per step (dense per-element FP64 "
                                   f"quadrature, numpy), rate scaled to DOFs by n_ldof/n_elem"},
        "e2e": {"value": value, "unit": "GDOF/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }
    print(json.dumps(line), flush=True)


def run_profile(args):
    """Three applies of one precision on the chosen workload (for ncu captures of the apply kernel)."""
    import torch
    import paper_2109_05072_gb300 as ceed
    wl = WORKLOADS[args.workload]
    m = synthetic.cube_mesh(wl["N"], wl["p"], seed=0)
    mesh = ceed.ceed_setup_mesh(m.n_elem, m.n_ldof, wl["p"], torch.from_numpy(m.elem_dofs).cuda(),
                                torch.from_numpy(m.vertices).cuda(), torch.from_numpy(m.boundary).cuda())
    prec = {"f64": ceed.CEED_F64, "f32": ceed.CEED_F32, "bf16": ceed.CEED_BF16, "f64df": ceed.CEED_F64_DF}[args.profile]
    qd = ceed.alloc_qdata(mesh, ceed.CEED_OP_DIFFUSION, prec)
    ceed.ceed_build_qdata(mesh, ceed.CEED_OP_DIFFUSION, ceed.CEED_COEFF_SINE, None, prec, qd)
    x = torch.from_numpy(synthetic.uniform(m.n_ldof, seed=1)).cuda()
    y = torch.empty_like(x)
    if args.variant:
        ne, stage = (int(v) for v in args.variant.split(","))
        ceed.ceed_set_apply_variant(mesh, ceed.CEED_OP_DIFFUSION, prec, ne, stage)
    for _ in range(3):
        ceed.ceed_apply_diffusion(mesh, qd, prec, x, y)
    torch.cuda.synchronize()
    print(json.dumps({"profile": args.profile, "workload": args.workload, "n_ldof": m.n_ldof,
                      "colors": mesh.n_colors, "variant": args.variant}))


def run_profile_cg(args):
    """A short mixed-precision (FP32 operator, reliable updates) CG on the chosen workload: two fused
    launches of 10 iterations each (for ncu captures of the fused PCG iteration kernel)."""
    import torch
    import paper_2109_05072_gb300 as ceed
    wl = WORKLOADS[args.workload]
    m = synthetic.cube_mesh(wl["N"], wl["p"], seed=0)
    mesh = ceed.ceed_setup_mesh(m.n_elem, m.n_ldof, wl["p"], torch.from_numpy(m.elem_dofs).cuda(),
                                torch.from_numpy(m.vertices).cuda(), torch.from_numpy(m.boundary).cuda())
    q64 = ceed.alloc_qdata(mesh, ceed.CEED_OP_DIFFUSION, ceed.CEED_F64)
    ceed.ceed_build_qdata(mesh, ceed.CEED_OP_DIFFUSION, ceed.CEED_COEFF_SINE, None, ceed.CEED_F64, q64)
    q32 = ceed.alloc_qdata(mesh, ceed.CEED_OP_DIFFUSION, ceed.CEED_F32)
    ceed.ceed_build_qdata(mesh, ceed.CEED_OP_DIFFUSION, ceed.CEED_COEFF_SINE, None, ceed.CEED_F32, q32)
    b = torch.empty(m.n_ldof, dtype=torch.float64, device="cuda")
    ceed.ceed_manufactured_rhs(mesh, ceed.CEED_COEFF_SINE, b, flags=ceed.CEED_APPLY_DIRICHLET)
    x = torch.empty_like(b)
    st, rep = ceed.ceed_cg_solve(mesh, q64, ceed.CEED_F64, b, x, mode=ceed.CEED_CG_MIXED_RELIABLE, tol=1e-10,
                                 max_iter=20, op=ceed.CEED_OP_DIFFUSION, qdata_lo=q32, prec_lo=ceed.CEED_F32,
                                 separate_kernels=args.cg_separate, raise_on_error=False)
    print(json.dumps({"profile": "cg", "workload": args.workload, "n_ldof": m.n_ldof, "status": st, **rep}))


def _time_cuda(fn, steps, warmup):
    import torch
    for _ in range(warmup):
        fn()
    torch.cuda.synchronize()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record()
    for _ in range(steps):
        fn()
    e1.record()
    torch.cuda.synchronize()
    return e0.elapsed_time(e1) / steps


def batched_model_flops(p, N):
    """Section 2 cost model for one column of an N^3 mesh of order p with q = p + 2 Gauss points: the
    contraction term doubled for the interpolation passes (2 x 12 P^4) plus 15 Q^3 pointwise flops."""
    P, Q = p + 1, p + 3
    return N ** 3 * (24 * P ** 4 + 15 * Q ** 3)


def run_batched(ceed, dev, args, peaks=None, nrhs_list=(1, 4, 8, 16), steps=5, prec=None):
    """Three independent meshes of order 3, 5, 7 (Gauss q = p+2: 5, 7, 9 points) on 48^3, 40^3, 32^3
    elements, 3-component diffusion, FP64, applied by one persistent launch replayed from a CUDA graph."""
    import torch
    prec = ceed.CEED_F64 if prec is None else prec
    specs = [(3, 48), (5, 40), (7, 32)]
    meshes, qds, nodes = [], [], []
    for p, N in specs:
        m = synthetic.cube_mesh(N, p, seed=0)
        mesh = ceed.ceed_setup_mesh(m.n_elem, m.n_ldof, p, torch.from_numpy(m.elem_dofs).to(dev),
                                    torch.from_numpy(m.vertices).to(dev), None, q_rule=ceed.CEED_QRULE_GAUSS, ncomp=3)
        qd = ceed.alloc_qdata(mesh, ceed.CEED_OP_DIFFUSION, prec, dev)
        ceed.ceed_build_qdata(mesh, ceed.CEED_OP_DIFFUSION, ceed.CEED_COEFF_SINE, None, prec, qd)
        meshes.append(mesh)
        qds.append(qd)
        nodes.append(m.n_ldof)
    out = {"meshes": [f"p={p}, {N}^3, Gauss q={p + 2}, n_ldof={n}" for (p, N), n in zip(specs, nodes)],
           "ncomp": 3, "dtype": "f64" if prec == ceed.CEED_F64 else "f32x2 (double-float, FP64-accurate)", "runs": [],
           "model": "per element and column 24 P^4 + 15 Q^3 flops (Section 2 model, contraction term doubled "
                    "for q = p + 2); fp64_frac: what is left of that on the FP64 pipe (p = 5 runs its 1D passes on the "
                    "tensor cores) against the measured FP64 FMA rate"}
    for nrhs in nrhs_list:
        xs = [torch.from_numpy(synthetic.uniform(n * 3 * nrhs, seed=7 + k)).to(dev) for k, n in enumerate(nodes)]
        ys = [torch.empty_like(x) for x in xs]
        batch = ceed.ceed_batch_create(meshes, qds, prec, ceed.CEED_OP_DIFFUSION, xs, ys, nrhs=nrhs)
        ceed.ceed_batch_autotune(batch)
        threads, stage, grid = ceed.ceed_batch_info(batch)
        ms = _time_cuda(lambda: ceed.ceed_batch_apply(batch), steps, 3)
        ceed.ceed_batch_status(batch)
        dofs = sum(nodes) * 3 * nrhs
        flops = sum(batched_model_flops(p, N) for p, N in specs) * 3 * nrhs
        row = {"nrhs": nrhs, "ms_per_apply": ms, "gdofs": dofs / ms / 1e6, "threads": threads,
               "tma_staging": stage, "grid": grid, "launches_per_apply": 1, "model_tflops": flops / ms / 1e9}
        if peaks and peaks.get("f64") and prec == ceed.CEED_F64:
            left = sum(fp64_pipe_flops(p, gauss=True) * N ** 3 for p, N in specs) * 3 * nrhs
            row["fp64_frac"] = left / ms / 1e9 / peaks["f64"]["tflops"]
        out["runs"].append(row)
        batch.close()
        del xs, ys
        torch.cuda.empty_cache()
    for mesh in meshes:
        mesh.close()
    return out


def run_adjoint(ceed, dev, args):
    """Forward A(k) x and the fused adjoint (dL/dx, dL/dk) with a lognormal per-point k, p = 4 and 8 on
    32^3 elements (GLL collocated), geometry stored vs recomputed from the vertices, and with stored
    geometry in the FP64-accurate double-float arithmetic."""
    import torch
    out = []
    for p in (4, 8):
        m = synthetic.cube_mesh(32, p, seed=0)
        mesh = ceed.ceed_setup_mesh(m.n_elem, m.n_ldof, p, torch.from_numpy(m.elem_dofs).to(dev),
                                    torch.from_numpy(m.vertices).to(dev), None)
        nq = (p + 1) ** 3
        k = torch.from_numpy(synthetic.lognormal(m.n_elem * nq, seed=3, sigma=0.5)).to(dev)
        x = torch.from_numpy(synthetic.uniform(m.n_ldof, seed=4)).to(dev)
        r = torch.from_numpy(synthetic.uniform(m.n_ldof, seed=5)).to(dev)
        y = torch.empty_like(x)
        dLdk = torch.empty_like(k)
        geo = ceed.alloc_qdata(mesh, ceed.CEED_OP_DIFFUSION, ceed.CEED_F64, dev)
        ceed.ceed_build_geometry(mesh, geo)
        row = {"p": p, "mesh": "32^3", "n_ldof": m.n_ldof, "n_qpts": m.n_elem * nq}
        for name, g, fl in (("stored", geo, 0), ("recomputed", None, 0),
                            ("stored_f64_df", geo, ceed.CEED_APPLY_F64_DF)):
            ms_f = _time_cuda(lambda: ceed.ceed_apply_diffusion_k(mesh, k, g, x, y, flags=fl), 5, 3)
            ms_a = _time_cuda(lambda: ceed.ceed_apply_diffusion_adjoint(mesh, k, g, x, r, y, dLdk, flags=fl), 5, 3)
            row[name] = {"forward_ms": ms_f, "adjoint_ms": ms_a, "forward_gdofs": m.n_ldof / ms_f / 1e6,
                         "adjoint_gdofs": m.n_ldof / ms_a / 1e6}
        out.append(row)
        mesh.close()
        del geo, k, x, r, y, dLdk
        torch.cuda.empty_cache()
    return out


def run_cg_c4(ceed, dev, args):
    """CG to a true relative residual of 1e-10 on 80^3 elements, p = 7 (176,558,481 DOFs): FP64
    Jacobi-PCG, mixed refinement and reliable updates with the FP32 operator; the mixed solutions'
    difference from the FP64 solution is reported."""
    import torch
    wl = WORKLOADS["c4"]
    m = synthetic.cube_mesh(wl["N"], wl["p"], seed=0)
    mesh = ceed.ceed_setup_mesh(m.n_elem, m.n_ldof, wl["p"], torch.from_numpy(m.elem_dofs).to(dev),
                                torch.from_numpy(m.vertices).to(dev), torch.from_numpy(m.boundary).to(dev))
    q64 = ceed.alloc_qdata(mesh, ceed.CEED_OP_DIFFUSION, ceed.CEED_F64, dev)
    ceed.ceed_build_qdata(mesh, ceed.CEED_OP_DIFFUSION, ceed.CEED_COEFF_SINE, None, ceed.CEED_F64, q64)
    q32 = ceed.alloc_qdata(mesh, ceed.CEED_OP_DIFFUSION, ceed.CEED_F32, dev)
    ceed.ceed_build_qdata(mesh, ceed.CEED_OP_DIFFUSION, ceed.CEED_COEFF_SINE, None, ceed.CEED_F32, q32)
    b = torch.empty(m.n_ldof, dtype=torch.float64, device=dev)
    ceed.ceed_manufactured_rhs(mesh, ceed.CEED_COEFF_SINE, b, flags=ceed.CEED_APPLY_DIRICHLET)
    out = {"workload": f"{wl['N']}^3, p={wl['p']}, n_ldof={m.n_ldof}"}
    x64 = torch.empty_like(b)
    st, rep = ceed.ceed_cg_solve(mesh, q64, ceed.CEED_F64, b, x64, mode=ceed.CEED_CG_FP64, tol=1e-10,
                                 max_iter=20000, op=ceed.CEED_OP_DIFFUSION, raise_on_error=False)
    out["fp64_to_1e-10"] = dict(rep, status=st)
    xm = torch.empty_like(b)
    for name, mode in (("mixed_f32", ceed.CEED_CG_MIXED), ("mixed_f32_reliable", ceed.CEED_CG_MIXED_RELIABLE)):
        st, repm = ceed.ceed_cg_solve(mesh, q64, ceed.CEED_F64, b, xm, mode=mode, tol=1e-10, max_iter=20000,
                                      op=ceed.CEED_OP_DIFFUSION, qdata_lo=q32, prec_lo=ceed.CEED_F32,
                                      raise_on_error=False)
        diff = float(torch.linalg.vector_norm(xm - x64) / torch.linalg.vector_norm(x64))
        out[f"{name}_to_1e-10"] = dict(repm, status=st, rel_diff_from_fp64_solution=diff)
        if rep["seconds"] > 0 and repm["seconds"] > 0:
            out[f"{name}_speedup"] = rep["seconds"] / repm["seconds"]
    mesh.close()
    del q64, q32, b, x64, xm
    torch.cuda.empty_cache()
    return out


def nt_workload(ceed, dev, p=4, q=5, N=48):
    """Degree-p tetrahedra, 6 per cube of the perturbed N^3 lattice, conical rule with q points per direction."""
    import torch
    m = synthetic.TetMesh(N, N, N, p, seed=0)
    interp, grad, qw, qref = ceed.ceed_simplex_basis(p, q)
    nt = ceed.ceed_nt_setup(m.n_elem, m.n_ldof, interp, grad, qw, qref, torch.from_numpy(m.elem_dofs).to(dev),
                            torch.from_numpy(m.vertices).to(dev), None)
    return m, nt


def run_nt_profile(args):
    """Three applies of the tetrahedral diffusion operator with one algorithm (for ncu captures)."""
    import torch
    import paper_2109_05072_gb300 as ceed
    dev = torch.device("cuda", 0)
    m, nt = nt_workload(ceed, dev)
    algo, prec = {"fused64": (ceed.CEED_NT_FUSED, ceed.CEED_F64), "fused32": (ceed.CEED_NT_FUSED, ceed.CEED_F32),
                  "gemm32": (ceed.CEED_NT_GEMM, ceed.CEED_F32), "tc": (ceed.CEED_NT_TC, ceed.CEED_F32)}[args.nt_profile]
    qd = ceed.alloc_nt_qdata(nt, ceed.CEED_OP_DIFFUSION, prec, dev)
    ceed.ceed_nt_build_qdata(nt, ceed.CEED_OP_DIFFUSION, ceed.CEED_COEFF_SINE, None, prec, qd)
    ceed.ceed_nt_set_algorithm(nt, ceed.CEED_OP_DIFFUSION, prec, algo)
    x = torch.from_numpy(synthetic.uniform(m.n_ldof, seed=1)).to(dev)
    y = torch.empty_like(x)
    for _ in range(3):
        ceed.ceed_nt_apply(nt, ceed.CEED_OP_DIFFUSION, qd, prec, x, y)
    ceed.ceed_nt_status(nt)
    print(json.dumps({"nt_profile": args.nt_profile, "n_elem": m.n_elem, "n_ldof": m.n_ldof}))


def run_nontensor(ceed, dev, args):
    """Non-tensor elements (the paper's GEMM formulation of the MAGMA backend, and the fused kernel):
    degree-4 tetrahedra, 6 per cube of the perturbed 48^3 lattice (663,552 elements, 7,189,057 nodes),
    conical rule with q = 5 points per direction (Q = 125), diffusion with the sine coefficient."""
    import torch
    p, q, N = 4, 5, 48
    m, nt = nt_workload(ceed, dev, p, q, N)
    P, Q, E = nt.P, nt.Q, m.n_elem
    x = torch.from_numpy(synthetic.uniform(m.n_ldof, seed=1)).to(dev)
    y = torch.empty_like(x)
    flops = E * (2 * 2 * 3 * Q * P + 15 * Q)
    out = {"workload": f"diffusion, degree-{p} tetrahedra (Kuhn split of the perturbed {N}^3 lattice), "
                       f"conical rule q={q}", "n_elem": E, "n_ldof": m.n_ldof, "P": P, "Q": Q,
           "flops_per_apply": flops, "runs": []}
    hbm_peak, _ = load_peaks()
    for prec, name, tb in ((ceed.CEED_F64, "f64", 8), (ceed.CEED_F64_DF, "f64df", 8), (ceed.CEED_F32, "f32", 4)):
        qd = ceed.alloc_nt_qdata(nt, ceed.CEED_OP_DIFFUSION, prec, dev)
        ceed.ceed_nt_build_qdata(nt, ceed.CEED_OP_DIFFUSION, ceed.CEED_COEFF_SINE, None, prec, qd)
        # algorithmic bytes: x and y once per node, the quadrature data, the int32 restriction
        by = 16 * m.n_ldof + 6 * Q * E * tb + 4 * P * E
        modes = [("fused", ceed.CEED_NT_FUSED, 0, 0), ("gemm_native", ceed.CEED_NT_GEMM, 0, 0),
                 ("gemm_emulated", ceed.CEED_NT_GEMM, 0, 1)]
        if prec == ceed.CEED_F64_DF:   # FP64 accuracy on the FP32 pipe: the fused algorithm only
            modes = modes[:1]
        if prec == ceed.CEED_F32:
            modes.append(("gemm_tf32", ceed.CEED_NT_GEMM, 0, 2))
            modes.append(("tensor_core_3xtf32", ceed.CEED_NT_TC, 0, 0))
        for label, algo, eta, gm in modes:
            ceed.ceed_nt_set_algorithm(nt, ceed.CEED_OP_DIFFUSION, prec, algo, eta, gm)
            ms = _time_cuda(lambda: ceed.ceed_nt_apply(nt, ceed.CEED_OP_DIFFUSION, qd, prec, x, y), 5, 3)
            out["runs"].append({"prec": name, "algo": label, "gemm_mode": gm, "ms": ms,
                                "gdofs": m.n_ldof / ms / 1e6, "tflops": flops / ms / 1e9,
                                "alg_gbs": by / ms / 1e6, "hbm_frac": by / ms / 1e6 / hbm_peak})
        if prec == ceed.CEED_F32:
            # the tensor-core kernel alone (without the transposed restriction), timed with CUDA events
            ceed.ceed_nt_set_algorithm(nt, ceed.CEED_OP_DIFFUSION, prec, ceed.CEED_NT_TC)
            tc_ms = _time_cuda(lambda: ceed.ceed_nt_apply(nt, ceed.CEED_OP_DIFFUSION, qd, prec, x, y), 5, 3)
            out["tensor_core_roofline"] = {
                "bound": "hbm", "kernel": "nt_tc_kernel<3,40,48>", "apply_ms": tc_ms,
                "alg_bytes_per_apply": by, "achieved_gbs_apply": by / tc_ms / 1e6, "peak": hbm_peak,
                "frac_apply": by / tc_ms / 1e6 / hbm_peak, "traffic_per_launch": NT_TC_TRAFFIC_PER_LAUNCH,
                "note": "apply = tensor-core kernel + deterministic transposed restriction"}
        algo, eta, gm, tms = ceed.ceed_nt_autotune(nt, ceed.CEED_OP_DIFFUSION, qd, prec, x, y)
        out[f"autotuned_{name}"] = {"algo": ["fused", "gemm", "tensor_core"][algo], "eta": eta, "gemm_mode": gm, "ms": tms}
        del qd
        torch.cuda.empty_cache()
    nt.close()
    return out


def run_hp(ceed, dev, args):
    """Conforming mixed-order space: orders 3, 5, 7 in x-slabs of a 48 x 24 x 24 perturbed lattice,
    Gauss q = p + 2, diffusion with the sine coefficient, Dirichlet boundary; one apply = P x, the three
    order groups' fused kernels, P^T."""
    import torch
    nx, ny, nz = 48, 24, 24
    orders = np.array([3 if (e % nx) < nx // 3 else 5 if (e % nx) < 2 * nx // 3 else 7 for e in range(nx * ny * nz)])
    m = synthetic.HexMesh(nx, ny, nz, 1, seed=0)
    t0 = time.perf_counter()
    h = ceed.ceed_hp_setup(nx, ny, nz, orders, torch.from_numpy(m.vertices).to(dev),
                           q_rule=ceed.CEED_QRULE_GAUSS, dirichlet=True)
    setup_s = time.perf_counter() - t0
    x = torch.from_numpy(synthetic.uniform(h.n_true, seed=1)).to(dev)
    y = torch.empty_like(x)
    out = {"workload": f"orders 3/5/7 in x-slabs of {nx}x{ny}x{nz} hexahedra, Gauss q=p+2, conforming (minimum rule)",
           "n_true": h.n_true, "n_elem_nodes": h.n_rows, "setup_s": setup_s, "runs": []}
    for name, prec in (("f64", ceed.CEED_F64), ("f64df", ceed.CEED_F64_DF), ("f32", ceed.CEED_F32)):
        ceed.ceed_hp_build_qdata(h, ceed.CEED_OP_DIFFUSION, ceed.CEED_COEFF_SINE, prec=prec)
        ms = _time_cuda(lambda: ceed.ceed_hp_apply(h, ceed.CEED_OP_DIFFUSION, prec, x, y,
                                                   flags=ceed.CEED_APPLY_DIRICHLET), 5, 3)
        out["runs"].append({"prec": name, "ms": ms, "gdofs_true": h.n_true / ms / 1e6,
                            "gdofs_elem_nodes": h.n_rows / ms / 1e6})
    h.close()
    return out


def compact_summary(line):
    """The headline numbers of every leg in a few hundred bytes (GDOF/s, fractions, CG seconds)."""
    r = lambda v, d=3: None if v is None else round(v, d)
    out = {"fp64_gdofs": r(line["value"]), "fp64_frac_of_measured_fp64": r(line["roofline"]["frac"]),
           "fp64_hbm_frac": r(line["roofline"]["hbm_frac"])}
    df = line.get("fp64_accurate_fp32_pipe")
    if df:
        out["df_gdofs"] = r(df["gdofs"])
        out["df_hbm_frac"] = r(df["roofline"]["frac"])
        out["df_rel_l2_vs_fp64"] = df["rel_l2_vs_fp64"]
        if df.get("fp32_pipe_ceiling"):
            out["df_ceiling_gdofs_dot2_16warps"] = r(df["fp32_pipe_ceiling"]["gdofs_at_dot2_rate_16warps"])
    for k, v in (line.get("mixed_apply") or {}).items():
        out[f"{k}_gdofs"] = r(v["gdofs"])
        out[f"{k}_hbm_frac"] = r(v["hbm_frac"])
        if v.get("roofline"):
            out[f"{k}_kernel"] = v["roofline"]["kernel"].split("<")[0]
        if v.get("element_kernel_ms"):
            out[f"{k}_element_kernel_gdofs"] = r(v["gdofs"] * v["ms"] / v["element_kernel_ms"])
    cg = line.get("cg") or {}
    if cg:
        f = cg.get("fp64_to_1e-10", {})
        out["cg_fp64_s"] = r(f.get("seconds"))
        out["cg_fp64_iters"] = f.get("iterations")
        out["cg_fp64_100_iters_fused_s"] = r(cg.get("fp64_100_iters_s"))
        out["cg_fp64_100_iters_separate_s"] = r(cg.get("fp64_100_iters_separate_kernels_s"))
        sep = cg.get("mixed_f32_reliable_separate_kernels_to_1e-10")
        if sep:
            out["cg_mixed_f32_reliable_separate_kernels_s"] = r(sep.get("seconds"))
        spl = cg.get("mixed_f32_reliable_iteration_split")
        if spl:
            out["cg_mixed_f32_iter_split_ms"] = {"apply": r(spl["apply_ms"]), "vector": r(spl["vector_ms"]),
                                                 "vector_hbm_frac": r(spl["vector_hbm_frac"])}
        for key in ("mixed_f32", "mixed_f32_reliable", "mixed_f64df_reliable", "pmg_fp32_smoothers"):
            d = cg.get(f"{key}_to_1e-10")
            if d:
                out[f"cg_{key}_s"] = r(d.get("seconds"))
                out[f"cg_{key}_iters"] = d.get("iterations")
                out[f"cg_{key}_rel_res"] = d.get("rel_residual")
                sp = cg.get(f"{key}_speedup") or cg.get(f"{key}_speedup_vs_fp64_jacobi")
                out[f"cg_{key}_speedup"] = r(sp)
    b = line.get("batched")
    if b:
        out["batched_gdofs_by_nrhs"] = {str(x["nrhs"]): r(x["gdofs"]) for x in b["runs"]}
        out["batched_fp64_frac_by_nrhs"] = {str(x["nrhs"]): r(x.get("fp64_frac")) for x in b["runs"]}
        if b.get("fp64_accurate_fp32_pipe"):
            out["batched_df_gdofs_by_nrhs"] = {str(x["nrhs"]): r(x["gdofs"]) for x in b["fp64_accurate_fp32_pipe"]}
    pk = line.get("peaks_measured") or {}
    out["peak_tflops"] = {k: r(v["tflops"]) for k, v in pk.items()}
    return out


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=20)
    ap.add_argument("--warmup", type=int, default=5)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--workload", default="c2", choices=sorted(WORKLOADS))
    ap.add_argument("--cg", type=int, default=1, help="run the CG measurements (1) or skip them (0)")
    ap.add_argument("--cg-workload", default="c2", choices=sorted(WORKLOADS))
    ap.add_argument("--cpu-sample", type=int, default=40000, help="elements in the timed oracle sample")
    ap.add_argument("--ref-sample", type=int, default=1000, help="elements per reference-arm step")
    ap.add_argument("--profile", default=None, choices=["f64", "f32", "bf16", "f64df", "cg", "batched"],
                    help="profiling case: set up the workload, run three applies in this precision (or, with "
                         "cg, 20 mixed-precision CG iterations), exit")
    ap.add_argument("--cg-separate", type=int, default=0, help="--profile cg: one kernel per CG step (1) or fused (0)")
    ap.add_argument("--variant", default=None, help="ne,stage for --profile (default: autotune)")
    ap.add_argument("--autotune", type=int, default=1, help="autotune the apply kernel before timing")
    ap.add_argument("--batched", type=int, default=1, help="measure the batched mixed-order apply")
    ap.add_argument("--adjoint", type=int, default=1, help="measure the adjoint kernels")
    ap.add_argument("--df", type=int, default=1, help="measure the double-float FP64-accurate operator")
    ap.add_argument("--nontensor", type=int, default=1, help="measure the non-tensor (tetrahedral) operator")
    ap.add_argument("--hp", type=int, default=1, help="measure the conforming mixed-order (hp) operator")
    ap.add_argument("--cg-c4", type=int, default=0,
                    help="also run CG to 1e-10 on 80^3 elements, p = 7 (FP64 vs mixed; about three minutes)")
    ap.add_argument("--nt-profile", default=None, choices=["fused64", "fused32", "gemm32", "tc"],
                    help="profiling case: three tetrahedral diffusion applies with one algorithm, then exit")
    args = ap.parse_args()
    if args.impl == "reference":
        return run_reference(args)
    if args.profile == "cg":
        return run_profile_cg(args)
    if args.profile == "batched":   # the persistent mixed-order launch, nrhs = 1 (for ncu captures)
        import torch
        import paper_2109_05072_gb300 as ceed
        out = run_batched(ceed, torch.device("cuda", 0), args, nrhs_list=(1,), steps=1)
        print(json.dumps({"profile": "batched", "runs": out["runs"]}))
        return
    if args.profile:
        return run_profile(args)
    if args.nt_profile:
        return run_nt_profile(args)
    if args.warmup < 3:
        raise SystemExit("--warmup must be >= 3")

    import torch
    ws, rank, local = dist_env()
    torch.cuda.set_device(local)
    if ws > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl")
    import paper_2109_05072_gb300 as ceed

    def barrier():
        if ws > 1:
            import torch.distributed as dist
            dist.barrier()

    wl = WORKLOADS[args.workload]
    N, p = wl["N"], wl["p"]
    m = synthetic.cube_mesh(N, p, seed=0)
    dev = torch.device("cuda", local)
    mesh = ceed.ceed_setup_mesh(m.n_elem, m.n_ldof, p, torch.from_numpy(m.elem_dofs).to(dev),
                                torch.from_numpy(m.vertices).to(dev), torch.from_numpy(m.boundary).to(dev))
    qd64 = ceed.alloc_qdata(mesh, ceed.CEED_OP_DIFFUSION, ceed.CEED_F64, dev)
    ceed.ceed_build_qdata(mesh, ceed.CEED_OP_DIFFUSION, ceed.CEED_COEFF_SINE, None, ceed.CEED_F64, qd64)
    n_apply = m.n_ldof
    x_host = synthetic.uniform(m.n_ldof, seed=1 + rank)
    x = torch.from_numpy(x_host).to(dev)
    y = torch.empty_like(x)
    stream = torch.cuda.current_stream()

    def timed(fn, steps, warmup):
        for _ in range(warmup):
            fn()
        torch.cuda.synchronize()
        barrier()
        torch.cuda.synchronize()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        for _ in range(steps):
            fn()
        e1.record(stream)
        torch.cuda.synchronize()
        barrier()
        ms = max_over_ranks(e0.elapsed_time(e1), ws, dev)
        return ms / steps

    # ---------------- arithmetic peaks of this GPU, measured now (the roofline denominators of the
    # FP64 operator and of the FP32-pipe operators): independent FMA chains on every SM
    peaks = {}
    for name, kind in (("f64", 0), ("f32", 1), ("f32x2", 2)):
        tf, per_clk, mhz = ceed.ceed_fma_throughput(kind)
        peaks[name] = {"tflops": tf, "fma_per_clk_per_sm": per_clk, "sm_mhz": mhz}
    # the double-float operator's packed compensated sums (Dot2 steps) alone, at its occupancy (16
    # warps per SM) and at 64: FP32 lane operations per clock per SM (the FMA pipe's peak is ~128)
    for name, kind in (("dot2_16warps", 3), ("dot2_64warps", 4)):
        tops, per_clk, mhz = ceed.ceed_fma_throughput(kind)
        peaks[name] = {"tflops": tops, "lane_ops_per_clk_per_sm": per_clk, "sm_mhz": mhz}

    # ---------------- headline: FP64 apply (variant chosen by the library's autotuner first)
    variants = {}
    if args.autotune:
        ne, st, tms = ceed.ceed_autotune_apply(mesh, ceed.CEED_OP_DIFFUSION, qd64, ceed.CEED_F64, x, y)
        variants["f64"] = {"elems_per_block": ne, "tma_staging": st, "tuning_ms": tms}
    apply64 = lambda: ceed.ceed_apply_diffusion(mesh, qd64, ceed.CEED_F64, x, y)
    with ClockSampler(local) as clk:
        ms64 = timed(apply64, args.steps, args.warmup)
    gdofs64 = whole_job_rate(n_apply, ws, ms64)
    reads, flops_el = cost_per_element(p)
    hbm_peak, hbm_kind = load_peaks()
    bytes64 = algorithmic_bytes(m, 8)
    launches_per_apply = mesh.n_colors
    v64 = variants.get("f64", {"elems_per_block": 1, "tma_staging": 0})
    kernel_id = (f"fix_kernel<{p + 1},{p + 1},DIFFUSION>" if 5 <= p <= 7 else  # integer slices: one kernel, no variants
                 f"apply_kernel<{p + 1},{p + 1},DIFFUSION,double,double,stage={v64['tma_staging']}>"
                 f"[ne={v64['elems_per_block']}]")
    ms_launch = ms64 / launches_per_apply
    flops_launch = fp64_pipe_flops(p) * m.n_elem / launches_per_apply
    achieved_tf = flops_launch / (ms_launch * 1e-3) / 1e12

    # ---------------- FP64-accurate operator on the FP32 pipe (double-float), and its agreement with FP64
    f64df = None
    if args.df:
        qdf = ceed.alloc_qdata(mesh, ceed.CEED_OP_DIFFUSION, ceed.CEED_F64_DF, dev)
        ceed.ceed_build_qdata(mesh, ceed.CEED_OP_DIFFUSION, ceed.CEED_COEFF_SINE, None, ceed.CEED_F64_DF, qdf)
        ydf = torch.empty_like(x)
        if args.autotune:
            ne, st, tms = ceed.ceed_autotune_apply(mesh, ceed.CEED_OP_DIFFUSION, qdf, ceed.CEED_F64_DF, x, ydf)
            variants["f64_df"] = {"elems_per_block": ne, "tma_staging": st, "tuning_ms": tms}
        ms_df = timed(lambda: ceed.ceed_apply_diffusion(mesh, qdf, ceed.CEED_F64_DF, x, ydf), args.steps, args.warmup)
        ceed.ceed_apply_diffusion(mesh, qd64, ceed.CEED_F64, x, y)
        ceed.ceed_apply_diffusion(mesh, qdf, ceed.CEED_F64_DF, x, ydf)
        torch.cuda.synchronize()
        rel = float(torch.linalg.vector_norm(ydf - y) / torch.linalg.vector_norm(y))
        relmax = float((ydf - y).abs().max() / y.abs().max())
        vdf = variants.get("f64_df", {"elems_per_block": 0, "tma_staging": 1})
        kid_df = (f"apply_kernel<8,8,DIFFUSION,DF,DF,stage={vdf['tma_staging']}>[ne={vdf['elems_per_block']}]")
        f64df = {"gdofs": whole_job_rate(n_apply, ws, ms_df), "ms": ms_df, "dtype": "f32x2 (double-float, compensated dot)",
                 "rel_l2_vs_fp64": rel, "rel_max_vs_fp64": relmax,
                 "flops_tflops_paper_model": flops_el * m.n_elem / (ms_df * 1e-3) / 1e12,
                 "speedup_vs_native_fp64": ms64 / ms_df,
                 "roofline": {"bound": "hbm", "achieved": bytes64 / launches_per_apply / (ms_df / launches_per_apply * 1e-3) / 1e9,
                              "peak": hbm_peak, "unit": "GB/s",
                              "frac": bytes64 / (ms_df * 1e-3) / 1e9 / hbm_peak,
                              "traffic": PROFILED_TRAFFIC_PER_LAUNCH.get(kid_df) if N == 64 else None,
                              "kernel": kid_df, "alg_bytes_per_launch": bytes64 / launches_per_apply,
                              "ms_per_launch": ms_df / launches_per_apply, "peak_kind": f"{hbm_kind} copy bandwidth",
                              "fp32_peak_tflops_measured": peaks["f32"]["tflops"]}}
        # FP32-pipe ceiling: lane operations per element of the compensated passes (6 passes x P^2
        # lines x 448 at P = 8, and 100 per point) at the rate measured for the bare Dot2 chains
        if p == 7:
            lane_ops_el = 6 * 64 * 448 + 512 * 100
            dofs_el = m.n_ldof / m.n_elem
            f64df["fp32_pipe_ceiling"] = {
                "lane_ops_per_element": lane_ops_el,
                "gdofs_at_fma_peak": peaks["f32"]["tflops"] * 1e12 / 2 / lane_ops_el * dofs_el / 1e9,
                "gdofs_at_dot2_rate_16warps": peaks["dot2_16warps"]["tflops"] * 1e12 / lane_ops_el * dofs_el / 1e9,
                "gdofs_at_dot2_rate_64warps": peaks["dot2_64warps"]["tflops"] * 1e12 / lane_ops_el * dofs_el / 1e9,
                "note": "the operator's compensated arithmetic alone, at the measured rates of the FMA pipe and "
                        "of bare packed Dot2 chains; HBM bound at 93 B/DOF for comparison: "
                        f"{hbm_peak / 93.1:.1f} GDOF/s"}
        del qdf, ydf
        torch.cuda.empty_cache()

    # ---------------- FP32-arithmetic operator (mixed), FP32 and BF16 quadrature data
    mixed = {}
    for name, prec, qb in (("f32", ceed.CEED_F32, 4), ("bf16", ceed.CEED_BF16, 2), ("f32geo", ceed.CEED_F32_GEO, 4)):
        qlo = ceed.alloc_qdata(mesh, ceed.CEED_OP_DIFFUSION, prec, dev)
        ceed.ceed_build_qdata(mesh, ceed.CEED_OP_DIFFUSION, ceed.CEED_COEFF_SINE, None, prec, qlo)
        if args.autotune:
            ne, st, tms = ceed.ceed_autotune_apply(mesh, ceed.CEED_OP_DIFFUSION, qlo, prec, x, y)
            variants[name] = {"elems_per_block": ne, "tma_staging": st, "tuning_ms": tms}
        ms = timed(lambda: ceed.ceed_apply_diffusion(mesh, qlo, prec, x, y), args.steps, args.warmup)
        by = algorithmic_bytes(m, qb, geo=(prec == ceed.CEED_F32_GEO))
        mixed[name] = {"gdofs": whole_job_rate(m.n_ldof, ws, ms), "ms": ms, "alg_bytes": by,
                       "hbm_gbs": by / (ms * 1e-3) / 1e9, "hbm_frac": by / (ms * 1e-3) / 1e9 / hbm_peak}
        v = variants.get(name, {"elems_per_block": 0, "tma_staging": 1})
        tq = {"f32": "float", "bf16": "bf16", "f32geo": "float,geo"}[name]
        if v["tma_staging"] >= 2:   # the brick kernel (2 x 2 x 1 elements per block)
            kid = f"brick_kernel<8,8,DIFFUSION,float,{tq},stage={v['tma_staging'] - 2}>"
            # the element kernel on the same buffers, for comparison
            ceed.ceed_set_apply_variant(mesh, ceed.CEED_OP_DIFFUSION, prec, 2, 1)
            mixed[name]["element_kernel_ms"] = timed(lambda: ceed.ceed_apply_diffusion(mesh, qlo, prec, x, y),
                                                     args.steps, args.warmup)
            ceed.ceed_set_apply_variant(mesh, ceed.CEED_OP_DIFFUSION, prec, 1, v["tma_staging"])
        else:
            kid = f"apply_kernel<8,8,DIFFUSION,float,{tq},stage={v['tma_staging']}>[ne={v['elems_per_block']}]"
        mixed[name]["roofline"] = {"bound": "hbm", "achieved": by / (ms * 1e-3) / 1e9, "peak": hbm_peak, "unit": "GB/s",
                                   "frac": by / (ms * 1e-3) / 1e9 / hbm_peak,
                                   "traffic": PROFILED_TRAFFIC_PER_LAUNCH.get(kid) if N == 64 else None,
                                   "kernel": kid, "alg_bytes_per_launch": by / launches_per_apply,
                                   "ms_per_launch": ms / launches_per_apply, "peak_kind": f"{hbm_kind} copy bandwidth"}
        del qlo
    torch.cuda.empty_cache()

    # ---------------- end to end through the C ABI's host-buffer call (pinned host x and y): the
    # library copies x in, applies, copies y out and returns when y is on the host
    xh = torch.from_numpy(x_host).pin_memory()
    yh = torch.empty_like(xh).pin_memory()

    def e2e_step():
        ceed.ceed_apply_host(mesh, ceed.CEED_OP_DIFFUSION, qd64, ceed.CEED_F64, xh, yh, x, y)
    ms_e2e = timed(e2e_step, max(3, args.steps // 2), 3)

    # ---------------- CG: 100 FP64 iterations, and time to 1e-10 (FP64 vs mixed refinement)
    cg = None
    if args.cg:
        cg = {}
        if args.cg_workload != args.workload:
            del qd64
            mesh.close()
            torch.cuda.empty_cache()
            wlc = WORKLOADS[args.cg_workload]
            m = synthetic.cube_mesh(wlc["N"], wlc["p"], seed=0)
            mesh = ceed.ceed_setup_mesh(m.n_elem, m.n_ldof, wlc["p"], torch.from_numpy(m.elem_dofs).to(dev),
                                        torch.from_numpy(m.vertices).to(dev), torch.from_numpy(m.boundary).to(dev))
            qd64 = ceed.alloc_qdata(mesh, ceed.CEED_OP_DIFFUSION, ceed.CEED_F64, dev)
            ceed.ceed_build_qdata(mesh, ceed.CEED_OP_DIFFUSION, ceed.CEED_COEFF_SINE, None, ceed.CEED_F64, qd64)
        b = torch.empty(m.n_ldof, dtype=torch.float64, device=dev)
        ceed.ceed_manufactured_rhs(mesh, ceed.CEED_COEFF_SINE, b, flags=ceed.CEED_APPLY_DIRICHLET)
        xs = torch.empty_like(b)
        st, rep = ceed.ceed_cg_solve(mesh, qd64, ceed.CEED_F64, b, xs, mode=ceed.CEED_CG_FP64, fixed_iters=100,
                                     op=ceed.CEED_OP_DIFFUSION)
        cg["fp64_100_iters_s"] = rep["seconds"]
        cg["fp64_100_iters_dof_iter_per_s"] = 100 * m.n_ldof / rep["seconds"]
        cg["fp64_100_iters_fused"] = rep["fused"]
        # the same 100 iterations with one kernel per step (apply, reductions, updates)
        st, rep_sep = ceed.ceed_cg_solve(mesh, qd64, ceed.CEED_F64, b, xs, mode=ceed.CEED_CG_FP64, fixed_iters=100,
                                         op=ceed.CEED_OP_DIFFUSION, separate_kernels=1)
        cg["fp64_100_iters_separate_kernels_s"] = rep_sep["seconds"]
        st, rep64 = ceed.ceed_cg_solve(mesh, qd64, ceed.CEED_F64, b, xs, mode=ceed.CEED_CG_FP64, tol=1e-10,
                                       max_iter=20000, op=ceed.CEED_OP_DIFFUSION, raise_on_error=False)
        cg["fp64_to_1e-10"] = dict(rep64, status=st, ms_per_iter=1e3 * rep64["seconds"] / max(1, rep64["iterations"]))
        # low-precision inner operators: iterative refinement (restarted inner PCG to 1e-4 per pass) and
        # reliable updates (one PCG run, true FP64 residual put in place at every 10x decrease)
        for name, prec, modes in (("f32", ceed.CEED_F32, ("", "reliable")), ("bf16", ceed.CEED_BF16, ("reliable",)),
                                  ("f32geo", ceed.CEED_F32_GEO, ("reliable",)),
                                  ("f64df", ceed.CEED_F64_DF, ("reliable",))):
            qlo = ceed.alloc_qdata(mesh, ceed.CEED_OP_DIFFUSION, prec, dev)
            ceed.ceed_build_qdata(mesh, ceed.CEED_OP_DIFFUSION, ceed.CEED_COEFF_SINE, None, prec, qlo)
            for mode in modes:
                key = f"mixed_{name}" + (f"_{mode}" if mode else "")
                st, repm = ceed.ceed_cg_solve(mesh, qd64, ceed.CEED_F64, b, xs,
                                              mode=ceed.CEED_CG_MIXED_RELIABLE if mode else ceed.CEED_CG_MIXED,
                                              tol=1e-10, max_iter=8000 if mode else 40000, op=ceed.CEED_OP_DIFFUSION, qdata_lo=qlo,
                                              prec_lo=prec, inner_tol=1e-4, raise_on_error=False)
                cg[f"{key}_to_1e-10"] = dict(repm, status=st, ms_per_iter=1e3 * repm["seconds"] / max(1, repm["iterations"]))
                if rep64["seconds"] > 0 and repm["seconds"] > 0:
                    cg[f"{key}_speedup"] = rep64["seconds"] / repm["seconds"]
                if name == "f32" and mode == "reliable":
                    # per-iteration split: the masked apply as the fused iteration runs it (element
                    # kernel, 2 elements per block, quadrature data read directly), timed on its own,
                    # and the rest of the iteration (the FP64 vector phases: 11 passes of 8 bytes per
                    # entry, the reductions, the grid barriers)
                    saved = variants.get(name)
                    ceed.ceed_set_apply_variant(mesh, ceed.CEED_OP_DIFFUSION, prec, 2, 0)
                    xm = torch.from_numpy(synthetic.uniform(m.n_ldof, seed=3)).to(dev)
                    ym = torch.empty_like(xm)
                    ms_ap = timed(lambda: ceed.ceed_apply_diffusion(mesh, qlo, prec, xm, ym,
                                                                    flags=ceed.CEED_APPLY_DIRICHLET), 10, 3)
                    del xm, ym
                    if saved:
                        ceed.ceed_set_apply_variant(mesh, ceed.CEED_OP_DIFFUSION, prec,
                                                    max(1, saved["elems_per_block"]), saved["tma_staging"])
                    ms_it = 1e3 * repm["seconds"] / max(1, repm["iterations"])
                    vec_bytes = 11 * 8 * m.n_ldof
                    cg["mixed_f32_reliable_iteration_split"] = {
                        "ms_per_iter": ms_it, "apply_ms": ms_ap, "vector_ms": ms_it - ms_ap,
                        "vector_bytes": vec_bytes, "vector_gbs": vec_bytes / ((ms_it - ms_ap) * 1e-3) / 1e9,
                        "vector_hbm_frac": vec_bytes / ((ms_it - ms_ap) * 1e-3) / 1e9 / load_peaks()[0],
                        "note": "apply timed stand-alone (masked, the fused iteration's element variant); "
                                "vector = the rest of the iteration"}
                    # the same solve with one kernel per step instead of the fused iteration
                    st, reps = ceed.ceed_cg_solve(mesh, qd64, ceed.CEED_F64, b, xs, mode=ceed.CEED_CG_MIXED_RELIABLE,
                                                  tol=1e-10, max_iter=8000, op=ceed.CEED_OP_DIFFUSION, qdata_lo=qlo,
                                                  prec_lo=prec, raise_on_error=False, separate_kernels=1)
                    cg[f"{key}_separate_kernels_to_1e-10"] = dict(
                        reps, status=st, ms_per_iter=1e3 * reps["seconds"] / max(1, reps["iterations"]))
            del qlo
        # p-multigrid-preconditioned (flexible) CG: levels p = 7, 3, 1 on the same elements, Chebyshev-Jacobi
        # smoothing (degree 3) with FP64 or FP32-arithmetic level operators, Jacobi-PCG on the p = 1 level
        Nc = WORKLOADS[args.cg_workload]["N"]
        lv_meshes, lv_q64, lv_q32, keep = [mesh], [qd64], [], []
        q32f = ceed.alloc_qdata(mesh, ceed.CEED_OP_DIFFUSION, ceed.CEED_F32, dev)
        ceed.ceed_build_qdata(mesh, ceed.CEED_OP_DIFFUSION, ceed.CEED_COEFF_SINE, None, ceed.CEED_F32, q32f)
        lv_q32.append(q32f)
        t0 = time.perf_counter()
        for pc in (3, 1):
            mcs = synthetic.cube_mesh(Nc, pc, seed=0)
            mc = ceed.ceed_setup_mesh(mcs.n_elem, mcs.n_ldof, pc, torch.from_numpy(mcs.elem_dofs).to(dev),
                                      torch.from_numpy(mcs.vertices).to(dev), torch.from_numpy(mcs.boundary).to(dev))
            q64c = ceed.alloc_qdata(mc, ceed.CEED_OP_DIFFUSION, ceed.CEED_F64, dev)
            ceed.ceed_build_qdata(mc, ceed.CEED_OP_DIFFUSION, ceed.CEED_COEFF_SINE, None, ceed.CEED_F64, q64c)
            q32c = ceed.alloc_qdata(mc, ceed.CEED_OP_DIFFUSION, ceed.CEED_F32, dev)
            ceed.ceed_build_qdata(mc, ceed.CEED_OP_DIFFUSION, ceed.CEED_COEFF_SINE, None, ceed.CEED_F32, q32c)
            lv_meshes.append(mc)
            lv_q64.append(q64c)
            lv_q32.append(q32c)
        for name, qlo, smoother in (("pmg_fp64_smoothers", None, 0), ("pmg_fp32_smoothers", lv_q32, 0),
                                    ("pmg_schwarz_fp32_smoothers", lv_q32, 1)):
            t1 = time.perf_counter()
            pmg = ceed.ceed_pmg_create(lv_meshes, lv_q64, qlo, prec_lo=ceed.CEED_F32, smoother=smoother)
            setup_s = time.perf_counter() - t1
            st, repp = ceed.ceed_cg_solve(mesh, qd64, ceed.CEED_F64, b, xs, mode=ceed.CEED_CG_FP64, tol=1e-10,
                                          max_iter=2000, op=ceed.CEED_OP_DIFFUSION, pmg=pmg, raise_on_error=False)
            cg[f"{name}_to_1e-10"] = dict(repp, status=st, setup_s=setup_s,
                                          lambda_max=[ceed.ceed_pmg_info(pmg, k) for k in range(2)])
            if rep64["seconds"] > 0 and repp["seconds"] > 0:
                cg[f"{name}_speedup_vs_fp64_jacobi"] = rep64["seconds"] / repp["seconds"]
            pmg.close()
        cg["pmg_levels"] = "p = 7, 3, 1 on the same elements (hierarchy built in %.1f s)" % (time.perf_counter() - t0)
        for mc in lv_meshes[1:]:
            mc.close()
        del lv_q64[1:], lv_q32
        cg["workload"] = f"{WORKLOADS[args.cg_workload]['N']}^3, p=7, n_ldof={m.n_ldof}"

    # ---------------- batched apply: p = 3, 5, 7 meshes (Gauss q = p+2), 3 components, 1..16 RHS, one launch
    batched = None
    if args.batched:
        batched = run_batched(ceed, dev, args, peaks)
        # the same batches with the FP64-accurate double-float operator
        batched["fp64_accurate_fp32_pipe"] = run_batched(ceed, dev, args, peaks, nrhs_list=(1, 4, 16),
                                                         prec=ceed.CEED_F64_DF)["runs"]

    # ---------------- adjoint: L = 0.5 ||A(k) x - b||^2, p = 4 and 8 on 32^3, geometry stored vs recomputed
    adjoint = None
    if args.adjoint:
        adjoint = run_adjoint(ceed, dev, args)

    # ---------------- non-tensor elements: degree-4 tetrahedra, fused kernel vs the GEMM formulation
    nontensor = None
    if args.nontensor:
        nontensor = run_nontensor(ceed, dev, args)

    # ---------------- conforming mixed-order (hp) space: orders 3, 5, 7 joined at their interfaces
    hp = None
    if args.hp:
        hp = run_hp(ceed, dev, args)

    # ---------------- CG on the 176.6M-DOF mesh (opt-in: minutes of solver time)
    cg_c4 = None
    if args.cg_c4:
        cg_c4 = run_cg_c4(ceed, dev, args)

    # ---------------- CPU oracle on a bounded sample (rank 0, N = 1 only)
    cpu = None
    if rank == 0 and ws == 1 and args.cpu_sample > 0:
        mc = synthetic.cube_mesh(N, p, seed=0)
        rate, dt = oracle_sample_rate(mc, min(args.cpu_sample, mc.n_elem))
        cpu = {"value": rate / 1e9, "unit": "GDOF/s", "cores": blas_threads(), "kind": "oracle",
               "sample": f"first {min(args.cpu_sample, mc.n_elem)} of {mc.n_elem} elements, dense FP64 "
                         f"per-element quadrature (numpy), {dt:.1f} s; DOFs counted as n_ldof/n_elem per element"}

    if rank == 0:
        line = {
            "metric": METRIC, "value": gdofs64, "unit": "GDOF/s", "n_gpus": ws, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": ms64, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": {"workload": f"FP64 diffusion apply, {N}^3 perturbed hexes (0.1h), p={p}, GLL collocated q=p+1, "
                                   f"6 stored geometric factors, k=1+0.5sin sin sin",
                       "n_ldof": n_apply,
                       "n_elem": N ** 3, "l2": "inputs larger than L2 (qdata 6.4 GB), no flush",
                       "parallelism": f"replicas x{ws}" if ws > 1 else "single GPU"},
            "roofline": {"bound": "alu", "achieved": achieved_tf, "peak": peaks["f64"]["tflops"], "unit": "TFLOP/s",
                         "frac": achieved_tf / peaks["f64"]["tflops"],
                         "traffic": PROFILED_TRAFFIC_PER_LAUNCH.get(kernel_id) if N == 64 else None,
                         "alg_bytes_per_launch": bytes64 / launches_per_apply,
                         "kernel": kernel_id,
                         "peak_kind": "measured in this run: FP64 FMA chains on every SM (ceed_fma_throughput), "
                                      f"{peaks['f64']['sm_mhz']:.0f} MHz; nominal {FP64_NOMINAL_TFLOPS}",
                         "peak_nominal": FP64_NOMINAL_TFLOPS,
                         "note": "achieved counts what is left on the FP64 pipe: 12 instructions a point (pointwise step and "
                                 "final sums, 2 flops each); the 1D passes run as exact integer slices on the tensor "
                                 "cores.  model_tflops: the paper's cost model (12 P^4 + 15 P^3 per element)",
                         "flops_per_launch": flops_launch, "ms_per_launch": ms_launch,
                         "model_tflops": flops_el * m.n_elem / (ms64 * 1e-3) / 1e12,
                         "hbm_gbs": bytes64 / (ms64 * 1e-3) / 1e9, "hbm_peak": hbm_peak, "hbm_peak_kind": hbm_kind,
                         "hbm_frac": bytes64 / (ms64 * 1e-3) / 1e9 / hbm_peak},
            "fp64_accurate_fp32_pipe": f64df,
            "mixed_apply": mixed,
            "apply_variants": variants,
            "e2e": {"value": whole_job_rate(n_apply, ws, ms_e2e),
                    "unit": "GDOF/s", "h2d_bytes_per_step": 8 * len(x_host), "d2h_bytes_per_step": 8 * len(x_host),
                    "call": "ceed_apply_host (pinned host x, y; copies and apply inside the timed region)"},
            "gpu_launches": args.steps * launches_per_apply,
            "clocks": clk.summary(),
            "cg": cg,
            "batched": batched,
            "adjoint": adjoint,
            "nontensor": nontensor,
            "hp": hp,
            "cg_80cube": cg_c4,
            "cpu_baseline": cpu,
            "peaks_measured": peaks,
        }
        line["summary"] = compact_summary(line)   # last key: the short record of every leg
        print(json.dumps(line), flush=True)
    if ws > 1:
        import torch.distributed as dist
        dist.destroy_process_group()


if __name__ == "__main__":
    main()
