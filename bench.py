#!/usr/bin/env python
"""Benchmark: sparse-grid DOF*steps/s of the Krylov IIF2 DG solver on one GB300.

A bench step is one IIF2 time step of the 3D cubic reaction-diffusion workload
(d = 3, level n = 6, degree k = 2, 18 576 DOF, f(u) = -100 u^3, diffusion
diag(1, 0.5, 0.1), M = 30, dt = 0.005): reaction term, predictor, Arnoldi with
CGS2 (30 matvecs), exp(dt H), basis combination and the Newton solve with CG.
The timed steps start from the projected seeded initial state (20 steps = the
whole configured solve).

Usage:  python bench.py [--gpus N] [--steps K] [--warmup W] [--precision mixed|fp64]
                        [--impl native|reference] [--no-cpu-baseline]
Prints one JSON line on rank 0.
"""
import argparse
import json
import os
import subprocess
import sys
import tempfile
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "sparse-grid DOF*steps/s (IIF2, FP64-oracle-checked)"
UNIT = "DOF*steps/s"


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=20)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--precision", choices=["mixed", "fp64"], default="mixed")
    ap.add_argument("--impl", choices=["native", "reference"], default="native")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-e2e", action="store_true")
    ap.add_argument("--no-accuracy", action="store_true", help="skip the FP64 comparison run")
    ap.add_argument("--served-requests", type=int, default=12,
                    help="requests of the served leg (0 skips it)")
    ap.add_argument("--served-workers", type=int, default=4)
    ap.add_argument("--batch-instances", type=int, default=256,
                    help="instances of the batched leg (0 skips it)")
    ap.add_argument("--no-matvec", action="store_true", help="skip the large stand-alone matvec leg")
    ap.add_argument("--no-iif3", action="store_true", help="skip the IIF3 leg")
    ap.add_argument("--no-schnak", action="store_true", help="skip the two-species 200-step leg")
    ap.add_argument("--no-sparse-reaction", action="store_true",
                    help="skip the legs of the sparse-grid interpolation form of the reaction term")
    ap.add_argument("--full-comparisons", action="store_true",
                    help="also run the comparison runs kept out of the default line for time: the batch with every "
                         "instance in its own whole-step graph, the served saturation run with the engine off, "
                         "the served requests above 1e-6 re-solved from perturbed inputs and with sub-projections, "
                         "and the interpolation form's served requests one at a time and its batch in FP64")
    ap.add_argument("--served-no-fp64", action="store_true",
                    help="skip the FP64 one-at-a-time baseline of the served leg (and its accuracy check)")
    ap.add_argument("--served-rates", default="1",
                    help="comma-separated arrival rates of the served leg, as multiples of the one-at-a-time "
                         "capacity (e.g. 0.5,1,2)")
    return ap.parse_args()


def workload_config():
    from paper_1810_11111_gb300 import workloads
    return workloads.cubic3d()


def workload_desc(cfg):
    return {"workload": "cubic3d: u_t = div(diag(1,0.5,0.1) grad u) - 100 u^3 on [0,1]^3, periodic, "
                        "sparse grid level 6, degree 2, 8 seeded Fourier modes, IIF2 M=30 dt=0.005",
            "d": cfg["d"], "level": cfg["n"], "degree": cfg["k"], "krylov_m": cfg["M"], "dt": cfg["dt"],
            "species": len(cfg["kappas"])}


# ----------------------------------------------------------------- clocks ---

class ClockSampler:
    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index):
        self.gpu = gpu_index
        self.proc = None
        self.path = None

    def start(self):
        try:
            fd, self.path = tempfile.mkstemp(suffix=".csv")
            os.close(fd)
            self.fh = open(self.path, "w")
            self.proc = subprocess.Popen(["nvidia-smi", "-i", str(self.gpu), "--query-gpu=" + self.FIELDS,
                                          "--format=csv,noheader,nounits", "-lms", "200"],
                                         stdout=self.fh, stderr=subprocess.DEVNULL)
        except (OSError, FileNotFoundError):
            self.proc = None

    def stop(self):
        if self.proc is None:
            return None
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except subprocess.TimeoutExpired:
            self.proc.kill()
        self.fh.close()
        rows = []
        with open(self.path) as fh:
            for ln in fh:
                parts = [p.strip() for p in ln.split(",")]
                if len(parts) >= 9:
                    rows.append(parts)
        os.unlink(self.path)
        if not rows:
            return None
        sm = [float(r[1]) for r in rows if r[1].replace(".", "").isdigit()]
        smax = [float(r[2]) for r in rows if r[2].replace(".", "").isdigit()]
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        reasons = sorted({names[i] for r in rows for i in range(4) if r[5 + i].lower() == "active"})
        return {"sm_mhz": float(np.median(sm)) if sm else None, "sm_max_mhz": max(smax) if smax else None,
                "reasons": reasons, "samples": len(rows)}


# --------------------------------------------------------------- roofline ---

def layout_sizes(d, n, k):
    """Sizes of the partially transformed arrays R_0..R_d (see reaction.cu)."""
    from itertools import product
    H = (k + 1) << n

    def count(l):
        return (k + 1) * (1 if l == 0 else 1 << (l - 1))

    def sparse_dof(dim):
        if dim == 0:
            return 1
        return sum(int(np.prod([count(v) for v in t])) for t in product(range(n + 1), repeat=dim) if sum(t) <= n)

    return [H ** i * sparse_dof(d - i) for i in range(d + 1)]


# DRAM bytes (read + write) of one launch from the committed ncu captures of
# the current kernels (cold, L2 flushed by ncu before the launch); a key is
# removed when the kernel changes.  Double-float F pencil launch (the
# dominant kernel of the cell-quadrature class in mixed mode), keyed by (d,
# level, degree, precision): profiles/pencil_kernel_cubic3d_l6k2_dfloat.md
PENCIL_TRAFFIC = {(3, 6, 2, "mixed"): 56705536 + 9454336}
# one persistent Arnoldi launch (one exponential), keyed by (d, level,
# degree, M, precision): profiles/arnoldi_kernel_cubic3d_l6k2_m30.md (the
# mixed-precision variant, double-float gather)
ARNOLDI_TRAFFIC = {(3, 6, 2, 30, "mixed"): 6524672 + 68352}


def pencil_q(cfg):
    """Gauss points per direction of the reaction quadrature, ceil((p k + k + 1)/2)."""
    p = max((sum(e) for terms in cfg["reaction"] for _, e in terms), default=0)
    k = cfg["k"]
    return max(1, (p * k + k + 1 + 1) // 2)


def measured_peaks():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(path):
        with open(path) as fh:
            return json.load(fh), "measured"
    return {"hbm_gbs": 6800.0, "bf16_tflops": 1900.0}, "fallback"


# ------------------------------------------------------------ native arm ---

def aggregate(units, ms, dist, device):
    """Whole-job throughput of independent replicas: the units of all ranks
    over the slowest rank's time (ms); returns (units/s, max ms)."""
    if dist is None:
        return units / (ms / 1e3), ms
    import torch
    t = torch.tensor([float(ms)], dtype=torch.float64, device=device)
    u = torch.tensor([float(units)], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    dist.all_reduce(u, op=dist.ReduceOp.SUM)
    return float(u) / (float(t) / 1e3), float(t)


def native(args, rank, world, local_rank):
    import torch

    from paper_1810_11111_gb300 import sgkiif
    from paper_1810_11111_gb300.runner import Problem

    torch.cuda.set_device(local_rank)
    dev = torch.device("cuda", local_rank)
    dist = None
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl", device_id=dev)
    cfg = workload_config()
    prec = sgkiif.SGK_MIXED if args.precision == "mixed" else sgkiif.SGK_FP64
    prob = Problem(cfg, prec, device=local_rank)
    dof, S = prob.dof, prob.nspecies
    elem = 4 if prec == sgkiif.SGK_MIXED else 8
    flush = torch.empty(64 * 1024 * 1024, dtype=torch.float32, device=dev)  # 256 MB > 129 MB L2
    stream = torch.cuda.current_stream(dev)

    def barrier():
        torch.cuda.synchronize(dev)
        if dist is not None:
            dist.barrier()

    # warm-up: one step outside any timing (module loading), then W steps as
    # timed below (CUDA graphs are captured on first use)
    prob.reset()
    prob.solver.step(1)
    prob.reset()
    for _ in range(args.warmup):
        prob.solver.step(1)

    # timed region: device time of each step, L2 flushed before each
    prob.reset()
    st0 = prob.solver.stats()
    barrier()
    visible = os.environ.get("CUDA_VISIBLE_DEVICES")
    clocks = ClockSampler(visible.split(",")[local_rank] if visible else local_rank)
    clocks.start()
    launches0 = prob.ctx.launches
    # the steps are queued (sgk_solver_step_async), so the host enqueues the
    # next flush and step while the GPU runs the current one; each step's
    # device time is still bracketed by its own pair of events
    ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(args.steps)]
    wall0 = time.perf_counter()
    for i in range(args.steps):
        flush.fill_(float(i))
        ev[i][0].record(stream)
        prob.solver.step_async(1)
        ev[i][1].record(stream)
    prob.solver.wait()
    torch.cuda.synchronize(dev)
    wall = time.perf_counter() - wall0
    total_ms = sum(a.elapsed_time(b) for a, b in ev)
    e0 = torch.cuda.Event(enable_timing=True)
    e1 = torch.cuda.Event(enable_timing=True)
    barrier()
    clk = clocks.stop()
    launches = prob.ctx.launches - launches0
    st1 = prob.solver.stats()
    final = prob.state()

    # the same K steps again with every kernel class event-timed (each launch
    # between two events); kernel timing runs the graph-captured sequences as
    # individual launches, so this pass is kept out of the headline number;
    # the dominant class is the one with the most device time over these steps
    prob.ctx.profile(0xFF)
    prob.reset()
    ps0 = prob.solver.stats()
    barrier()
    prof_ms = 0.0
    for i in range(args.steps):
        flush.fill_(float(i))
        e0.record(stream)
        prob.solver.step(1)
        e1.record(stream)
        e1.synchronize()
        prof_ms += e0.elapsed_time(e1)
    kprof = prob.ctx.profile_read()
    prob.ctx.profile(0)
    ps1 = prob.solver.stats()
    dominant = max(kprof, key=lambda c: kprof[c][0])

    # accuracy: against the oracle's state after the same steps (stored by
    # tests/golden/make_full_size.py, which calls only the oracle), and
    # against the FP64 GPU path
    acc, acc_oracle = None, None
    golden = os.path.join(ROOT, "tests", "golden", "cubic3d_steps.npz")
    if os.path.exists(golden):
        g = np.load(golden)
        key = "U%d" % args.steps
        if key in g.files:
            want = g[key]
            acc_oracle = float(np.sqrt(sum(np.sum((final[s] - want[s]) ** 2) for s in range(S)) /
                                       sum(np.sum(want[s] ** 2) for s in range(S))))
    if prec == sgkiif.SGK_MIXED and not args.no_accuracy:
        ref = Problem(cfg, sgkiif.SGK_FP64, device=local_rank)
        ref.reset()
        ref.solver.step(args.steps)
        rs = ref.state()
        acc = float(np.sqrt(sum(np.sum((final[s] - rs[s]) ** 2) for s in range(S)) /
                            sum(np.sum(rs[s] ** 2) for s in range(S))))
        ref.close()

    # end to end through the C ABI with host buffers: every step copies the
    # state in from pinned host memory and the result back out
    e2e = None
    if not args.no_e2e:
        host_in = [torch.from_numpy(u.cpu().numpy()).pin_memory() for u in prob.U0]
        host_out = [torch.empty(dof, dtype=torch.float64).pin_memory() for _ in range(S)]
        barrier()
        t_ms = 0.0
        for i in range(args.steps):
            flush.fill_(float(i))
            e0.record(stream)
            for s in range(S):
                sgkiif.sgk_solver_set_state(prob.solver.h, s, host_in[s].data_ptr(), 0)
            prob.solver.step(1)
            for s in range(S):
                sgkiif.sgk_solver_get_state(prob.solver.h, s, host_out[s].data_ptr(), dof, 0)
            e1.record(stream)
            e1.synchronize()
            t_ms += e0.elapsed_time(e1)
            host_in, host_out = host_out, host_in
        e2e_value, _ = aggregate(dof * S * args.steps, t_ms, dist, dev)
        e2e = {"value": e2e_value, "unit": UNIT,
               "h2d_bytes_per_step": dof * S * 8, "d2h_bytes_per_step": dof * S * 8}

    value, total_ms = aggregate(dof * S * args.steps, total_ms, dist, dev)

    # roofline of the dominant kernel class: algorithmic work per launch over
    # its event-timed average launch time in the profiled pass
    peaks, peak_kind = measured_peaks()
    nF = args.steps * 1 + (ps1["newton_iters"] - ps0["newton_iters"]) + args.steps  # predictor + residuals
    nJ = ps1["inner_iters"] - ps0["inner_iters"]
    sizes = layout_sizes(cfg["d"], cfg["n"], cfg["k"])
    ms, nl = kprof[dominant]
    d, kp1, N = cfg["d"], cfg["k"] + 1, cfg["n"]
    q = pencil_q(cfg)
    # per pass of the reaction term: the fused last-direction (pencil) kernel
    # reads R_{d-1}(U) (and R_{d-1}(w) for a Jacobian product) and writes
    # G_{d-1}; its arithmetic is the sum-factorised quadrature of every finest
    # cell plus the two-scale pyramids of every fiber.  The fiber transforms
    # of directions 0..d-2 read R_i and write R_{i+1}; the Krylov matvec (FP64
    # in both modes) reads x and writes y.
    bytes_algo, flops_algo = None, None
    if dominant == "cell_quadrature":
        last = sizes[d - 1]
        cells = (1 << N) ** d
        pencils = (1 << N) ** (d - 1)
        P = kp1 ** (d - 1)
        fwd = sum(q ** (m + 1) * kp1 ** (d - m) for m in range(d))  # FMAs per cell and set
        pyr = 2 * kp1 * kp1 * ((1 << (N + 1)) - 2)                  # FMAs per fiber and direction
        fma_F = cells * S * 2 * fwd + pencils * (S * P + S * P) * pyr
        fma_J = cells * S * 3 * fwd + pencils * (2 * S * P + S * P) * pyr
        # passes of the profiled steps (host-driven: the predictor's F is
        # evaluated at the first step and reused after it): in mixed mode
        # the F passes that decide (predictor, residuals after a correction)
        # run in double-float, the first residual of every step and the
        # Jacobian products in FP32; in FP64 mode every pass is FP64
        newton = ps1["newton_iters"] - ps0["newton_iters"]
        if prec == sgkiif.SGK_MIXED:
            nF_df, nF_32 = 1 + newton, args.steps
            bytes_algo = (nF_df * 2 * S * last * 8 + nF_32 * 2 * S * last * 4 + nJ * 3 * S * last * 4)
            # FP32 issue slots: one per FP32 multiply-add; a double-float
            # multiply-add is 12 FP32 operations (4 for the product, 8 for
            # the TwoSum addition; sgk_dfloat.h)
            slots = nF_df * fma_F * 12 + nF_32 * fma_F + nJ * fma_J
            flops_algo = 2.0 * slots
            pass_mix = {"double_float_F": nF_df, "fp32_F": nF_32, "fp32_J": nJ}
        else:
            nF_64 = 1 + newton + args.steps
            bytes_algo = (nF_64 * 2 * S * last + nJ * 3 * S * last) * 8
            flops_algo = 2.0 * (nF_64 * fma_F + nJ * fma_J)
            pass_mix = {"fp64_F": nF_64, "fp64_J": nJ}
    elif dominant in ("to_finest", "from_finest"):
        bytes_algo = (nF + nJ) * S * sum(sizes[i] + sizes[i + 1] for i in range(d - 1)) * elem
    elif dominant == "matvec":
        bytes_algo = nl * 2 * dof * 8
    elif dominant == "arnoldi":
        # one launch = the Arnoldi process of one exponential.  Algorithmic
        # bytes (FP64 vectors): per step j the two Gram-Schmidt passes read
        # the j + 1 basis columns twice each (V^T w, then w - V h), i.e.
        # 4 (j + 1) DOF 8 bytes, and the matvec reads x and writes y,
        # 2 DOF 8 bytes.  Arithmetic: the Gram-Schmidt passes, the norm and
        # the scaling in FP64; the matvec's multiply-adds in double-float
        # (FP32 pipe) in mixed mode, FP64 otherwise.
        M = cfg["M"]
        madds = prob.ops[0].madds()
        bytes_algo = sum(4 * (j + 1) * dof * 8 for j in range(M)) + 2 * M * dof * 8
        flops_gs = 2.0 * (sum(4 * (j + 1) * dof + 2 * dof for j in range(M)) + dof)
        flops_mv = 2.0 * M * madds
    roofline = None
    if nl > 0 and ms > 0 and (bytes_algo or flops_algo):
        t = ms / 1e3
        common = {"kernel_class": dominant, "avg_launch_us": ms / nl * 1e3, "launches": nl,
                  "share_of_profiled_step_time": ms / prof_ms,
                  "timing": "CUDA events around each launch of the class, on the library stream, over a "
                            "second pass of the same timed steps with graph replay off"}
        if dominant == "arnoldi":
            achieved = nl * bytes_algo / t / 1e9
            clock = (clk or {}).get("sm_max_mhz") or 2070.0
            fp32_peak = 152 * 128 * 2 * clock * 1e6 / 1e12
            fp64_peak = 1.25
            mixed = prec == sgkiif.SGK_MIXED
            # ALU view: time the FP64 work would take at the FP64 rate plus
            # the matvec's work at its pipe's rate (double-float: about 20
            # FP32 operations per multiply-add), as a fraction of the launch
            alu_s = flops_gs / (fp64_peak * 1e12) + (
                flops_mv / 2 * 20 / (fp32_peak * 1e12) if mixed else flops_mv / (fp64_peak * 1e12))
            roofline = dict(common, bound="hbm", achieved=achieved, peak=peaks["hbm_gbs"], unit="GB/s",
                            frac=achieved / peaks["hbm_gbs"],
                            peak_source="%s copy bandwidth (MEASURED_PEAKS.json)" % peak_kind,
                            algorithmic_bytes_per_launch=bytes_algo,
                            algorithmic_bytes_formula="sum_{j<M} 4 (j+1) DOF 8 + 2 M DOF 8",
                            alu_view={"fp64_tflops": nl * flops_gs / t / 1e12,
                                      "fp64_peak_tflops": fp64_peak,
                                      "fp64_peak_source": "nominal FP64 rate of the part (1.25 TFLOP/s)",
                                      "matvec_madds_per_launch": M * madds,
                                      "matvec_arith": "double-float on the FP32 pipe" if mixed else "FP64",
                                      "fp32_peak_tflops": fp32_peak,
                                      "fp32_peak_source": "derived: 152 SMs x 128 FP32 lanes x 2 x max SM clock",
                                      "measured_fp64_peak_tflops": alu_peaks_tflops()["fp64"],
                                      "measured_fp32_peak_tflops": alu_peaks_tflops()["fp32"],
                                      "measured_peak_method": ALU_PROBE,
                                      "busy_frac": alu_s / (t / nl)},
                            traffic=ARNOLDI_TRAFFIC.get((d, N, cfg["k"], cfg["M"], args.precision)),
                            traffic_note="dram read + write of one launch, ncu cold capture "
                                         "(profiles/arnoldi_kernel_cubic3d_l6k2_m30.md); null when no capture "
                                         "of the current kernel exists; far below the algorithmic bytes because "
                                         "the basis stays in shared memory and L2")
        elif flops_algo:
            clock = (clk or {}).get("sm_max_mhz") or 2070.0
            mixed = prec == sgkiif.SGK_MIXED
            peak = 152 * 128 * 2 * clock * 1e6 / 1e12 if mixed else 1.25
            achieved = flops_algo / t / 1e12
            meas = alu_peaks_tflops()["fp32" if mixed else "fp64"]
            roofline = dict(common, bound="alu", achieved=achieved, peak=peak, unit="TFLOP/s",
                            frac=achieved / peak, passes=pass_mix,
                            measured_peak=meas, frac_of_measured=achieved / meas, measured_peak_method=ALU_PROBE,
                            work_model="FP32-pipe flops: 2 per FP32 multiply-add, 24 per double-float "
                                       "multiply-add (12 FP32 operations); algorithmic multiply-adds of the "
                                       "sum-factorised quadrature and the two-scale pyramids of the last "
                                       "direction (the kernel's even and odd sums do about half of them)" if mixed else "FP64 flops, 2 per multiply-add",
                            peak_source="derived: 152 SMs x 128 FP32 lanes x 2 flop x max SM clock" if mixed
                            else "nominal FP64 rate of the part (1.25 TFLOP/s)",
                            algorithmic_flops_per_launch=flops_algo / nl,
                            algorithmic_bytes_per_launch=bytes_algo / nl,
                            hbm_view={"achieved_gbs": bytes_algo / t / 1e9, "peak_gbs": peaks["hbm_gbs"],
                                      "frac": bytes_algo / t / 1e9 / peaks["hbm_gbs"], "peak_source": peak_kind},
                            traffic=PENCIL_TRAFFIC.get((d, N, cfg["k"], args.precision)),
                            traffic_note="dram read + write of one double-float F launch, ncu cold capture "
                                         "(profiles/pencil_kernel_cubic3d_l6k2_dfloat.md); null when no capture "
                                         "of the current kernel exists")
        else:
            achieved = bytes_algo / t / 1e9
            roofline = dict(common, bound="hbm", achieved=achieved, peak=peaks["hbm_gbs"], unit="GB/s",
                            frac=achieved / peaks["hbm_gbs"], traffic=None, peak_source=peak_kind,
                            algorithmic_bytes_per_launch=bytes_algo / nl)

    # the persistent Arnoldi kernel's own roofline when another class leads:
    # the HBM fraction of its algorithmic vector bytes per launch (one
    # exponential), sum_{j<M} 4 (j+1) DOF 8 + 2 M DOF 8
    roofline_arnoldi = None
    ams, anl = kprof.get("arnoldi", (0.0, 0))
    if dominant != "arnoldi" and anl > 0 and ams > 0:
        M = cfg["M"]
        abytes = sum(4 * (j + 1) * dof * 8 for j in range(M)) + 2 * M * dof * 8
        aach = anl * abytes / (ams / 1e3) / 1e9
        roofline_arnoldi = {"kernel_class": "arnoldi", "avg_launch_us": ams / anl * 1e3, "launches": anl,
                            "bound": "hbm", "achieved": aach, "peak": peaks["hbm_gbs"], "unit": "GB/s",
                            "frac": aach / peaks["hbm_gbs"], "peak_source": peak_kind,
                            "algorithmic_bytes_per_launch": abytes,
                            "traffic": ARNOLDI_TRAFFIC.get((d, N, cfg["k"], cfg["M"], args.precision)),
                            "note": "latency-bound (grid barriers); the basis stays in shared memory and L2, "
                                    "so DRAM traffic is far below the algorithmic bytes"}

    out = {"metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps,
           "warmup": args.warmup, "ms_per_step": total_ms / args.steps, "higher_is_better": True,
           "scaling": "weak", "vs_baseline": None,
           "dtype": "f64 + double-float (f32 pairs) + f32 Jacobian products" if prec == sgkiif.SGK_MIXED else "f64",
           "data": "synthetic (seeded Fourier-mode initial data)",
           "config": native_config(cfg, args.precision, world),
           "rel_l2_vs_oracle": acc_oracle,
           "rel_l2_vs_oracle_note": "final state after the timed steps against the FP64 oracle's state after "
                                    "the same steps (tests/golden/cubic3d_steps.npz); null when no stored state "
                                    "exists for this step count",
           "rel_l2_vs_fp64_gpu": acc,
           "e2e": e2e, "gpu_launches": launches, "roofline": roofline, "roofline_arnoldi": roofline_arnoldi,
           "clocks": clk, "device": device_info(),
           "host_wall_s": wall,
           "profiled_pass_ms_per_step": prof_ms / args.steps,
           "solver": {"newton_iters": st1["newton_iters"] - st0["newton_iters"],
                      "inner_iters": nJ, "last_m_eff": st1["last_m_eff"],
                      "max_krylov_err_est": st1["max_krylov_err_est"]},
           "kernel_ms_per_step": {c: round(v[0] / args.steps, 4) for c, v in kprof.items() if v[1] > 0}}
    prob.close()
    legs = {}  # host wall seconds of every leg after the headline one

    def leg(name, fn):
        # a leg that raises is reported in the line; the headline stands
        t0 = time.perf_counter()
        try:
            out[name] = fn()
        except Exception as e:  # noqa: BLE001
            out[name] = {"error": "%s: %s" % (type(e).__name__, e)}
        legs[name] = round(time.perf_counter() - t0, 1)

    if world == 1 and not args.no_matvec:
        leg("matvec", lambda: matvec_leg(peaks, peak_kind))
    if world == 1 and not args.no_iif3:
        leg("iif3", lambda: iif3_leg(cfg, args))
    if world == 1 and not args.no_schnak:
        leg("schnak2d", lambda: schnak_leg(args))
    if world == 1 and not args.no_sparse_reaction:
        leg("sparse_reaction", lambda: guarded_leg(sparse_reaction_leg, cfg, args, peaks, peak_kind))
    if args.batch_instances > 0:
        leg("batched", lambda: batched_leg(args, dist, rank, world))
    if world == 1 and args.served_requests > 0:
        leg("served", lambda: served_leg(args))
    if world == 1 and args.served_requests > 0 and not args.no_sparse_reaction:
        leg("served_sparse_reaction", lambda: guarded_leg(served_sparse_leg, args))
    if world == 1 and args.batch_instances > 0 and not args.no_sparse_reaction:
        leg("batched_sparse_reaction", lambda: guarded_leg(batched_sparse_leg, args))
    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        leg("cpu_baseline", lambda: cpu_baseline(cfg, args.steps))
    out["leg_wall_s"] = legs
    if dist is not None:
        dist.destroy_process_group()
    return out


# ------------------------------------------------------------- IIF3 leg ---

def iif3_leg(cfg, args):
    """The same workload stepped with IIF3 (eq. krylov6: a second Krylov
    projection over 2 dt per step, Newton weight 5/12 dt; the first step is
    IIF2), in mixed precision, device-timed over K steps from the initial
    state with the L2 flushed before each, and its distance to the FP64
    IIF3 path after those steps.  IIF3 steps are host-driven (one graph per
    phase instead of one per step)."""
    import torch
    from paper_1810_11111_gb300 import sgkiif
    from paper_1810_11111_gb300.runner import Problem
    dev = torch.device("cuda", torch.cuda.current_device())
    stream = torch.cuda.current_stream(dev)
    c3 = dict(cfg, scheme=sgkiif.SGK_IIF3)
    flush = torch.empty(64 * 1024 * 1024, dtype=torch.float32, device=dev)
    out = {"workload": "as the headline, scheme IIF3", "steps": args.steps}
    states = {}
    for name, prec in (("mixed", sgkiif.SGK_MIXED), ("fp64", sgkiif.SGK_FP64)):
        prob = Problem(c3, prec)
        prob.reset()
        prob.solver.step(2)  # graph capture of every phase outside the timing
        prob.reset()
        e0 = torch.cuda.Event(enable_timing=True)
        e1 = torch.cuda.Event(enable_timing=True)
        tot = 0.0
        for i in range(args.steps):
            flush.fill_(float(i))
            e0.record(stream)
            prob.solver.step(1)
            e1.record(stream)
            e1.synchronize()
            tot += e0.elapsed_time(e1)
        states[name] = prob.state()
        out[name] = {"ms_per_step": tot / args.steps,
                     "dof_steps_per_s": prob.dof * prob.nspecies * args.steps / (tot / 1e3)}
        prob.close()
    num = sum(float(np.sum((states["mixed"][s] - states["fp64"][s]) ** 2)) for s in range(len(states["fp64"])))
    den = sum(float(np.sum(states["fp64"][s] ** 2)) for s in range(len(states["fp64"])))
    out["rel_l2_mixed_vs_fp64"] = float(np.sqrt(num / den))
    return out



# ------------------------------- sparse-grid interpolation form of F ---

def guarded_leg(fn, *a):
    """A leg of the interpolation form; an exception is reported in the
    line instead of ending the run."""
    try:
        return fn(*a)
    except Exception as e:  # noqa: BLE001
        return {"error": "%s: %s" % (type(e).__name__, e)}


def sparse_reaction_leg(cfg, args, peaks, peak_kind):
    """The headline workload with the sparse-grid interpolation form of the
    reaction term (SGK_REACTION_INTERP: F_I = C^{-1} f(C U) by 4d direction
    passes, the implicit stage solved pointwise at the collocation points; a
    deviation from the paper's finest-grid F for its first stated future
    direction).  K steps from the initial state, queued, device-timed with the
    L2 flushed before each, in both precisions; accuracy against the
    oracle's stored run of the same form (tests/golden/cubic3d_interp_steps.npz),
    and its distance to the paper's form (the quadrature oracle's state): the
    difference between the two discretisations, not an error of either."""
    import torch
    from paper_1810_11111_gb300 import sgkiif
    from paper_1810_11111_gb300.runner import Problem
    dev = torch.device("cuda", torch.cuda.current_device())
    stream = torch.cuda.current_stream(dev)
    ci = dict(cfg, reaction_form="interp")
    flush = torch.empty(64 * 1024 * 1024, dtype=torch.float32, device=dev)
    out = {"workload": "as the headline, reaction term in the sparse-grid interpolation form", "steps": args.steps}
    states, prof = {}, None
    for name, prec in (("mixed", sgkiif.SGK_MIXED), ("fp64", sgkiif.SGK_FP64)):
        prob = Problem(ci, prec)
        prob.reset()
        prob.solver.step(1)
        prob.reset()
        ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(args.steps)]
        l0 = prob.ctx.launches
        for i in range(args.steps):
            flush.fill_(float(i))
            ev[i][0].record(stream)
            prob.solver.step_async(1)
            ev[i][1].record(stream)
        prob.solver.wait()
        torch.cuda.synchronize(dev)
        tot = sum(a.elapsed_time(b) for a, b in ev)
        launches = prob.ctx.launches - l0
        states[name] = prob.state()
        st = prob.solver.stats()
        out[name] = {"ms_per_step": tot / args.steps,
                     "dof_steps_per_s": prob.dof * prob.nspecies * args.steps / (tot / 1e3),
                     "gpu_launches": launches, "pointwise_newton_corrections": st["newton_iters"]}
        if name == "mixed":
            # kernel classes over the same steps, each launch event-timed
            prob.ctx.profile(0xFF)
            prob.reset()
            for i in range(args.steps):
                flush.fill_(float(i))
                prob.solver.step(1)
            torch.cuda.synchronize(dev)
            kp = prob.ctx.profile_read()
            prob.ctx.profile(0)
            names = {"to_finest": "to_points", "from_finest": "from_points", "cell_quadrature": "point_kernels"}
            prof = {names.get(c, c): (v[0] / args.steps, v[1] / args.steps) for c, v in kp.items() if v[1] > 0}
        prob.close()
    out["kernel_ms_per_step"] = {c: round(v[0], 4) for c, v in prof.items()}
    # the transform passes: algorithmic bytes of one direction pass = read and
    # write the vectors it maps (DOF x 8 B each way per vector); latency-bound
    # at this size (the vectors stay in L2)
    dof = sgkiif.dof_of(cfg["d"], cfg["n"], cfg["k"])
    tp_ms = prof.get("to_points", (0, 0))[0] + prof.get("from_points", (0, 0))[0]
    tp_n = prof.get("to_points", (0, 0))[1] + prof.get("from_points", (0, 0))[1]
    out["transform_passes"] = {"ms_per_step": tp_ms, "launch_groups_per_step": tp_n,
                               "dof": dof, "passes_per_application": 2 * cfg["d"]}
    for key, golden, form in (("rel_l2_vs_oracle", "cubic3d_interp_steps.npz", "interp"),
                              ("rel_l2_vs_quadrature_form_oracle", "cubic3d_steps.npz", "quadrature")):
        path = os.path.join(ROOT, "tests", "golden", golden)
        out[key] = None
        if os.path.exists(path):
            g = np.load(path)
            k = "U%d" % args.steps
            if k in g.files:
                out[key] = {p: float(np.linalg.norm(states[p][0] - g[k][0]) / np.linalg.norm(g[k][0]))
                            for p in states}
    out["note"] = ("rel_l2_vs_quadrature_form_oracle is the distance between the two discretisations of F "
                   "(interpolation error of f(u_h) amplified over the steps), not a parity figure")
    return out


def served_sparse_leg(args):
    """The served draws (seed 4) with the interpolation form of F and no
    finest-grid cap: every draw is admitted (the form holds only sparse-grid
    vectors).  All requests submitted at t = 0 (the server's capacity) and
    one at a time; mixed precision."""
    from paper_1810_11111_gb300 import sgkiif, workloads
    reqs, rejected = workloads.served_requests(count=args.served_requests, seed=4, max_nodal_bytes=float("inf"))
    reqs = [dict(r, reaction_form="interp") for r in reqs]
    work = [sgkiif.dof_of(r["d"], r["n"], r["k"]) * len(r["kappas"]) * r["steps"] for r in reqs]
    caps = [4 * sgkiif.dof_of(r["d"], r["n"], r["k"]) for r in reqs]
    fails = []

    def run(workers, at_once):
        srv = sgkiif.Server(0, workers=workers, engine=True)
        t0 = time.perf_counter()
        lat = []
        if at_once:
            tickets = [srv.submit(r, sgkiif.SGK_MIXED) for r in reqs]
            infos = [srv.wait(t, cap=c)[1] for t, c in zip(tickets, caps)]
        else:
            infos = [srv.wait(srv.submit(r, sgkiif.SGK_MIXED), cap=c)[1] for r, c in zip(reqs, caps)]
        wall = time.perf_counter() - t0
        for i, info in enumerate(infos):
            lat.append(info["latency_ms"])
            if info["status"] != sgkiif.SGK_OK:
                q = reqs[i]
                fails.append("request %d (%s, d %d, level %d, degree %d): status %d: %s after %d steps"
                             % (i, q["name"], q["d"], q["n"], q["k"], info["status"], info["error"], info["steps"]))
        st = srv.stats()
        srv.close()
        lat = np.sort(np.asarray(lat))
        return {"p50_ms": float(np.percentile(lat, 50)), "p99_ms": float(np.percentile(lat, 99)),
                "dof_steps_per_s": float(sum(work) / wall), "wall_s": wall, "max_concurrent": st["max_concurrent"]}

    srv = sgkiif.Server(0, workers=1)
    for r in reqs:  # first-use costs of every shape
        srv.wait(srv.submit(dict(r, steps=1), sgkiif.SGK_MIXED))
    srv.close()
    sat = run(args.served_workers, True)
    one = run(1, False) if args.full_comparisons else None
    return {"workload": "served draws (seed 4, %d requests; d 3-4, level 6-9, degree 1-3, cubic or Schnakenberg, "
                        "10-100 IIF2 steps) with the interpolation form of F; no finest-grid cap: %d of %d draws "
                        "rejected" % (len(reqs), rejected, len(reqs) + rejected),
            "largest_dof": max(sgkiif.dof_of(r["d"], r["n"], r["k"]) for r in reqs),
            "dof_steps_total": int(sum(work)), "precision": "mixed", "saturation": sat, "one_at_a_time": one,
            "saturation_vs_one_at_a_time": sat["dof_steps_per_s"] / one["dof_steps_per_s"] if one else None,
            "failed_requests": len(fails), "first_failure": fails[0] if fails else None}


def batched_sparse_leg(args):
    """The batch draws (seed 3, 256 instances) with the interpolation form of
    F and no finest-grid cap (none rejected), one untimed step then 5 timed
    batch steps, mixed precision; with --full-comparisons the FP64 run of
    the same batch gives the per-instance mixed error."""
    import torch
    from paper_1810_11111_gb300 import sgkiif, workloads
    insts, rejected = workloads.batch_instances(count=args.batch_instances, seed=3, max_nodal_bytes=float("inf"))
    insts = [dict(c, reaction_form="interp") for c in insts]
    work = sum(sgkiif.dof_of(c["d"], c["n"], c["k"]) for c in insts)
    steps = 5
    res, states = {}, {}
    runs = (("mixed", sgkiif.SGK_MIXED), ("fp64", sgkiif.SGK_FP64))
    for name, prec in runs if args.full_comparisons else runs[:1]:
        b = sgkiif.Batch(0, streams=8)
        for c in insts:
            b.add(c, prec)
        rc0, _ = b.step(1)
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        rc, st = b.step(steps)
        wall = time.perf_counter() - t0
        states[name] = [np.concatenate(b.state(i)) for i in range(len(insts))]
        res[name] = {"dof_steps_per_s": work * steps / wall, "wall_s": wall,
                     "failed": sum(1 for x in st if x != sgkiif.SGK_OK), "status": max(rc0, rc),
                     "batched_arnoldi_launches": b.launches()}
        b.close()
    errs = np.array([float(np.linalg.norm(m - f) / max(np.linalg.norm(f), 1e-300))
                     for m, f in zip(states["mixed"], states["fp64"])]) if "fp64" in states else None
    return {"workload": "batch draws (seed 3, %d scalar cubic instances; d 2-4, level 5-8, degree 1-2) with the "
                        "interpolation form of F; no finest-grid cap: %d rejected" % (len(insts), rejected),
            "dof_total": work, "largest_dof": max(sgkiif.dof_of(c["d"], c["n"], c["k"]) for c in insts),
            "steps": steps, "untimed_first_steps": 1, "mixed": res["mixed"], "fp64": res.get("fp64"),
            "rel_l2_mixed_vs_fp64": {"median": float(np.median(errs)), "max": float(errs.max()),
                                     "above_1e-6": int((errs > 1e-6).sum())} if errs is not None else
            "FP64 run with --full-comparisons",
            "timing": "host wall clock around the batch steps"}


# ------------------------------------------------- two-species leg ---

def schnak_leg(args):
    """The two-species Schnakenberg workload at its configured size (d = 2,
    level 8, degree 2, 11 520 coefficients per species, kappa 0.01 / 0.5,
    M = 40, dt = 0.05, 200 IIF2 steps; Newton with GMRES, host-driven
    steps), mixed and FP64, device-timed over all 200 steps; the mixed
    state after 10 steps against the oracle's (tests/golden/schnak2d_steps.npz)
    and after 200 steps against the FP64 GPU path."""
    import torch
    from paper_1810_11111_gb300 import sgkiif, workloads
    from paper_1810_11111_gb300.runner import Problem
    dev = torch.device("cuda", torch.cuda.current_device())
    stream = torch.cuda.current_stream(dev)
    cfg = workloads.schnak2d()
    nsteps = cfg["steps"]
    golden = os.path.join(ROOT, "tests", "golden", "schnak2d_steps.npz")
    g = np.load(golden) if os.path.exists(golden) else None
    out = {"workload": "schnak2d: u_t = 0.01 Lap u + 0.1 - u + u^2 v, v_t = 0.5 Lap v + 0.9 - u^2 v, periodic, "
                       "level 8, degree 2, M 40, dt 0.05, %d IIF2 steps (GMRES)" % nsteps}
    finals = {}
    for name, prec in (("mixed", sgkiif.SGK_MIXED), ("fp64", sgkiif.SGK_FP64)):
        prob = Problem(cfg, prec)
        prob.reset()
        prob.solver.step(1)  # graph capture of every phase
        prob.reset()
        prob.solver.step(10)
        if g is not None:
            want = g["U10"]
            got = np.stack(prob.state())
            out[name + "_rel_l2_vs_oracle_step10"] = float(np.linalg.norm(got - want) / np.linalg.norm(want))
        prob.reset()
        e0 = torch.cuda.Event(enable_timing=True)
        e1 = torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        e0.record(stream)
        prob.solver.step(nsteps)
        e1.record(stream)
        e1.synchronize()
        ms = e0.elapsed_time(e1)
        finals[name] = np.concatenate(prob.state())
        st = prob.solver.stats()
        out[name] = {"ms_per_step": ms / nsteps, "dof_steps_per_s": prob.dof * 2 * nsteps / (ms / 1e3),
                     "newton_iters": st["newton_iters"], "inner_iters": st["inner_iters"],
                     "max_krylov_err_est": st["max_krylov_err_est"]}
        prob.close()
    out["rel_l2_mixed_vs_fp64_after_%d_steps" % nsteps] = float(
        np.linalg.norm(finals["mixed"] - finals["fp64"]) / np.linalg.norm(finals["fp64"]))
    return out


# ------------------------------------------------------ measured peaks ---

def device_info():
    """Name, SM count and L2 size of the device the bench ran on."""
    import torch
    p = torch.cuda.get_device_properties(torch.cuda.current_device())
    return {"name": p.name, "sms": p.multi_processor_count,
            "l2_bytes": getattr(p, "L2_cache_size", None), "hbm_bytes": p.total_memory}


_ALU = {}


def alu_peaks_tflops():
    """FMA peaks of the FP32 and FP64 pipes measured on this device by the
    library's probe kernel (sgk_alu_peak: independent FMA chains, best of 5
    launches), in TFLOP/s; taken once, outside every timed region."""
    if not _ALU:
        from paper_1810_11111_gb300 import sgkiif
        import torch
        dev = torch.cuda.current_device()
        _ALU["fp32"] = sgkiif.alu_peak(dev, "fp32") / 1e12
        _ALU["fp64"] = sgkiif.alu_peak(dev, "fp64") / 1e12
    return _ALU


ALU_PROBE = "sgk_alu_peak: 8 independent FMA chains per thread, 8 CTAs of 256 threads per SM, best of 5 launches"


# ----------------------------------------------------------- matvec leg ---

def matvec_leg(peaks, peak_kind):
    """The stand-alone sparse-grid matvec (sgk_matvec, one launch for all
    directions) on the largest served shape, d = 4, level 9, degree 3
    (6.8 M coefficients, 55 MB per FP64 vector), L2 flushed before every
    launch.  Against the FP64 (nominal 1.25 TFLOP/s) and FP32 (152 x 128 x 2
    x 2.07 GHz) rates and the measured HBM copy bandwidth."""
    import torch
    from paper_1810_11111_gb300 import sgkiif
    dev = torch.device("cuda", torch.cuda.current_device())
    stream = torch.cuda.current_stream(dev)
    ctx = sgkiif.Context(dev.index, stream.cuda_stream, sgkiif.SGK_FP64)
    idx = sgkiif.IndexSet(ctx, 4, 9, 3)
    op = sgkiif.Operator(ctx, idx, [1.0, 0.5, 0.1, 0.7])
    dof, madds = idx.dof, op.madds()
    flush = torch.empty(64 * 1024 * 1024, dtype=torch.float32, device=dev)
    g = torch.Generator(device="cpu").manual_seed(5)
    out = {"workload": "sparse-grid matvec, d 4, level 9, degree 3, diag(1, 0.5, 0.1, 0.7), periodic",
           "dof": dof, "madds_per_matvec": madds, "l2": "flushed (256 MB write) before every launch"}
    for name, prec, dt, peak in (("fp64", sgkiif.SGK_FP64, torch.float64, 1.25),
                                 ("fp32", sgkiif.SGK_MIXED, torch.float32, 152 * 128 * 2 * 2.07e9 / 1e12)):
        x = torch.randn(dof, dtype=torch.float64, generator=g).to(dev).to(dt)
        y = torch.empty_like(x)
        for _ in range(2):
            op.matvec(x.data_ptr(), y.data_ptr(), prec)
        e0 = torch.cuda.Event(enable_timing=True)
        e1 = torch.cuda.Event(enable_timing=True)
        tot = 0.0
        reps = 10
        for i in range(reps):
            flush.fill_(float(i))
            e0.record(stream)
            op.matvec(x.data_ptr(), y.data_ptr(), prec)
            e1.record(stream)
            e1.synchronize()
            tot += e0.elapsed_time(e1)
        t = tot / reps / 1e3
        es = x.element_size()
        tf = 2.0 * madds / t / 1e12
        gbs = 2.0 * dof * es / t / 1e9
        meas = alu_peaks_tflops()[name]
        out[name] = {"us_per_matvec": t * 1e6, "achieved_tflops": tf, "peak_tflops": peak, "frac_alu": tf / peak,
                     "measured_peak_tflops": meas, "frac_alu_of_measured": tf / meas, "measured_peak_method": ALU_PROBE,
                     "algorithmic_gbs": gbs, "hbm_peak_gbs": peaks["hbm_gbs"], "frac_hbm": gbs / peaks["hbm_gbs"],
                     "hbm_peak_source": peak_kind}
    out["bound"] = "FP64 pipe (the part's FP64 rate is ~50x below what HBM feeds at this arithmetic intensity)"
    op.close()
    idx.close()
    ctx.close()
    return out


# ------------------------------------------------------- conditioning ---

def fp64_sensitivity(cfg, steps, seed=31, substeps=1):
    """Relative change of the FP64 GPU result after `steps` IIF2 steps when
    the initial state is perturbed by 1e-14 relative (seeded): how far
    rounding at that level moves the answer of this instance."""
    from paper_1810_11111_gb300 import sgkiif
    from paper_1810_11111_gb300.runner import Problem
    rng = np.random.default_rng(seed)
    outs = []
    for perturb in (False, True):
        p = Problem(cfg, sgkiif.SGK_FP64)
        p.solver.set_krylov_substeps(substeps)
        p.reset()
        if perturb:
            for s_ in range(p.nspecies):
                u = p.U0[s_].cpu().numpy()
                p.solver.set_state(s_, u * (1.0 + 1e-14 * rng.standard_normal(u.shape)))
        p.solver.step(steps)
        outs.append(np.concatenate(p.state()))
        p.close()
    return float(np.linalg.norm(outs[1] - outs[0]) / max(np.linalg.norm(outs[0]), 1e-300))


def with_substeps(cfg, steps, substeps):
    """The instance solved alone in both precisions with every exponential
    taken as `substeps` sub-projections: mixed vs FP64, the FP64 result's
    sensitivity to a 1e-14 input perturbation, and the largest Krylov error
    estimate of the FP64 run."""
    from paper_1810_11111_gb300 import sgkiif
    from paper_1810_11111_gb300.runner import Problem
    outs, est = {}, None
    for prec in (sgkiif.SGK_FP64, sgkiif.SGK_MIXED):
        p = Problem(cfg, prec)
        p.solver.set_krylov_substeps(substeps)
        p.reset()
        p.solver.step(steps)
        outs[prec] = np.concatenate(p.state())
        if prec == sgkiif.SGK_FP64:
            est = p.solver.stats()["max_krylov_err_est"]
        p.close()
    f, m = outs[sgkiif.SGK_FP64], outs[sgkiif.SGK_MIXED]
    return {"substeps": substeps, "krylov_err_est": est,
            "rel_l2_mixed_vs_fp64": float(np.linalg.norm(m - f) / max(np.linalg.norm(f), 1e-300)),
            "fp64_change_under_1e-14_input_perturbation": fp64_sensitivity(cfg, steps, substeps=substeps)}


# ---------------------------------------------------------- batched leg ---

def batched_leg(args, dist=None, rank=0, world=1):
    """Independent scalar cubic instances of uneven size (seed 3) stepped
    together through sgk_batch_*, against the same batch on one stream, and
    the per-instance error of the mixed path against the FP64 path.  With
    several ranks, each rank steps its share of the instances (the library's
    cost-based partition, no collective on the data path) and the throughput
    is the DOF x steps of all ranks over the slowest rank's wall time.

    Conditioning: each instance's FP64 run is repeated from its initial
    state perturbed by 1e-14 relative (seeded); the relative change of the
    FP64 result measures how far rounding at that level moves the answer.
    An instance whose FP64 result moves by more than 1e-8 is reported as
    ill-conditioned at this precision: no two implementations that round
    differently (the oracle included) agree on it to 1e-6."""
    import torch
    from paper_1810_11111_gb300 import sgkiif, sharding, workloads
    insts, rejected = workloads.batch_instances(count=args.batch_instances, seed=3, max_nodal_bytes=256 << 20)
    total = len(insts)
    mine = sharding.my_share(insts, rank, world, steps=1) if world > 1 else list(range(total))
    insts = [insts[i] for i in mine]
    work_per_step = sum(sgkiif.dof_of(c["d"], c["n"], c["k"]) for c in insts)
    # the configured 20 steps per instance: one untimed, then the timed ones
    steps = max(1, args.steps - 1)
    res, states, u0s = {}, {}, None
    # batched Arnoldi launches (default) and, for comparison, every instance
    # in its own whole-step graph on the same 8 streams
    runs = ((8, sgkiif.SGK_MIXED, "mixed"), (8, sgkiif.SGK_MIXED, "mixed_per_instance_graphs"),
            (8, sgkiif.SGK_FP64, "fp64"))
    if not args.full_comparisons:
        runs = (runs[0], runs[2])
    if world > 1:
        runs = runs[:1]
    # every run takes 1 + steps steps from the initial states: one untimed
    # (graph capture, first launches), then the timed ones
    for streams, prec, name in runs:
        b = sgkiif.Batch(0, streams=streams, fused=name != "mixed_per_instance_graphs")
        for c in insts:
            b.add(c, prec)
        rc, _ = b.step(1)
        torch.cuda.synchronize()
        if dist is not None:
            dist.barrier()
        t0 = time.perf_counter()
        rc2, st = b.step(steps)
        wall = time.perf_counter() - t0
        states[name] = [np.concatenate(b.state(i)) for i in range(len(insts))]
        if name == "mixed":
            kest = np.array([b.stats(i)["max_krylov_err_est"] for i in range(len(insts))])
        res[name] = dict(dof_steps_per_s=work_per_step * steps / wall, wall_s=wall,
                         failed=sum(1 for x in st if x != sgkiif.SGK_OK), status=max(rc, rc2),
                         batched_arnoldi_launches=b.launches())
        b.close()
    if world > 1:
        value, wall_max = aggregate(work_per_step * steps, res["mixed"]["wall_s"] * 1e3, dist,
                                    torch.device("cuda", torch.cuda.current_device()))
        return dict(workload="batch: %d scalar cubic instances over %d ranks (cost-based partition)" % (total, world),
                    precision="mixed", instances_this_rank=len(insts), steps=steps,
                    dof_steps_per_s=value, slowest_rank_wall_s=wall_max / 1e3, scaling="weak (instances split)")

    def rel(a, b):
        return float(np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-300))

    errs = np.array([rel(m, f) for m, f in zip(states["mixed"], states["fp64"])])
    # conditioning of the instances above the budget (each solved alone in
    # FP64 from its initial state and from a 1e-14 perturbation of it)
    sens = np.zeros(len(insts))
    for i in np.nonzero(errs > 1e-6)[0]:
        sens[i] = fp64_sensitivity(insts[i], 1 + steps)
    ill = sens > 1e-8
    well = ~ill
    return dict(workload="batch: %d scalar cubic instances (seed 3; d 2-4, level 5-8, degree 1-2, kappa_i ~ "
                         "U(0.05,1), f = -c u^3 with c ~ U(1,100), 8-mode Fourier u0; M 30, dt 0.005; draws above "
                         "256 MB of finest-grid FP64 nodal values rejected: %d of %d)"
                         % (total, rejected, total + rejected),
                precision="mixed", dof_total=work_per_step, steps=steps, untimed_first_steps=1, streams=8,
                dof_steps_per_s=res["mixed"]["dof_steps_per_s"], wall_s=res["mixed"]["wall_s"],
                batched_arnoldi_launches=res["mixed"]["batched_arnoldi_launches"],
                per_instance_graphs_dof_steps_per_s=res["mixed_per_instance_graphs"]["dof_steps_per_s"]
                if "mixed_per_instance_graphs" in res else None,
                speedup_vs_per_instance_graphs=res["mixed"]["dof_steps_per_s"] /
                res["mixed_per_instance_graphs"]["dof_steps_per_s"] if "mixed_per_instance_graphs" in res else None,
                batched_equals_per_instance_bitwise=all(
                    np.array_equal(x, y) for x, y in zip(states["mixed"], states["mixed_per_instance_graphs"]))
                if "mixed_per_instance_graphs" in res else None,
                failed_instances=res["mixed"]["failed"], fp64_dof_steps_per_s=res["fp64"]["dof_steps_per_s"],
                rel_l2_vs_fp64={"median": float(np.median(errs)), "p90": float(np.percentile(errs, 90)),
                                "max": float(errs.max()), "above_1e-6": int((errs > 1e-6).sum()),
                                "well_conditioned": int(well.sum()),
                                "max_well_conditioned": float(errs[well].max()) if well.any() else None,
                                "above_1e-6_well_conditioned": int((errs[well] > 1e-6).sum()),
                                "ill_conditioned": [{"instance": int(i), "rel_l2_mixed_vs_fp64": float(errs[i]),
                                                     "fp64_change_under_1e-14_input_perturbation": float(sens[i]),
                                                     "krylov_err_est": float(kest[i]),
                                                     "with_substeps": [with_substeps(insts[i], 1 + steps, sub)
                                                                       for sub in (8, 64)]}
                                                    for i in np.nonzero(ill)[0]],
                                "note": "per instance after the timed steps; every instance above 1e-6 is "
                                        "solved again alone in FP64 from its initial state perturbed by 1e-14 "
                                        "relative: ill-conditioned = the FP64 result itself moves by more than "
                                        "1e-8 (an M = 30 Krylov projection far from converged at dt rho(A) ~ 1e4 "
                                        "amplifies rounding-level perturbations)"},
                krylov_err_est={"median": float(np.median(kest)), "max": float(kest.max()),
                                "above_1e-6": int((kest > 1e-6).sum()),
                                "max_well_conditioned": float(kest[well].max()) if well.any() else None,
                                "note": "largest a-posteriori estimate h_{m+1,m} |[exp(dt H) e1]_m| / "
                                        "||exp(dt H) e1|| of each instance's projections over its mixed steps"},
                timing="host wall clock around the batch steps (each step waits for every stream)")


# ----------------------------------------------------------- served leg ---

def served_leg(args):
    """Poisson stream of whole solve requests through the request server
    (the engine batches the single-species requests step by step on the
    batched Arnoldi launches, workers take the systems; memory admission),
    at each arrival rate of --served-rates and all at once (saturation),
    against the same requests one at a time.  Latency is submit -> result on the host,
    measured by the server; throughput counts DOF x species x steps of all
    requests over first submission -> last completion."""
    from paper_1810_11111_gb300 import sgkiif, workloads
    reqs, rejected = workloads.served_requests(count=args.served_requests, seed=4, max_nodal_bytes=512 << 20)
    work = [sgkiif.dof_of(r["d"], r["n"], r["k"]) * len(r["kappas"]) * r["steps"] for r in reqs]

    failures = []

    kest = {}

    def record(info, i=None):
        if info["status"] != sgkiif.SGK_OK:
            failures.append("status %d: %s" % (info["status"], info["error"]))
        if i is not None:
            kest[i] = info["krylov_err_est"]
        return info["latency_ms"]

    caps = [4 * sgkiif.dof_of(r["d"], r["n"], r["k"]) for r in reqs]

    def one_at_a_time(prec, outs=None):
        srv = sgkiif.Server(0, workers=1)
        lat, t0 = [], time.perf_counter()
        for r, cap in zip(reqs, caps):
            out, info = srv.wait(srv.submit(r, prec), cap=cap)
            lat.append(record(info))
            if outs is not None:
                outs.append(out)
        wall = time.perf_counter() - t0
        srv.close()
        return lat, wall

    def summary(lat, wall):
        lat = np.sort(np.asarray(lat))
        return {"p50_ms": float(np.percentile(lat, 50)), "p99_ms": float(np.percentile(lat, 99)),
                "mean_ms": float(lat.mean()), "dof_steps_per_s": float(sum(work) / wall), "wall_s": wall}

    # warm: module loading and first-use costs of every kernel shape
    srv = sgkiif.Server(0, workers=1)
    for r in reqs:
        srv.wait(srv.submit(dict(r, steps=1), sgkiif.SGK_MIXED))
    srv.close()
    lat_m, wall_m = one_at_a_time(sgkiif.SGK_MIXED)
    mean_service_s = wall_m / len(reqs)
    capacity_rate = 1.0 / mean_service_s  # requests/s one at a time

    def serve(rate, engine=True, keep_est=False):
        """Requests arriving as a Poisson stream at `rate` per second (all at
        t = 0 when rate is None); returns summary, outputs, server stats."""
        arrivals = workloads.poisson_arrivals(len(reqs), rate, seed=4) if rate else [0.0] * len(reqs)
        srv = sgkiif.Server(0, workers=args.served_workers, engine=engine)
        t0 = time.perf_counter()
        tickets = []
        for r, ta in zip(reqs, arrivals):
            delay = ta - (time.perf_counter() - t0)
            if delay > 0:
                time.sleep(delay)
            tickets.append(srv.submit(r, sgkiif.SGK_MIXED))
        lat, outs = [], []
        for i, (t, cap) in enumerate(zip(tickets, caps)):
            out, info = srv.wait(t, cap=cap)
            lat.append(record(info, i if keep_est else None))
            outs.append(out)
        wall = time.perf_counter() - t0
        st = srv.stats()
        srv.close()
        return summary(lat, wall), outs, st

    rates = [float(x) for x in args.served_rates.split(",") if x.strip()]
    by_rate = {}
    outs_served = None
    for r_mult in rates:
        summ, outs, st = serve(r_mult * capacity_rate)
        by_rate["%gx" % r_mult] = dict(summ, rate_per_s=r_mult * capacity_rate, max_concurrent=st["max_concurrent"],
                                       peak_reserved_gb=st["peak_reserved_bytes"] / 1e9)
        if outs_served is None:
            outs_served = outs
    sat, outs_sat, st_sat = serve(None, keep_est=True)
    sat_workers = serve(None, engine=False)[0] if args.full_comparisons else None
    outs64 = []
    lat64, wall64 = one_at_a_time(sgkiif.SGK_FP64, outs64) if not args.served_no_fp64 else ([0.0], 0.0)

    def rel(m, f):
        return float(np.linalg.norm(m - f) / max(np.linalg.norm(f), 1e-300))

    errs = [rel(m, f) for m, f in zip(outs_sat, outs64) if m.size and f.size]
    over = [i for i, e in enumerate(errs) if e > 1e-6]
    # the conditioning of the requests above 1e-6 (FP64 re-solves from a
    # perturbed input and with sub-projections) runs with --full-comparisons
    ill = [{"request": i, "rel_l2_mixed_vs_fp64": errs[i],
            "fp64_change_under_1e-14_input_perturbation": fp64_sensitivity(reqs[i], reqs[i]["steps"]),
            "krylov_err_est": kest.get(i),
            "with_substeps": [with_substeps(reqs[i], reqs[i]["steps"], sub) for sub in (8, 64)]}
           for i in over] if args.full_comparisons else None
    first = by_rate["%gx" % rates[0]] if rates else sat
    base64 = summary(lat64, wall64) if not args.served_no_fp64 else None
    mixed1 = summary(lat_m, wall_m)
    return dict(first,
                workload="served: %d requests (seed 4; d 3-4, level 6-9, degree 1-3, cubic or Schnakenberg, "
                         "10-100 IIF2 steps, M 30, dt 0.005; draws above 512 MB of finest-grid FP64 nodal "
                         "values rejected: %d of %d)" % (len(reqs), rejected, len(reqs) + rejected),
                precision="mixed", workers=args.served_workers, arrival="poisson",
                offered_load="multiples of the one-at-a-time mixed capacity (%.3f requests/s)" % capacity_rate,
                by_rate=by_rate,
                saturation=dict(sat, note="every request submitted at t = 0: the server's capacity",
                                max_concurrent=st_sat["max_concurrent"]),
                saturation_workers_only=None if sat_workers is None else dict(
                    sat_workers, note="the same with the engine off: every request "
                                                               "on a worker thread"),
                one_at_a_time_mixed=mixed1,
                one_at_a_time_fp64=base64,
                speedup_vs_fp64_one_at_a_time=first["dof_steps_per_s"] / base64["dof_steps_per_s"] if base64 else None,
                saturation_vs_one_at_a_time_mixed=sat["dof_steps_per_s"] / mixed1["dof_steps_per_s"],
                failed_requests=len(failures), first_failure=failures[0] if failures else None,
                max_rel_l2_vs_fp64=max(errs) if errs else None,
                above_1e_6=len(over),
                max_rel_l2_vs_fp64_well_conditioned=max([e for i, e in enumerate(errs)
                                                        if not any(x["request"] == i and
                                                                   x["fp64_change_under_1e-14_input_perturbation"]
                                                                   > 1e-8 for x in ill)], default=None)
                if ill is not None else None,
                conditioning_of_requests_above_1e_6=ill if ill is not None else
                "not run (--full-comparisons): each request above 1e-6 re-solved in FP64 from a 1e-14-perturbed "
                "input and with 8 and 64 sub-projections",
                krylov_err_est_of_requests_above_1e_6={i: kest.get(i) for i in over},
                krylov_err_est={"median": float(np.median(list(kest.values()))) if kest else None,
                                "max": max(kest.values()) if kest else None,
                                "above_1e_6": sum(1 for v in kest.values() if v > 1e-6),
                                "note": "per request of the saturation run: the largest a-posteriori Krylov "
                                        "error estimate over its steps"},
                note="mixed results of the saturation run against the FP64 one-at-a-time results; a request "
                     "whose FP64 result moves by more than 1e-8 under a 1e-14 input perturbation is "
                     "ill-conditioned at this precision")


# --------------------------------------------------------- oracle timing ---

def oracle_steps(cfg, max_steps, budget_s):
    """Time full oracle IIF2 steps of the workload until max_steps or budget_s."""
    from oracle.iif import IIF2Solver
    from oracle.index_set import IndexSet
    from oracle.operator import sipg_1d
    from oracle.projection import project_separable
    idx = IndexSet(cfg["d"], cfg["n"], cfg["k"])
    init = cfg["init"][0]
    U = [project_separable(idx, init["amp"], init["wavenum"], init["kind"], init["const"])]
    sol = IIF2Solver(idx, sipg_1d(cfg["n"], cfg["k"]), cfg["kappas"], cfg["reaction"], cfg["dt"], cfg["M"])
    t0 = time.perf_counter()
    done = 0
    while done < max_steps and (done == 0 or time.perf_counter() - t0 < budget_s):
        U = sol.run(U, 1)
        done += 1
    return done, time.perf_counter() - t0, idx.dof


def cores():
    try:
        return len(os.sched_getaffinity(0))
    except AttributeError:
        return os.cpu_count()


def cpu_baseline(cfg, steps, budget_s=30.0):
    """The oracle on the host cores over the first of the timed GPU steps
    (from the projected initial state), a bounded sample: it stops after
    the step that crosses budget_s.  These first steps take the most Newton
    corrections of the solve, so the sample's rate is, if anything, below
    the whole solve's (`bench.py --impl reference` times all of them)."""
    done, secs, dof = oracle_steps(cfg, steps, budget_s)
    return {"value": dof * done / secs, "unit": UNIT, "cores": cores(), "kind": "oracle",
            "sample": "IIF2 steps 1..%d of the %d-step workload from the projected initial state (numpy FP64 "
                      "oracle, %.1f s; the run stops after the step that crosses %.0f s)" % (done, steps, secs,
                                                                                         budget_s)}


def native_config(cfg, precision, world):
    return dict(workload_desc(cfg), l2="flushed (256 MB write) before every timed step",
                precision=precision, parallelism="replicas" if world > 1 else "single GPU")


def reference(args, rank):
    """The oracle (numpy FP64, host cores) on the native arm's workload: W
    untimed warm-up steps from the initial state, then K timed steps from the
    initial state again (the same steps the native arm times), capped at
    150 s of timed work."""
    if rank != 0:
        return None
    cfg = workload_config()
    if args.warmup > 0:
        oracle_steps(cfg, args.warmup, 60.0)
    done, secs, dof = oracle_steps(cfg, args.steps, 150.0)
    value = dof * done / secs
    return {"impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": args.gpus,
            "steps": done, "warmup": args.warmup, "ms_per_step": secs / done * 1e3, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic (seeded Fourier-mode initial data)",
            "config": native_config(cfg, args.precision, args.gpus),
            "reference_arithmetic": "FP64 (the oracle)",
            "cpu_baseline": {"value": value, "unit": UNIT, "cores": cores(), "kind": "oracle",
                             "sample": "%d full IIF2 steps of the workload from the initial state after %d "
                                       "untimed warm-up steps (timed steps capped at 150 s)" % (done, args.warmup)},
            "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}


def main():
    args = parse()
    rank = int(os.environ.get("RANK", 0))
    world = int(os.environ.get("WORLD_SIZE", 1))
    local_rank = int(os.environ.get("LOCAL_RANK", 0))
    if args.impl == "reference":
        out = reference(args, rank)
    else:
        out = native(args, rank, world, local_rank)
    if rank == 0 and out is not None:
        print(json.dumps(out))


if __name__ == "__main__":
    main()
