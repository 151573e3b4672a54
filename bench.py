#!/usr/bin/env python
"""Benchmark of the MPFC solver: time steps/s and fine-grid cell-updates/s.

Workload (default): first-order convex-splitting scheme (Sec. 3.1) on a 1024 x 1024
periodic grid, h = 0.5, M = 1, epsilon = 0.025, beta = 0.9, s = 0.01, phi^0 =
0.07 + 0.05 U(-1, 1) (seeded), psi^0 = 0, FAS V(2,2) cycles to scaled residual 1e-10,
plain FP64.  One benchmark "step" is one time step of that solve.

Prints one JSON line (rank 0).  Timing: W warm-up steps, then K steps, each on the
device between CUDA events on the solver's stream, with a 512 MB write between steps
to flush L2 (outside the events).  Under torchrun each rank advances its own
independent instance (weak scaling, no collective on the data path); the time is the
maximum over ranks.

--impl reference times the CPU oracle (plain C, FP64; its OpenMP build on every host
core, which gives the serial oracle's bits) on the same workload.
"""
from __future__ import annotations

import argparse
import hashlib
import json
import os
import statistics
import subprocess
import sys
import tempfile
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

METRIC = "MPFC steps/s & cell-updates/s at 1024^2: plain FAS vs learned/FP32/batched, tol 1e-10"
UNIT = "steps/s"

# Instructions of one cell update of the correction form's half sweep (scheme 1): ncu's
# smsp__inst_executed.sum of k_df_smooth at 1024^2 times 32 lanes over its 2^19 cells
# (profiles/launches_correction_form_1024.md).
DF_SMOOTH_INSTR_PER_CELL = 536
# Algorithmic FP64 flops of one red-black sweep of the FP64 V-cycle per cell (scheme 1, relaxed update):
# neighbour sums 9, right-hand sides 7, Newton terms of the cubic 5, determinant 2,
# reciprocal 1, Cramer numerators 9, phi/mu products 2, kappa 2, relaxation 9.
SMOOTH_FLOPS_PER_CELL = 46
# Algorithmic bytes of one sweep per cell: read u (24) and S (24), write u (24).
SMOOTH_BYTES_PER_CELL = 72
# FP32 inner V-cycles per FP64 outer iteration of each mixed-precision workload: the
# measured best for its time step s (2 at s <= 0.01, 3 at s = 0.02 and for the pinned
# crystal, 4 for the polycrystal at s = 1; more cycles per outer iteration pay where the
# inner smoother converges more slowly per cycle).  The library's default is 2.
INNER_CYCLES = {"fp32_inner": 2, "mixed_precision_2048": 3, "neumann_polycrystal": 4, "pinning_strained_crystal": 3}


def parse_args():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=100)
    ap.add_argument("--warmup", type=int, default=10)
    ap.add_argument("--impl", choices=["ours", "reference"], default="ours")
    ap.add_argument("--size", type=int, default=1024, help="grid cells per side (workload is named by it)")
    ap.add_argument("--scheme", type=int, default=1)
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-e2e", action="store_true")
    ap.add_argument("--no-batch", action="store_true")
    ap.add_argument("--no-learned", action="store_true")
    ap.add_argument("--no-polycrystal", action="store_true")
    ap.add_argument("--no-configs", action="store_true", help="skip the second-order and mixed-precision runs")
    ap.add_argument("--profile", action="store_true", help="steps only, no flush and no extras (ncu launch list)")
    ap.add_argument("--form", choices=["fp64", "fp32", "learned"], default="fp64",
                    help="with --profile: which solver form the launch list runs")
    ap.add_argument("--profile-conv", action="store_true",
                    help="only the 32 -> 32 channel convolution of the learned guess (GELU, bf16 out), four "
                         "launches at --size^2 (ncu capture of the network's top kernel)")
    ap.add_argument("--profile-smooth", action="store_true",
                    help="only the finest-level sweep kernel, two sweeps (ncu capture of the top kernel)")
    ap.add_argument("--profile-batch", action="store_true",
                    help="only the batched form's sweep kernel: 16 instances of the --size^2 workload, default tiles, "
                         "two red-black sweeps of their finest levels (ncu capture of kb_smooth)")
    ap.add_argument("--profile-sweep32", action="store_true",
                    help="only the mixed-precision form's tiled FP32 sweep at 2048^2, two there-and-back pairs "
                         "(ncu capture of the HBM-bound kernel)")
    return ap.parse_args()


def workload(size, scheme):
    return {"workload": f"mpfc-scheme{scheme}-{size}x{size}-fp64-fas-v22", "m": size, "n": size, "h": 0.5,
            "M": 1.0, "epsilon": 0.025, "beta": 0.9, "dt": 0.01, "scheme": scheme, "tol": 1e-10,
            "cycle": "V(2,2)", "omega": 0.8, "guess": "extrapolated", "init": "0.07+0.05*U(-1,1) seed 1",
            "l2": "flushed between steps (512 MB write)"}


# ----------------------------------------------------------------------------- clocks
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
            self.proc = subprocess.Popen(["nvidia-smi", "-i", str(self.gpu), f"--query-gpu={self.FIELDS}",
                                          "--format=csv,noheader,nounits", "-lms", "200"],
                                         stdout=open(self.path, "w"), stderr=subprocess.DEVNULL)
        except Exception:
            self.proc = None

    def stop(self):
        out = {"sm_mhz": None, "sm_max_mhz": None, "reasons": [], "samples": 0}
        if self.proc is None:
            return out
        time.sleep(0.25)
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except Exception:
            self.proc.kill()
        lines = open(self.path).read().splitlines()
        os.unlink(self.path)
        return self.parse(lines)

    @staticmethod
    def parse(lines):
        """Median SM clock, maximum clock and the throttle reasons seen in nvidia-smi CSV
        lines of FIELDS (noheader, nounits)."""
        out = {"sm_mhz": None, "sm_max_mhz": None, "reasons": [], "samples": 0}
        rows = []
        for line in lines:
            parts = [x.strip() for x in line.split(",")]
            if len(parts) >= 9:
                rows.append(parts)
        if not rows:
            return out
        sm = [float(r[1]) for r in rows if r[1].replace(".", "").isdigit()]
        mx = [float(r[2]) for r in rows if r[2].replace(".", "").isdigit()]
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        reasons = set()
        for r in rows:
            for nm, v in zip(names, r[5:9]):
                if v.lower().startswith("active"):
                    reasons.add(nm)
        out.update(sm_mhz=statistics.median(sm) if sm else None, sm_max_mhz=max(mx) if mx else None,
                   reasons=sorted(reasons), samples=len(rows))
        return out


# ----------------------------------------------------------------------------- helpers
def kernel_launches_per_step(solver, scheme, cycles):
    """The library's own kernels launched by one FP64 step of `cycles` V-cycles."""
    per_step, per_cycle = solver.launch_counts(scheme)
    return per_step + cycles * per_cycle


def measured_peaks():
    """HBM GB/s and dense bf16 TFLOP/s of the GB300s from MEASURED_PEAKS.json, with
    `source` "measured"; if the file is absent, one earlier GB300 measurement ("fallback")."""
    try:
        d = json.load(open(os.path.join(ROOT, "MEASURED_PEAKS.json")))
        return {"hbm_gbs": float(d["hbm_gbs"]), "bf16_tflops": float(d["bf16_tflops"]), "source": "measured"}
    except Exception:
        return {"hbm_gbs": 6800.0, "bf16_tflops": 1900.0, "source": "fallback"}


def traffic_for(kernel, size):
    """DRAM bytes per launch from the committed ncu summary, if the kernel source it
    was taken on is unchanged; else None."""
    path = os.path.join(ROOT, "profiles", "traffic.json")
    try:
        data = json.load(open(path))
    except Exception:
        return None
    ent = data.get(kernel)
    if not ent:
        return None
    srcs = ent["source"] if isinstance(ent["source"], list) else [ent["source"]]
    h = hashlib.sha256()
    try:
        for src in srcs:
            h.update(open(os.path.join(ROOT, src), "rb").read())
    except Exception:
        return None
    digest = h.hexdigest()
    if digest != ent.get("sha256"):
        return None
    return ent["bytes_per_launch_per_cell"] * size * size


def cpu_oracle_rate(size, scheme, max_steps, budget_s, warmup=0, threaded=False):
    """The oracle as it stands on the same workload: steps/s.  Serial C on one core,
    or (threaded) its OpenMP build on every host core, which gives the same bits.
    Returns (steps/s, steps, seconds, V-cycles, threads used)."""
    import oracle
    from paper_1208_2643_gb300 import inputs
    oracle.build()
    w = workload(size, scheme)
    nthreads = oracle.threads(os.cpu_count() or 1) if threaded else 1
    sol = oracle.Solver(oracle.Params(m=size, n=size, h=w["h"], M=w["M"], eps=w["epsilon"], beta=w["beta"],
                                      s=w["dt"], omega=w["omega"]), threaded=threaded)
    sol.set_state(inputs.noise_field(size, size, 0.07, 0.05, 1))
    for _ in range(warmup):
        sol.step(scheme, tol=w["tol"], guess=oracle.GUESS_EXTRAP)
    t0 = time.perf_counter()
    done = 0
    cycles = 0
    while done < max_steps:
        r = sol.step(scheme, tol=w["tol"], guess=oracle.GUESS_EXTRAP)
        cycles += r["cycles"]
        done += 1
        if time.perf_counter() - t0 > budget_s:
            break
    dt = time.perf_counter() - t0
    return done / dt, done, dt, cycles, nthreads


def issue_peak(clk):
    """Warp instructions per second of this GPU: four sub-partitions an SM, one a cycle, at the
    median SM clock under load (the maximum where no sample was taken)."""
    import torch
    mhz = clk.get("sm_mhz") or clk.get("sm_max_mhz") or 2070.0
    return 4.0 * torch.cuda.get_device_properties(torch.cuda.current_device()).multi_processor_count * mhz * 1e6


# ----------------------------------------------------------------------------- reference arm
def conv32_timing(size, launches=10, flush_between=True):
    """The learned guess's 32 -> 32 channel convolution (GELU, bf16 out, the solver's
    inference form) on a size^2 image, timed alone with CUDA events on its stream, with
    and without an L2 flush before each launch; roofline against the measured peaks."""
    import numpy as np
    import torch
    from paper_1208_2643_gb300 import guess as gmod
    lib = gmod._lib()
    st = torch.cuda.current_stream()
    s = st.cuda_stream
    g = torch.Generator(device="cuda").manual_seed(0)
    x = torch.randn(1, size, size, 32, device="cuda", generator=g).bfloat16()
    wt = torch.randn(9, 32, 32, device="cuda", generator=g) * 0.1
    bias = torch.zeros(32, device="cuda")
    wk = torch.empty(32 * 288, dtype=torch.bfloat16, device="cuda")
    y = torch.empty(1, size, size, 32, dtype=torch.bfloat16, device="cuda")
    if lib.mpfc_cnn_pack_weights(wt.data_ptr(), 32, 32, 32, 32, 0, wk.data_ptr(), s) != 0:
        raise RuntimeError("mpfc_cnn_pack_weights failed")

    def one():
        if lib.mpfc_cnn_conv_forward(x.data_ptr(), 1, size, size, 32, wk.data_ptr(), bias.data_ptr(), 32, 32, 0,
                                     y.data_ptr(), None, None, s) != 0:
            raise RuntimeError("mpfc_cnn_conv_forward failed")

    flush = torch.empty(256 << 20, dtype=torch.uint8, device="cuda") if flush_between else None
    out = {}
    for label, use_flush in (("us_flushed", True), ("us_no_flush", False)):
        if use_flush and flush is None:
            continue
        for _ in range(3):
            one()
        ts = []
        for _ in range(launches):
            if use_flush:
                flush.zero_()
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record(st)
            one()
            e1.record(st)
            torch.cuda.synchronize()
            ts.append(e0.elapsed_time(e1) * 1e3)
        out[label] = float(np.median(ts))
    px = size * size
    flops = 2.0 * 9 * 32 * 32 * px
    bytes_ = (32 * 2 + 32 * 2) * px                 # read the bf16 input once, write the bf16 output
    peaks = measured_peaks()
    t = out.get("us_flushed", out["us_no_flush"]) * 1e-6
    out.update({"image": f"1 x {size} x {size} x 32 bf16", "tflops": flops / t / 1e12,
                f"frac_of_{peaks['source']}_bf16": flops / t / 1e12 / peaks["bf16_tflops"],
                "gbs_algorithmic": bytes_ / t / 1e9, f"frac_of_{peaks['source']}_hbm": bytes_ / t / 1e9 / peaks["hbm_gbs"],
                "bound": "neither: the single-thread MMA issue and the GELU epilogue, balanced near 1.9 k cycles per 128-pixel tile"})
    return out


def run_reference(args):
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return
    size, scheme = args.size, args.scheme
    rate, done, dt, cycles, nthr = cpu_oracle_rate(size, scheme, max(args.steps, 1), budget_s=120.0,
                                                   warmup=min(args.warmup, 1), threaded=True)
    w = workload(size, scheme)
    line = {"impl": "reference", "metric": METRIC, "value": rate, "unit": UNIT, "n_gpus": args.gpus,
            "steps": done, "warmup": min(args.warmup, 1), "ms_per_step": 1e3 * dt / done,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": w,
            "cpu_baseline": {"value": rate, "unit": UNIT, "cores": nthr, "kind": "oracle",
                             "sample": f"{done} time steps of the {size}^2 workload (time budget 120 s), "
                                       f"{cycles / done:.2f} V-cycles/step, the oracle's OpenMP build on "
                                       f"{nthr} host threads (bitwise the serial oracle)"},
            "e2e": {"value": rate, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
            "cell_updates_per_s": rate * size * size}
    print(json.dumps(line), flush=True)


# ----------------------------------------------------------------------------- our arm
def run_ours(args):
    import numpy as np
    import torch
    import torch.distributed as dist
    from paper_1208_2643_gb300 import inputs, mpfc

    from paper_1208_2643_gb300 import replicas
    rank, world, local = replicas.rank_info()
    torch.cuda.set_device(local)
    if world > 1:
        dist.init_process_group("nccl", device_id=torch.device("cuda", local))
    size, scheme = args.size, args.scheme
    w = workload(size, scheme)
    p = mpfc.default_params(m=size, n=size, h=w["h"], M=w["M"], epsilon=w["epsilon"], beta=w["beta"], dt=w["dt"],
                            tol=w["tol"], omega=w["omega"], guess=mpfc.MPFC_GUESS_EXTRAP)
    if args.profile and args.form == "fp32":
        p.precision = mpfc.MPFC_FP32_INNER
    if args.profile and args.form == "learned":
        p.guess = mpfc.MPFC_GUESS_LEARNED
    if args.profile_sweep32:
        big = mpfc.Solver(mpfc.default_params(m=2048, n=2048, h=w["h"], dt=0.02, precision=mpfc.MPFC_FP32_INNER))
        big.set_state(inputs.noise_field(2048, 2048, 0.07, 0.05, 3))
        big.set_fp32_sweep(16, 2048 * 2048)
        us = [big.fp32_time_smooth(0, 2) * 1e3 / 2 for _ in range(2)]
        big.close()
        if rank == 0:
            print(json.dumps({"profile_sweep32": True, "us_per_sweep": us}), flush=True)
        return
    if args.profile_batch:
        bq = mpfc.BatchSolver([mpfc.default_params(m=size, n=size, h=w["h"], dt=w["dt"]) for _ in range(16)])
        for i in range(16):
            bq.set_state(i, inputs.noise_field(size, size, 0.07, 0.05, 1 + i))
        ms = bq.time_smooth(scheme, 0, reps=1)
        bq.close()
        if rank == 0:
            print(json.dumps({"profile_batch": True, "ms": ms}), flush=True)
        return
    if args.profile_conv:
        r = conv32_timing(size, launches=4, flush_between=False)
        if rank == 0:
            print(json.dumps({"profile_conv": True, "us": r["us_no_flush"]}), flush=True)
        return
    stream = torch.cuda.Stream()
    torch.cuda.set_stream(stream)
    solver = mpfc.Solver(p, stream=stream)
    if args.profile and args.form == "learned":
        from paper_1208_2643_gb300 import guess as gmod
        gmod.attach(solver, gmod.load())
    phi0 = inputs.noise_field(size, size, 0.07, 0.05, replicas.instance_seed(1, rank))
    solver.set_state(phi0)
    if args.profile_smooth:
        phik, _, _ = solver.get_state(device=True)
        S = solver.op_source(scheme, phik, phik, torch.zeros_like(phik))
        u = [phik.clone(), torch.zeros_like(phik), torch.zeros_like(phik)]
        solver.op_smooth(scheme, 0, u, S, phik if scheme == 2 else None, 2)
        torch.cuda.synchronize()
        if rank == 0:
            print(json.dumps({"profile_smooth": True}), flush=True)
        return
    if args.profile:
        solver.set_launch_mode(mpfc.MPFC_LAUNCH_STREAM)   # profilers cannot see inside conditional graph nodes
    solver.step(scheme, max(args.warmup, 0))

    flush = torch.empty(512 * 1024 * 1024 // 4, dtype=torch.float32, device="cuda")

    def timed_steps(slv, K, warm, sch=None):
        """K steps of slv, each between events on the stream, L2 flushed in between."""
        sch = scheme if sch is None else sch
        slv.step(sch, warm)
        st = [torch.cuda.Event(enable_timing=True) for _ in range(K)]
        en = [torch.cuda.Event(enable_timing=True) for _ in range(K)]
        torch.cuda.synchronize()
        for k in range(K):
            flush.fill_(float(k))
            st[k].record(stream)
            slv.step_async(sch, 1)
            en[k].record(stream)
        torch.cuda.synchronize()
        rc_, recs_, _ = slv.records(max(K, 1))
        if rc_ != mpfc.MPFC_OK:
            raise mpfc.MPFCError(rc_, "timed steps")
        return sum(a.elapsed_time(b) for a, b in zip(st, en)), recs_

    K = args.steps
    starts = [torch.cuda.Event(enable_timing=True) for _ in range(K)]
    ends = [torch.cuda.Event(enable_timing=True) for _ in range(K)]
    clocks = ClockSampler(local)
    if world > 1:
        dist.barrier()
    torch.cuda.synchronize()
    clocks.start()
    for k in range(K):
        if not args.profile:
            flush.fill_(float(k))
        starts[k].record(stream)
        solver.step_async(scheme, 1)
        ends[k].record(stream)
    torch.cuda.synchronize()
    clk = clocks.stop()
    rc, recs, count = solver.records(max(K, 1))
    if rc != mpfc.MPFC_OK:
        raise mpfc.MPFCError(rc, "timed steps")
    recs_main = recs
    ms = replicas.job_time_ms(sum(s.elapsed_time(e) for s, e in zip(starts, ends)), device="cuda")
    if world > 1:
        dist.barrier()
    cycles = [r["cycles"] for r in recs]
    steps_per_s = replicas.throughput(K, world, ms)
    # counted for the FP64 step (the headline); the profiling forms (--form fp32|learned) have none
    launches = (sum(kernel_launches_per_step(solver, scheme, c) for c in cycles)
                if args.form == "fp64" else None)

    if args.profile:
        if rank == 0:
            print(json.dumps({"profile_run": True, "ms": ms, "cycles": cycles[:5]}), flush=True)
        return

    # dominant kernel: the finest level's red-black sweep in float-float, timed through the batch's
    # sweep timer on one instance (the cell function of the step's k_df_smooth, two launches)
    from paper_1208_2643_gb300 import tuning
    one = mpfc.BatchSolver([p], stream=stream)
    one.set_state(0, phi0)
    tuning.autotune(one, scheme, reps=2)
    df_sweep_ms = one.time_smooth(scheme, 0, reps=50)
    one.close()
    df_winstr = DF_SMOOTH_INSTR_PER_CELL * size * size / 32.0 / (df_sweep_ms * 1e-3)

    # the FP64 V-cycle's sweep (steps outside the correction form's range), on the solver's stream
    phik, _, _ = solver.get_state(device=True)
    S = solver.op_source(scheme, phik, phik, torch.zeros_like(phik))
    u = [phik.clone(), torch.zeros_like(phik), torch.zeros_like(phik)]
    reps = 20
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    _check = mpfc._check
    for it in range(2):
        flush.fill_(1.0)
        e0.record(stream)
        _check(solver.lib.mpfc_op_smooth(solver.h, scheme, 0, u[0].data_ptr(), u[1].data_ptr(), u[2].data_ptr(),
                                         S[0].data_ptr(), S[1].data_ptr(), S[2].data_ptr(),
                                         phik.data_ptr() if scheme == 2 else None, reps), "smooth")
        e1.record(stream)
        torch.cuda.synchronize()
    sweep_ms = e0.elapsed_time(e1) / reps
    fp64_peak = mpfc.probe_fp64_tflops(stream)
    achieved = SMOOTH_FLOPS_PER_CELL * size * size / (sweep_ms * 1e-3) / 1e12
    achieved_gbs = SMOOTH_BYTES_PER_CELL * size * size / (sweep_ms * 1e-3) / 1e9
    # context: the same sweep on a 4096^2 grid, where each launch's ramp-up and drain are
    # a small part of it (the kernel's steady state); not the headline workload
    steady = None
    if size < 4096:
        big = mpfc.Solver(mpfc.default_params(m=4096, n=4096, h=w["h"], dt=w["dt"]), stream=stream)
        ub = [inputs.noise_field_torch(4096, 4096, 0.07, 0.05, 1), inputs.noise_field_torch(4096, 4096, 0.0, 1.0, 2),
              inputs.noise_field_torch(4096, 4096, 0.0, 1.0, 3)]
        Sb = [inputs.noise_field_torch(4096, 4096, 0.0, 1.0, 4 + i) for i in range(3)]
        argsb = [x.data_ptr() for x in ub] + [x.data_ptr() for x in Sb] + [None]
        torch.cuda.synchronize()
        for it in range(2):
            e0.record(stream)
            _check(big.lib.mpfc_op_smooth(big.h, 1, 0, *argsb, 4), "smooth 4096")
            e1.record(stream)
            torch.cuda.synchronize()
        ms_b = e0.elapsed_time(e1) / 4
        steady = {"size": 4096, "sweep_ms": ms_b,
                  "achieved": SMOOTH_FLOPS_PER_CELL * 4096 * 4096 / (ms_b * 1e-3) / 1e12,
                  "frac": SMOOTH_FLOPS_PER_CELL * 4096 * 4096 / (ms_b * 1e-3) / 1e12 / fp64_peak,
                  "note": "scheme 1, 4 sweeps in 8 launches on noise data; context for the ramp-up and drain of each "
                          "launch at the headline size, not the headline workload"}
        big.close()
        del ub, Sb

    # end to end through the public API with host buffers
    e2e = None
    if not args.no_e2e:
        pin = torch.from_numpy(phi0).pin_memory()
        out_pin = torch.empty_like(pin).pin_memory()
        Ke = K
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        _check(solver.lib.mpfc_set_state(solver.h, pin.data_ptr(), None, None), "set_state")
        infos = (mpfc.mpfc_step_info * 1)()
        for _ in range(Ke):
            _check(solver.lib.mpfc_step(solver.h, scheme, 1, infos), "step")
        _check(solver.lib.mpfc_get_state(solver.h, out_pin.data_ptr(), None, None), "get_state")
        t1 = time.perf_counter()
        G = size * size
        e2e = {"value": world * Ke / (t1 - t0), "unit": UNIT, "h2d_bytes_per_step": 8 * G / Ke,
               "d2h_bytes_per_step": (8 * G + Ke * 24) / Ke,
               "how": "mpfc_set_state from pinned host phi^0, then K x mpfc_step(1) (each reads its step "
                      "record back), then mpfc_get_state to pinned host; host wall clock"}

    # the other forms on the same workload and protocol
    forms = {"fp64": {"steps_per_s": steps_per_s, "vcycles_per_step": float(np.mean(cycles)),
                      "error_vs_fp64_oracle": "lockstep parity <= 1e-10 per step (tests)"}}
    p32 = mpfc.default_params(m=size, n=size, h=w["h"], M=w["M"], epsilon=w["epsilon"], beta=w["beta"], dt=w["dt"],
                              tol=w["tol"], omega=w["omega"], guess=mpfc.MPFC_GUESS_EXTRAP,
                              precision=mpfc.MPFC_FP32_INNER, inner_cycles=INNER_CYCLES["fp32_inner"])
    s32 = mpfc.Solver(p32, stream=stream)
    s32.set_state(phi0)
    ms32, recs32 = timed_steps(s32, K, max(args.warmup, 0))
    ms32 = replicas.job_time_ms(ms32, device="cuda")
    # error of the mixed-precision steps against the FP64 path, 5 steps from phi^0
    a64 = mpfc.Solver(p, stream=stream)
    a32 = mpfc.Solver(p32, stream=stream)
    a64.set_state(phi0)
    a32.set_state(phi0)
    err32 = 0.0
    for _ in range(5):
        a64.step(scheme, 1)
        a32.step(scheme, 1)
        x64, x32 = a64.get_state()[0], a32.get_state()[0]
        err32 = max(err32, float(np.abs(x32 - x64).max() / np.abs(x64).max()))
    forms["fp32_inner"] = {"steps_per_s": world * K / (ms32 * 1e-3),
                           "outer_iterations_per_step": float(np.mean([r["cycles"] for r in recs32])),
                           "inner_cycles": INNER_CYCLES["fp32_inner"],
                           "fp32_vcycles_per_outer": 2,
                           "max_rel_error_vs_fp64_per_step": err32,
                           "speedup_vs_fp64": (world * K / (ms32 * 1e-3)) / steps_per_s}
    for obj in (s32, a64, a32):
        obj.close()
    # the FP32 sweep against the HBM roofline, at 2048^2 (the mixed-precision workload's size,
    # planes 7 x 16 MB), as mpfc_set_fp32_sweep selects it (by default a level's sweeps are part of
    # its one-launch ways): after an L2 flush, one pair of red-black sweeps in one launch each
    # over shared-memory tiles, there and back between the two copies of e, per sweep = half the
    # pair; median of 7.  Beside it the
    # two-launch sweep (one launch per colour, in place).  40 algorithmic bytes per cell (e
    # read and written, r and q read).
    if rank == 0:
        peaks = measured_peaks()
        big = mpfc.Solver(mpfc.default_params(m=2048, n=2048, h=w["h"], precision=mpfc.MPFC_FP32_INNER), stream=stream)

        def sweep_us(rows):
            big.set_fp32_sweep(rows, 2048 * 2048)
            big.fp32_time_smooth(0, 2)
            tsw = []
            for _ in range(7):
                flush.fill_(2.0)
                tsw.append(big.fp32_time_smooth(0, 2) / 2)
            return statistics.median(tsw) * 1e3

        us_tiled, us_two = sweep_us(16), sweep_us(0)
        big.close()
        gbs = 40.0 * 2048 * 2048 / (us_tiled * 1e-6) / 1e9
        gbs2 = 40.0 * 2048 * 2048 / (us_two * 1e-6) / 1e9
        forms["fp32_inner"]["sweep_roofline"] = {
            "kernel": "k_sweep32_tiles<16>, one red+black sweep at 2048^2 (half of a there-and-back pair after an "
                      "L2 flush; selected by mpfc_set_fp32_sweep, not launched by default)", "us": us_tiled,
            "bound": "hbm", "achieved_gbs": gbs, "peak_gbs": peaks["hbm_gbs"], "frac": gbs / peaks["hbm_gbs"],
            "peak_source": ("MEASURED_PEAKS.json hbm_gbs (of measured)" if peaks["source"] == "measured"
                            else "6.8 TB/s, an earlier GB300 measurement (of fallback)"),
            "two_launch": {"kernel": "k_smooth32 (one launch per colour, in place)", "us": us_two,
                           "achieved_gbs": gbs2, "frac": gbs2 / peaks["hbm_gbs"]}}

    # batched ensemble: 64 instances, sizes uniform from {128, 256, 512, 1024}^2, eps ~ U[0.02, 0.1],
    # beta ~ U[0.5, 1.5], mean density ~ U[0.05, 0.1], h = 0.5, s = 0.01, noise 0.05 U (seed 4)
    if not args.no_batch:
        from paper_1208_2643_gb300 import tuning
        ens = inputs.ensemble_instances(64, seed=4, rank=rank)
        bps = [mpfc.default_params(m=e["m"], n=e["n"], h=e["h"], dt=e["dt"], epsilon=e["epsilon"], beta=e["beta"],
                                   tol=w["tol"], omega=w["omega"]) for e in ens]
        b = mpfc.BatchSolver(bps, stream=stream)
        for i, e in enumerate(ens):
            b.set_state(i, e["phi0"])
        tiles = tuning.autotune(b, scheme, reps=3)
        b.step(scheme, 2)
        Kb = 100   # the workload list's length for the ensemble (config 4)
        eb0, eb1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        flush.fill_(3.0)
        eb0.record(stream)
        rcb, stb, cyb = b.step(scheme, Kb)
        eb1.record(stream)
        torch.cuda.synchronize()
        msb = eb0.elapsed_time(eb1)
        cells_b = sum(bp.m * bp.n for bp in bps)
        # the same instances one by one through the single-instance solver, same protocol
        seq_ms = 0.0
        for i, bp in enumerate(bps[:16]):   # a quarter of the instances, the same steps
            g1 = mpfc.Solver(bp, stream=stream)
            g1.set_state(ens[i]["phi0"])
            g1.step(scheme, 2)
            ea, eb = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            ea.record(stream)
            g1.step(scheme, Kb)
            eb.record(stream)
            torch.cuda.synchronize()
            seq_ms += ea.elapsed_time(eb)
            g1.close()
        seq_cells = sum(bp.m * bp.n for bp in bps[:16])
        forms["batched"] = {"workload": "64 instances, sizes U{128,256,512,1024}^2, eps U[0.02,0.1], "
                                        "beta U[0.5,1.5], mean U[0.05,0.1], h 0.5, s 0.01, fp64, tol 1e-10",
                            "instance_steps_per_s": world * 64 * Kb / (msb * 1e-3),
                            "cell_updates_per_s": world * cells_b * Kb / (msb * 1e-3),
                            "vcycles_per_instance_step": float(np.mean(cyb)) / Kb,
                            "sequential_cell_updates_per_s": seq_cells * Kb / (seq_ms * 1e-3),
                            "speedup_vs_sequential": (cells_b * Kb / (msb * 1e-3)) / (seq_cells * Kb / (seq_ms * 1e-3)),
                            "tiles": {str(k): v[:2] for k, v in tiles.items()},
                            "steps": Kb}
        b.close()
        # 64 instances of the headline workload at 1024^2 in one batch (8 GB of workspace)
        bp64 = [mpfc.default_params(m=size, n=size, h=w["h"], M=w["M"], epsilon=w["epsilon"], beta=w["beta"], dt=w["dt"],
                                    tol=w["tol"], omega=w["omega"]) for _ in range(64)]
        b64 = mpfc.BatchSolver(bp64, stream=stream)
        for i in range(64):
            b64.set_state(i, phi0)
        tuning.autotune(b64, scheme, reps=2)
        b64.step(scheme, 1)
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        flush.fill_(3.0)
        e0.record(stream)
        _, _, cy64 = b64.step(scheme, 2)
        e1.record(stream)
        torch.cuda.synchronize()
        ms64 = e0.elapsed_time(e1)
        # the batch's dominant kernel: one red-black sweep of every instance's finest level
        # (the tuned tiles)
        ms_kb = b64.time_smooth(scheme, 0, reps=10)
        kb_cells = 64 * size * size / (ms_kb * 1e-3)
        forms["batched_64x1024"] = {"workload": "64 x the headline workload (1024^2) in one batch, fp64, tol 1e-10",
                                    "instance_steps_per_s": world * 64 * 2 / (ms64 * 1e-3),
                                    "cell_updates_per_s": world * 64 * size * size * 2 / (ms64 * 1e-3),
                                    "vs_single_instance_cell_updates": (64 * size * size * 2 / (ms64 * 1e-3)) /
                                                                       (steps_per_s / world * size * size),
                                    "vcycles_per_instance_step": float(np.mean(cy64)) / 2, "steps": 2,
                                    "smooth_sweep": {"kernel": "kb_df_half<1>, one red+black sweep of the 64 finest "
                                                              "levels in float-float (two launches)",
                                                    "ms": ms_kb, "cell_updates_per_s": kb_cells,
                                                    "bound": "instruction issue and memory",
                                                    "frac_of_issue": DF_SMOOTH_INSTR_PER_CELL * kb_cells / 32.0 /
                                                    issue_peak(clk)}}
        b64.close()

    # learned initial guess (model trained by paper_1208_2643_gb300.guess on solver data at 256^2)
    if not args.no_learned:
        from paper_1208_2643_gb300 import guess as gmod
        blob = gmod.load()
        if blob is not None:
            pl = mpfc.default_params(m=size, n=size, h=w["h"], M=w["M"], epsilon=w["epsilon"], beta=w["beta"],
                                     dt=w["dt"], tol=w["tol"], omega=w["omega"], guess=mpfc.MPFC_GUESS_LEARNED)
            sl = mpfc.Solver(pl, stream=stream)
            gmod.attach(sl, blob)
            sl.set_state(phi0)
            Kl = 1000   # the workload list's inference length (config 5)
            msl, recl = timed_steps(sl, Kl, max(args.warmup, 0))
            msl = replicas.job_time_ms(msl, device="cuda")
            # the plain extrapolated guess over the same 1000 steps from the same state
            sx = mpfc.Solver(p, stream=stream)
            sx.set_state(phi0)
            msx, recx = timed_steps(sx, Kl, max(args.warmup, 0))
            msx = replicas.job_time_ms(msx, device="cuda")
            sx.close()

            def hist(recs_):
                cyc = [r["cycles"] for r in recs_]
                return {str(c): cyc.count(c) for c in sorted(set(cyc))}
            # the network's own cost: the five convolutions and the features, timed alone
            ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            ev0.record(stream)
            for _ in range(10):
                sl.lib.mpfc_op_learned_guess(sl.h)
            ev1.record(stream)
            torch.cuda.synchronize()
            forms["learned"] = {"workload": "the headline workload, 1000 steps after the warm-up, learned guess "
                                            "against the extrapolated one over the same steps",
                                "steps": Kl,
                                "steps_per_s": world * Kl / (msl * 1e-3),
                                "vcycles_per_step": float(np.mean([r["cycles"] for r in recl])),
                                "vcycle_histogram": hist(recl),
                                "res0_mean": float(np.mean([r["res0"] for r in recl])),
                                "extrapolated": {"steps_per_s": world * Kl / (msx * 1e-3),
                                                 "vcycles_per_step": float(np.mean([r["cycles"] for r in recx])),
                                                 "vcycle_histogram": hist(recx),
                                                 "res0_mean": float(np.mean([r["res0"] for r in recx]))},
                                "network_ms_per_step": ev0.elapsed_time(ev1) / 10,
                                "guess_gate": 2.6e4 * w["tol"],
                                "gated_steps_in_extrapolated_run": int(sum(r["res0"] >= 2.6e4 * w["tol"] for r in recx)),
                                "speedup_vs_fp64": msx / msl,
                                "conv32": conv32_timing(size),
                                "model": "5 x conv3x3 (3-32-32-32-32-1), GELU, bf16/fp32-acc; the 32-input-channel "
                                         "layers on tcgen05 (TMEM accumulators, TMA), the first on mma.sync; "
                                         "trained on solver trajectories at 256^2; run on the steps whose "
                                         "extrapolated guess has a scaled residual of at least guess_gate"}
            sl.close()

    # the PFC variant (Sec. 1, (1)) on the headline workload
    pq = mpfc.default_params(m=size, n=size, h=w["h"], M=w["M"], epsilon=w["epsilon"], beta=w["beta"], dt=w["dt"],
                             tol=w["tol"], omega=w["omega"], guess=mpfc.MPFC_GUESS_EXTRAP, model=mpfc.MPFC_MODEL_PFC)
    sq = mpfc.Solver(pq, stream=stream)
    sq.set_state(phi0)
    msq, recq = timed_steps(sq, K, max(args.warmup, 0))
    msq = replicas.job_time_ms(msq, device="cuda")
    forms["pfc"] = {"workload": "the headline workload with the PFC model (d_t phi = M Delta mu, Sec. 1)",
                    "steps_per_s": world * K / (msq * 1e-3),
                    "vcycles_per_step": float(np.mean([r["cycles"] for r in recq]))}
    sq.close()

    # mixed boundary conditions: the polycrystal run of Sec. 4.5 (periodic in x,
    # homogeneous Neumann in y), 2048^2, scheme 2, s = 1
    if not args.no_polycrystal:
        Np = 2048
        pp = mpfc.default_params(m=Np, n=Np, h=804.0 / 2048, M=1.0, epsilon=0.25, beta=0.9, dt=1.0, tol=w["tol"],
                                 omega=w["omega"], guess=mpfc.MPFC_GUESS_EXTRAP, bc=mpfc.MPFC_BC_NEUMANN_Y)
        sp = mpfc.Solver(pp, stream=stream)
        sp.set_state(inputs.polycrystal_seeds(Np, Np, 0.285, 3, 16, 0.3, replicas.instance_seed(2, rank)))
        Kp = 10
        msp, recp = timed_steps(sp, Kp, 3, sch=2)
        msp = replicas.job_time_ms(msp, device="cuda")
        cyc_p = float(np.mean([r["cycles"] for r in recp]))
        forms["neumann_polycrystal"] = {
            "workload": "2048^2, h = 804/2048, scheme 2, M = 1, eps = 0.25, beta = 0.9, s = 1, mean 0.285 with "
                        "three 16-cell seeds on y = 0, periodic x / homogeneous Neumann y, FP64, tol 1e-10",
            "steps_per_s": world * Kp / (msp * 1e-3), "vcycles_per_step": cyc_p,
            "cell_updates_per_s": world * Kp * Np * Np / (msp * 1e-3), "steps": Kp}
        sp.close()
        # the same run in the mixed-precision form (FP64 outer defect correction)
        pp.precision = mpfc.MPFC_FP32_INNER
        pp.inner_cycles = INNER_CYCLES["neumann_polycrystal"]
        sp = mpfc.Solver(pp, stream=stream)
        sp.set_state(inputs.polycrystal_seeds(Np, Np, 0.285, 3, 16, 0.3, replicas.instance_seed(2, rank)))
        msp32, recp32 = timed_steps(sp, Kp, 3, sch=2)
        msp32 = replicas.job_time_ms(msp32, device="cuda")
        forms["neumann_polycrystal"]["fp32_inner"] = {
            "steps_per_s": world * Kp / (msp32 * 1e-3),
            "outer_iterations_per_step": float(np.mean([r["cycles"] for r in recp32])),
            "inner_cycles": INNER_CYCLES["neumann_polycrystal"],
            "speedup_vs_fp64": msp / msp32}
        sp.close()

    # pinning: the strained-crystal run of Sec. 4.6 (scheme 2, weight 2 in strips around
    # the top and bottom of a crystal slab, target = the slab sheared by 4 % of 2 pi);
    # 512 x 384 instead of the paper's 512 x 400, whose odd factor 25 stops the
    # coarsening above the coarsest grid the direct solve takes
    if not args.no_polycrystal:
        mE, nE = 512, 384
        hE = 4.0 * np.pi / (16.0 * np.sqrt(3.0))
        pe = mpfc.default_params(m=mE, n=nE, h=hE, M=15.0 ** 2, epsilon=0.6, beta=0.2, dt=0.025 * hE * hE,
                                 tol=w["tol"], omega=w["omega"], guess=mpfc.MPFC_GUESS_EXTRAP, pinning=1)
        se = mpfc.Solver(pe, stream=stream)
        rows = np.arange(nE)[:, None] * np.ones((1, mE))
        lo, hi = int(0.2 * nE), int(0.8 * nE)
        inside = (rows >= lo) & (rows < hi)
        liquid = np.full((nE, mE), 0.57)
        slab = inputs.one_mode_crystal(mE, nE, hE, 0.395, 0.6)
        band = int(round(np.pi / hE))
        Wp = np.zeros((nE, mE))
        Wp[lo:lo + band] = 2.0
        Wp[hi - band:hi] = 2.0
        target = np.where(inside, inputs.one_mode_crystal(mE, nE, hE, 0.395, 0.6, shift=0.04 * 2 * np.pi), liquid)
        se.set_pinning(Wp, target)
        se.set_state(np.where(inside, slab, liquid))
        Ke = 20
        mse_, rece = timed_steps(se, Ke, 3, sch=2)
        mse_ = replicas.job_time_ms(mse_, device="cuda")
        forms["pinning_strained_crystal"] = {
            "workload": "512 x 384, h = 4 pi/(16 sqrt 3), scheme 2, M = 225, eps = 0.6, beta = 0.2, s = 0.025 h^2, "
                        "crystal slab (rows 20-80 %) in liquid 0.57, pinning weight 2 in pi-wide strips at the slab's "
                        "top and bottom, target sheared by 4 % of 2 pi; FP64, tol 1e-10",
            "steps_per_s": world * Ke / (mse_ * 1e-3),
            "vcycles_per_step": float(np.mean([r["cycles"] for r in rece])),
            "cell_updates_per_s": world * Ke * mE * nE / (mse_ * 1e-3), "steps": Ke}
        se.close()
        # the same run in the mixed-precision form
        pe.precision = mpfc.MPFC_FP32_INNER
        pe.inner_cycles = INNER_CYCLES["pinning_strained_crystal"]
        se = mpfc.Solver(pe, stream=stream)
        se.set_pinning(Wp, target)
        se.set_state(np.where(inside, slab, liquid))
        mse32, rece32 = timed_steps(se, Ke, 3, sch=2)
        mse32 = replicas.job_time_ms(mse32, device="cuda")
        forms["pinning_strained_crystal"]["fp32_inner"] = {
            "steps_per_s": world * Ke / (mse32 * 1e-3),
            "outer_iterations_per_step": float(np.mean([r["cycles"] for r in rece32])),
            "inner_cycles": INNER_CYCLES["pinning_strained_crystal"],
            "speedup_vs_fp64": mse_ / mse32}
        se.close()

    # the workload list's second-order run (config 2): 512^2, h = pi/4, eps = 0.25,
    # beta = 0.9, mean -0.285, s = 0.05, three crystallites of radius 20h with 1e-3 noise,
    # 500 steps, FP64
    if not args.no_configs:
        m2 = 512
        p2 = mpfc.default_params(m=m2, n=m2, h=np.pi / 4, epsilon=0.25, beta=0.9, dt=0.05, tol=w["tol"],
                                 omega=w["omega"], guess=mpfc.MPFC_GUESS_EXTRAP)
        s2 = mpfc.Solver(p2, stream=stream)
        s2.set_state(inputs.crystallite_field(m2, m2, np.pi / 4, -0.285, 0.25, count=3, radius_cells=20, noise=1e-3,
                                              seed=replicas.instance_seed(2, rank)))
        ms2, rec2 = timed_steps(s2, 500, 3, sch=2)
        ms2 = replicas.job_time_ms(ms2, device="cuda")
        forms["second_order_crystallites_512"] = {
            "workload": "512^2, h = pi/4, scheme 2, eps = 0.25, beta = 0.9, mean -0.285, s = 0.05, three crystallites "
                        "of radius 20h + 1e-3 noise, 500 timed steps after 3 warm-up steps, FP64, tol 1e-10",
            "steps": 500, "steps_per_s": world * 500 / (ms2 * 1e-3),
            "cell_updates_per_s": world * 500 * m2 * m2 / (ms2 * 1e-3),
            "vcycles_per_step": float(np.mean([r["cycles"] for r in rec2]))}
        s2.close()
        # the workload list's mixed-precision run (config 3): 2048^2, scheme 1, s = 0.02,
        # 200 steps; then, step by step from the FP64 path's states, the largest relative
        # max-norm difference of the mixed form's step from the FP64 step
        m3 = 2048
        p3 = mpfc.default_params(m=m3, n=m3, h=0.5, dt=0.02, tol=w["tol"], omega=w["omega"],
                                 guess=mpfc.MPFC_GUESS_EXTRAP, precision=mpfc.MPFC_FP32_INNER,
                                 inner_cycles=INNER_CYCLES["mixed_precision_2048"])
        phi3 = inputs.noise_field(m3, m3, 0.07, 0.05, replicas.instance_seed(3, rank))
        s3 = mpfc.Solver(p3, stream=stream)
        s3.set_state(phi3)
        ms3, rec3 = timed_steps(s3, 200, 3, sch=1)
        ms3 = replicas.job_time_ms(ms3, device="cuda")
        p3.precision = mpfc.MPFC_FP64
        r3 = mpfc.Solver(p3, stream=stream)
        r3.set_state(phi3)
        s3.set_state(phi3)
        ms3_64 = 0.0
        err3 = 0.0
        for _ in range(200):
            st3 = r3.get_state(device=True)
            s3.set_state(*st3)
            s3.step(1, 1)
            ea, eb = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            flush.fill_(4.0)
            ea.record(stream)
            r3.step_async(1, 1)
            eb.record(stream)
            torch.cuda.synchronize()
            ms3_64 += ea.elapsed_time(eb)
            a3, b3 = s3.get_state(device=True)[0], r3.get_state(device=True)[0]
            err3 = max(err3, float((a3 - b3).abs().max() / b3.abs().max()))
        rc3, _, _ = r3.records(1024)
        if rc3 != mpfc.MPFC_OK:
            raise mpfc.MPFCError(rc3, "config-3 FP64 steps")
        ms3_64 = replicas.job_time_ms(ms3_64, device="cuda")
        forms["mixed_precision_2048"] = {
            "workload": "2048^2, h = 0.5, scheme 1, eps = 0.025, beta = 0.9, s = 0.02, noise 0.07 + 0.05 U, 200 steps, "
                        "FP32 inner V-cycles in FP64 outer defect correction, tol 1e-10 (200 timed steps after 3 warm-up steps)",
            "steps": 200, "steps_per_s": world * 200 / (ms3 * 1e-3),
            "cell_updates_per_s": world * 200 * m3 * m3 / (ms3 * 1e-3),
            "outer_iterations_per_step": float(np.mean([r["cycles"] for r in rec3])),
            "inner_cycles": INNER_CYCLES["mixed_precision_2048"],
            "fp64_steps_per_s": world * 200 / (ms3_64 * 1e-3),
            "speedup_vs_fp64": ms3_64 / ms3,
            "max_rel_error_vs_fp64_per_step": err3,
            "error_note": "each of the 200 steps taken by both forms from the FP64 path's state; the FP64 path is the "
                          "oracle's in lockstep (tests), and the mixed form is within 1e-8 of the oracle on a "
                          "3-step prefix (tests)"}
        s3.close()
        r3.close()

    cpu = None
    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        # all host cores (the oracle's OpenMP build, bitwise the serial one), then one core
        rate, done, dt, cyc, nthr = cpu_oracle_rate(size, scheme, 12, budget_s=15.0, threaded=True)
        rate1, done1, dt1, cyc1, _ = cpu_oracle_rate(size, scheme, 3, budget_s=12.0)
        cpu = {"value": rate, "unit": UNIT, "cores": nthr, "kind": "oracle",
               "sample": f"{done} time steps of the same {size}^2 workload from phi^0 "
                         f"({cyc / done:.2f} V-cycles/step), the C oracle's OpenMP build on {nthr} threads "
                         f"(nproc {os.cpu_count()})",
               "serial": {"value": rate1, "unit": UNIT, "cores": 1,
                          "sample": f"{done1} time steps from phi^0 ({cyc1 / done1:.2f} V-cycles/step), serial C"}}

    if rank == 0:
        line = {"metric": METRIC, "value": steps_per_s, "unit": UNIT, "n_gpus": world, "steps": K,
                "warmup": args.warmup, "ms_per_step": ms / K, "higher_is_better": True, "scaling": "weak",
                "vs_baseline": None, "dtype": "f64", "data": "synthetic", "config": w,
                "cell_updates_per_s": steps_per_s * size * size,
                "vcycles_per_step": float(np.mean(cycles)) if cycles else None,
                "sweep_cell_updates_per_s": steps_per_s * size * size * (p.nu1 + p.nu2) *
                (float(np.mean(cycles)) if cycles else 0.0),
                "roofline": {"bound": "instruction issue",
                             "kernel": "kb_df_half<1> on one instance: one red+black sweep of the finest level in "
                                       "float-float (the cell function of k_df_smooth, which leads the step), back to "
                                       "back, planes in L2",
                             "achieved": df_winstr / 1e9, "peak": issue_peak(clk) / 1e9, "unit": "G warp instructions/s",
                             "frac": df_winstr / issue_peak(clk),
                             "peak_source": "one instruction a cycle and sub-partition at the median SM clock of the "
                                            "timed region",
                             "sweep_ms": df_sweep_ms, "instructions_per_cell": DF_SMOOTH_INSTR_PER_CELL, "traffic": None},
                "roofline_fp64_cycle": {"bound": "alu",
                                        "kernel": "k_smooth<1>, one red+black sweep of the finest level in FP64 (not "
                                                  "launched by the timed steps: the FP64 V-cycle runs outside the "
                                                  "correction form's range)",
                                        "achieved": achieved, "peak": fp64_peak, "unit": "TFLOP/s (FP64, FMA = 2)",
                                        "frac": achieved / fp64_peak,
                                        "peak_source": "measured live: FP64 FMA-chain probe on this GPU",
                                        "hbm_gbs_algorithmic": achieved_gbs,
                                        "sweep_ms": sweep_ms,
                                        "traffic": traffic_for("k_smooth", size),
                                        "steady_state": steady},
                "forms": forms,
                "e2e": e2e, "gpu_launches": launches, "clocks": clk, "cpu_baseline": cpu}
        print(json.dumps(line), flush=True)
    if world > 1:
        dist.destroy_process_group()


def main():
    args = parse_args()
    if args.impl == "reference":
        run_reference(args)
    else:
        run_ours(args)


if __name__ == "__main__":
    main()
