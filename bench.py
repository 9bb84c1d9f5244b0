"""Benchmark: amplitudes/s of random grid circuits by complex graphical-model
variable elimination on one GB300 (and N replicas under torchrun).

Default workload: 5x9 grid, depth 40, seed 0, a batch of 1000 uniformly random
output bitstrings, computed in passes of 4 (the plan that fits one GPU: a
55 GB workspace).  One step = one full pass of the path (leaf factors for the
pass's bitstrings, every elimination step -- GEMM-shaped steps on the tensor
cores as split-FP16 products, the rest on the FP32 cores --, FP64
accumulation).  The same passes are also timed with split-BF16 GEMM steps and
with every GEMM step on the FP32 cores (plain complex64); each precision's
error against the FP64 oracle's stored amplitudes is stated.  Prints ONE JSON
line (rank 0).

  python bench.py [--gpus N] [--steps K] [--warmup W] [--workload NAME]
  python bench.py --impl reference   # the FP64 CPU oracle on a bounded sample
"""
from __future__ import annotations

import argparse
import hashlib
import json
import os
import statistics
import subprocess
import sys
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

import qgm_inputs as qi  # noqa: E402

METRIC = "amplitudes/sec on 1 GB300 at stated rel. error vs FP64; % of tensor/HBM roofline"
UNIT = "amplitudes/s"
L2_BYTES = 129 * 2 ** 20
# bitstrings per pass where the whole batch does not fit one plan
PASS_BATCH = {"grid5x9_d40_b1000": 4}
# FP64 oracle amplitudes stored for the workloads (tests/golden/, written by
# tests/golden/make_golden.py from the oracle only)
GOLDEN = {"grid5x9_d40_b1000": "amps_grid5x9_d40.json", "grid6x6_d25_b1000": "amps_grid6x6_d25.json"}
PRECISIONS = [("split_fp16", "fp16"), ("split_bf16", "bf16"), ("c64", "fp32")]

# DRAM traffic per launch of the dominant kernel from one ncu capture, keyed
# by workload and the sha1 of exec.cu it was taken on (null once it changed)
NCU_TRAFFIC = {}


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=10)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--workload", default="grid5x9_d40_b1000", choices=sorted(qi.WORKLOADS))
    ap.add_argument("--grad", action="store_true",
                    help="parametrised workload: time amplitudes plus the gradient of sum log|a|^2")
    ap.add_argument("--precision", default="fp16", choices=["fp16", "bf16", "fp32"],
                    help="GEMM steps of the headline value: split FP16, split BF16 or FP32 cores")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-precisions", action="store_true", help="time the headline precision only")
    ap.add_argument("--executor", type=int, default=0, help="0 auto, 1 stepwise, 2 resident, 3 compiled resident")
    ap.add_argument("--no-autotune", action="store_true", help="fixed launch rules instead of the autotuner")
    ap.add_argument("--tc-convert", action="store_true",
                    help="folded tensor-core steps convert their batched operand in the product kernel")
    ap.add_argument("--custom", default=None, metavar="RxC,DEPTH,BATCH",
                    help="a smaller seed-0 grid circuit instead of a workload (profiling captures), e.g. 4x8,40,4")
    a = ap.parse_args()
    if a.custom:
        g, d, b = a.custom.split(",")
        r, c = g.split("x")
        name = f"grid{r}x{c}_d{d}_b{b}"
        qi.WORKLOADS[name] = (int(r), int(c), int(d), int(b), False)
        PASS_BATCH[name] = int(b)
        a.workload = name
    return a


def dist_env():
    return (int(os.environ.get("RANK", "0")), int(os.environ.get("WORLD_SIZE", "1")),
            int(os.environ.get("LOCAL_RANK", "0")))


def peaks():
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as f:
            d = json.load(f)
        return {"hbm_gbs": float(d["hbm_gbs"]), "bf16_tflops": float(d["bf16_tflops"]),
                "bf16_tflops_sustained": float(d["bf16_tflops_sustained"]), "source": "measured"}
    except Exception:
        return {"hbm_gbs": 6800.0, "bf16_tflops": 1900.0, "bf16_tflops_sustained": 1700.0, "source": "fallback"}


def exec_hash():
    h = hashlib.sha1()
    with open(os.path.join(ROOT, "paper_1712_05384_gb300", "csrc", "exec.cu"), "rb") as f:
        h.update(f.read())
    return h.hexdigest()[:12]


class Clocks:
    """nvidia-smi sampling of SM clocks and throttle reasons during the timed region."""
    Q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
         "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
         "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index):
        self.idx = gpu_index
        self.proc = None
        self.out = ""

    def __enter__(self):
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", f"--id={self.idx}", f"--query-gpu={self.Q}",
                 "--format=csv,noheader,nounits", "-lms", "100"],
                stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
        except Exception:
            self.proc = None
        return self

    def __exit__(self, *a):
        if self.proc is not None:
            self.proc.terminate()
            try:
                self.out, _ = self.proc.communicate(timeout=5)
            except Exception:
                self.proc.kill()
                self.out = ""

    def summary(self):
        sm, mx, reasons = [], None, set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for line in self.out.strip().splitlines():
            f = [x.strip() for x in line.split(",")]
            if len(f) < 9:
                continue
            try:
                sm.append(float(f[1]))
                mx = float(f[2])
            except ValueError:
                continue
            for n, v in zip(names, f[5:9]):
                if v.lower().startswith("active"):
                    reasons.add(n)
        if not sm:
            return None
        return {"sm_mhz": statistics.median(sm), "sm_max_mhz": mx, "reasons": sorted(reasons), "samples": len(sm)}


def golden(workload):
    name = GOLDEN.get(workload)
    path = os.path.join(ROOT, "tests", "golden", name) if name else None
    if not path or not os.path.exists(path):
        return None
    with open(path) as f:
        d = json.load(f)
    xs = np.array([int(e["x"]) for e in d["amplitudes"]], dtype=np.uint64)
    ref = np.array([complex(e["re"], e["im"]) for e in d["amplitudes"]])
    return (xs, ref) if len(xs) else None


def reference_amplitudes(workload, c, bits):
    """(bitstrings, FP64 oracle amplitudes) to state the error against: the
    stored oracle values, else the state vector on a sample (n <= 25)."""
    g = golden(workload)
    if g is not None:
        return g
    if c.n <= 25:
        from oracle import statevector as sv
        xs = bits[:64]
        return xs, sv.amplitudes(c, xs)
    return None


def error_measures(a, ref, n):
    d = np.abs(a - ref)
    rms = 2.0 ** (-n / 2)
    big = np.abs(ref) >= rms
    wide = np.abs(ref) >= 1e-3 * rms
    return {"max_rel_err": float(np.max(d[big] / np.abs(ref[big]))) if big.any() else None,
            "max_rel_err_cut": "|a_ref| >= 2^-n/2",
            "max_rel_err_1e3": float(np.max(d[wide] / np.abs(ref[wide]))) if wide.any() else None,
            "excluded_1e3": int((~wide).sum()),
            "max_abs_err_rms": float(np.max(d) * 2.0 ** (n / 2)), "count": int(len(ref)), "against": "FP64 oracle"}


def cpu_oracle_sample(workload, c, bits):
    """The FP64 oracle (oracle/ve.c, plain C, OpenMP over each bucket's
    entries on every host core) on a bounded sample: (amplitudes/s, sample
    description, cores).  5x9 depth 40: one of the 2^7 conditioned parts of
    one bitstring (the oracle slices it to fit host memory), scaled to a
    whole amplitude; smaller circuits: whole amplitudes for about 10 s on a
    pool of threads over bitstrings."""
    from oracle import order as O
    from oracle import ugm, vec
    cores = os.cpu_count() or 1
    m = ugm.build(c)
    adj = O.graph(m)
    order, w = O.min_fill(adj)
    pr = vec.Prepared(m)
    if w > 31:
        sl = O.slice_greedy(adj, order, max_clique=30)
        part = [v for v in sl]
        fixed_first = part[:]  # time slice 0 of the first bitstring
        t0 = time.perf_counter()
        _one_slice(m, pr, order, fixed_first, int(bits[0]))
        dt = time.perf_counter() - t0
        n_parts = 2 ** len(sl)
        return 1.0 / (dt * n_parts), (f"one of the {n_parts} conditioned parts (slices) of bitstring 0 in "
                                      f"{dt:.1f} s, scaled to a whole amplitude; oracle/ve.c FP64 bucket "
                                      f"elimination, min-fill order, {cores} threads"), cores
    t0 = time.perf_counter()
    done = 0
    while done < len(bits) and time.perf_counter() - t0 < 10.0:
        chunk = bits[done:done + 4 * cores]
        vec.amplitudes_parallel(c, chunk, order=order, model=m, prepared=pr, workers=cores)
        done += len(chunk)
    dt = time.perf_counter() - t0
    return done / dt, (f"{done} bitstrings in {dt:.1f} s; oracle/ve.c FP64 bucket elimination, min-fill "
                       f"order, a pool of {cores} host threads over bitstrings"), cores


def _one_slice(m, pr, order, slice_vars, x):
    from oracle import vec
    fixed = np.full(m.n_vars, -1, dtype=np.int32)
    for v in m.inputs:
        fixed[v] = 0
    for j, v in enumerate(m.outputs):
        fixed[v] = (x >> j) & 1
    for v in slice_vars:
        fixed[v] = 0
    elim = np.array([v for v in order if v not in set(slice_vars)], dtype=np.int32)
    out = np.zeros(2)
    vec.lib().ve_amplitude(m.n_vars, len(m.factors), pr.rank.ctypes.data, pr.off.ctypes.data, pr.vars.ctypes.data,
                           pr.toff.ctypes.data, pr.tables.ctypes.data, fixed.ctypes.data, elim.ctypes.data,
                           len(elim), 0, out.ctypes.data)


def run_reference(args, rank, world):
    if rank != 0:
        return
    rows, cols, depth, B, param = qi.WORKLOADS[args.workload]
    c = qi.grid_circuit(rows, cols, depth, 0, param=param)
    bits = qi.bitstrings(c.n, B, 0)
    cores = os.cpu_count() or 1
    ts, dts = [], []
    sample = ""
    warm = max(args.warmup, 3)
    for s in range(warm + args.steps):
        t0 = time.perf_counter()
        rate, sample, cores = cpu_oracle_sample(args.workload, c, bits[s % len(bits):])
        if s >= warm:
            ts.append(rate)
            dts.append(time.perf_counter() - t0)
    v = float(np.mean(ts))
    print(json.dumps({
        "impl": "reference", "metric": METRIC, "value": v, "unit": UNIT, "n_gpus": world,
        "steps": args.steps, "warmup": warm, "ms_per_step": 1e3 * float(np.mean(dts)),
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "config": {"workload": args.workload, "grid": f"{rows}x{cols}", "depth": depth, "batch": B, "seed": 0,
                   "parallelism": "replicas1"},
        "cpu_baseline": {"value": v, "unit": UNIT, "cores": cores, "kind": "oracle",
                         "sample": "each step: " + sample},
        "e2e": {"value": v, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }), flush=True)


def run_secondary(args):
    """Secondary lines on one GPU: all 2^n amplitudes of a small circuit
    (open outputs, qgm_eliminate), or amplitudes plus the gradient of
    L = sum log|a|^2 (qgm_amplitudes, then qgm_amplitude_grad, as the
    torch.autograd wrapper runs them).  Parity of both is in the GPU tests."""
    import torch
    import paper_1712_05384_gb300 as q
    from paper_1712_05384_gb300 import build
    build.build()
    q.lib()
    rows, cols, depth, B, param = qi.WORKLOADS[args.workload]
    model = q.Model(q.Circuit.grid(rows, cols, depth, 0, param))
    n = rows * cols
    stream = torch.cuda.current_stream()
    flush = torch.empty(2 * L2_BYTES // 4, dtype=torch.float32, device="cuda")
    if B == 0:
        plan = q.Plan(model, output_mode=q.OUT_OPEN).bind()
        d_out = torch.empty(2 << n, dtype=torch.float64, device="cuda")
        step = lambda: plan.eliminate(d_out, stream=stream)
        amps, what = 1 << n, "all 2^n amplitudes (open outputs)"
        h_out = torch.empty(2 << n, dtype=torch.float64).pin_memory()
        e2e_step = lambda: (step(), h_out.copy_(d_out, non_blocking=True))
        hb, db = 0, 16 << n
    else:
        bits = qi.bitstrings(n, B, 0)
        plan = q.Plan(model, batch=B, gradients=bool(args.grad)).bind()
        d_bits = torch.from_numpy(bits.astype(np.int64)).cuda()
        d_out = torch.empty(2 * B, dtype=torch.float64, device="cuda")
        d_g = torch.empty(2 * B, dtype=torch.float64, device="cuda")
        n_par = 2 * len(q.Circuit.grid(rows, cols, depth, 0, param).param_gates()) if param else 0
        d_grad = torch.empty(max(n_par, 1), dtype=torch.float64, device="cuda")

        def step():
            plan.amplitudes(d_bits, d_out, stream=stream)
            if args.grad:
                a = torch.view_as_complex(d_out.view(B, 2))
                d_g.copy_(torch.view_as_real(a / (a.abs() ** 2)).reshape(-1))  # g = dL/d(conj a)
                plan.amplitude_grad(d_bits, d_g, d_grad, stream=stream)
        amps, what = B, ("amplitudes and the gradient of sum log|a|^2 (%d angles)" % n_par if args.grad
                         else "amplitudes")
        h_bits = torch.from_numpy(bits.astype(np.int64)).pin_memory()
        h_grad = torch.empty_like(d_grad, device="cpu").pin_memory()

        def e2e_step():
            d_bits.copy_(h_bits, non_blocking=True)
            step()
            (h_grad.copy_(d_grad, non_blocking=True) if args.grad else h_out_b.copy_(d_out, non_blocking=True))
        h_out_b = torch.empty(2 * B, dtype=torch.float64).pin_memory()
        hb, db = 8 * B, (8 * n_par if args.grad else 16 * B)
    for _ in range(max(args.warmup, 3)):
        step()
    torch.cuda.synchronize()
    evs = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(args.steps)]
    with Clocks(0) as clk:
        for i in range(args.steps):
            flush.fill_(float(i))
            evs[i][0].record(stream)
            step()
            evs[i][1].record(stream)
        torch.cuda.synchronize()
    if plan.status(stream) != 0:
        raise RuntimeError("device status not OK in the timed region")
    t_ms = sum(a.elapsed_time(b) for a, b in evs)
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    for _ in range(args.steps):
        e2e_step()
    torch.cuda.synchronize()
    e2e_s = time.perf_counter() - t0
    print(json.dumps({
        "metric": METRIC, "value": amps * args.steps / (t_ms / 1e3), "unit": UNIT, "n_gpus": 1,
        "steps": args.steps, "warmup": max(args.warmup, 3), "ms_per_step": t_ms / args.steps,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "c64", "data": "synthetic",
        "config": {"workload": args.workload, "grid": f"{rows}x{cols}", "depth": depth, "batch": B, "seed": 0,
                   "what": what, "executor": {1: "stepwise", 2: "resident", 3: "compiled resident"}.get(
                       plan.executor()[0]),
                   "l2": "flushed between timed steps (264 MB write, untimed)"},
        "e2e": {"value": amps * args.steps / e2e_s, "unit": UNIT, "h2d_bytes_per_step": hb, "d2h_bytes_per_step": db},
        "clocks": clk.summary() if hasattr(clk, "summary") else None,
    }), flush=True)


def main():
    args = parse()
    rank, world, local = dist_env()
    if args.impl == "reference":
        run_reference(args, rank, world)
        return
    if qi.WORKLOADS[args.workload][3] == 0 or args.grad:
        if rank == 0:
            run_secondary(args)
        return
    import torch
    import torch.distributed as dist
    import paper_1712_05384_gb300 as q
    from paper_1712_05384_gb300 import build, shard

    if world > 1:
        dist.init_process_group("nccl")
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    if rank == 0 or world == 1:
        build.build()
    if world > 1:
        dist.barrier()
    q.lib()

    rows, cols, depth, B, param = qi.WORKLOADS[args.workload]
    P = PASS_BATCH.get(args.workload, B)
    c_py = qi.grid_circuit(rows, cols, depth, 0, param=param)
    n = c_py.n
    # weak scaling: each rank takes its own block of B bitstrings (no
    # data-path collective)
    bits = shard.shard(qi.bitstrings(n, B * world, 0), rank, world)
    model = q.Model(q.Circuit.grid(rows, cols, depth, 0, param))
    stream = torch.cuda.current_stream(dev)
    d_all = torch.from_numpy(bits.astype(np.int64)).to(dev)
    d_pass = torch.empty(P, dtype=torch.int64, device=dev)
    d_out = torch.empty(2 * P, dtype=torch.float64, device=dev)
    flush = torch.empty(2 * L2_BYTES // 4, dtype=torch.float32, device=dev)
    n_pass = (len(bits) + P - 1) // P
    ref = reference_amplitudes(args.workload, c_py, bits) if rank == 0 else None
    pk = peaks()

    def make_plan(precision):
        # the autotuner picks per-step launch parameters at bind (untimed)
        return q.Plan(model, batch=P, executor=args.executor, precision=precision, autotune=not args.no_autotune,
                      tc_convert=args.tc_convert,
                      order_kind=q.ORDER_MINFILL if P < B else q.ORDER_AUTO).bind()

    def run_pass(plan, i):
        k = i % n_pass
        m = min(P, len(bits) - k * P)
        d_pass[:m].copy_(d_all[k * P:k * P + m])
        plan.amplitudes(d_pass, d_out, B=m, stream=stream)

    def amplitudes_of(plan, xs):
        out = []
        for k in range(0, len(xs), P):
            out.append(plan.amplitudes_host(np.asarray(xs[k:k + P], dtype=np.uint64)))
        return np.concatenate(out)

    def timed(plan, steps, warmup, clocks=None):
        for i in range(max(warmup, 3)):
            run_pass(plan, i)
        torch.cuda.synchronize()
        if plan.status(stream) != 0:
            raise RuntimeError("device status not OK after warm-up")
        evs = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(steps)]
        if world > 1:
            dist.barrier()
        torch.cuda.synchronize()
        ctx = Clocks(local) if clocks else None
        if ctx:
            ctx.__enter__()
        # an NVTX range around the timed passes of the headline plan, so that a
        # profiler can select exactly these launches (ncu --nvtx --nvtx-include timed/)
        torch.cuda.nvtx.range_push("timed" if clocks else "timed_other")
        for i in range(steps):
            flush.fill_(float(i))
            evs[i][0].record(stream)
            run_pass(plan, i)
            evs[i][1].record(stream)
        torch.cuda.synchronize()
        torch.cuda.nvtx.range_pop()
        if ctx:
            ctx.__exit__()
        if plan.status(stream) != 0:
            raise RuntimeError("device status not OK in the timed region")
        t_ms = sum(a.elapsed_time(b) for a, b in evs)
        if world > 1:
            dist.barrier()
            t = torch.tensor([t_ms], device=dev, dtype=torch.float64)
            dist.all_reduce(t, op=dist.ReduceOp.MAX)
            t_ms = float(t.item())
        return t_ms, ctx

    # ---- headline precision
    plan = make_plan(args.precision)
    info = plan.info
    t_ms, clk = timed(plan, args.steps, args.warmup, clocks=True)
    amps_per_step = min(P, len(bits))
    value = world * amps_per_step * args.steps / (t_ms / 1e3)
    err = error_measures(amplitudes_of(plan, ref[0]), ref[1], n) if ref is not None else None

    # ---- end to end through the public host API: host bitstrings in, host
    # amplitudes out, copies inside the timed region
    hb = torch.from_numpy(bits[:P].view(np.int64).copy()).pin_memory()
    hout = torch.empty(2 * P, dtype=torch.float64).pin_memory()
    for _ in range(3):
        q._lib.check(q.lib().qgm_amplitudes_host(plan._h, hb.data_ptr(), P, hout.data_ptr(), stream.cuda_stream))
    if world > 1:
        dist.barrier()
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    for i in range(args.steps):
        k = i % n_pass
        m = min(P, len(bits) - k * P)
        hb[:m].copy_(torch.from_numpy(bits[k * P:k * P + m].view(np.int64)))
        q._lib.check(q.lib().qgm_amplitudes_host(plan._h, hb.data_ptr(), m, hout.data_ptr(), stream.cuda_stream))
    e2e_s = time.perf_counter() - t0
    if world > 1:
        t = torch.tensor([e2e_s], device=dev, dtype=torch.float64)
        dist.all_reduce(t, op=dist.ReduceOp.MAX)
        e2e_s = float(t.item())
    e2e = world * amps_per_step * args.steps / e2e_s

    # ---- roofline per step class, from per-launch CUDA events of one pass
    step_bytes, step_flops = plan.step_costs()
    ex_kind, ex_chunk, ex_smem = plan.executor()
    kinds = plan.step_kernels()
    gemms = plan.gemm_shapes()
    reps = 3
    roof_steps = {}
    fp32_peak = q._lib.measure_fp32_peak(stream.cuda_stream) if hasattr(q._lib, "measure_fp32_peak") else None
    if ex_kind == q.EXEC_STEPWISE:
        ms = np.zeros(info.n_steps + 2)
        ms_split = np.zeros(len(gemms))
        ms_prod = np.zeros(len(gemms))
        for _ in range(reps):
            # per-launch event timing; unavailable under a kernel profiler,
            # where the pass's own launches are what is measured
            try:
                flush.fill_(1.0)
                ms += plan.profile(d_pass, d_out, B=P, stream=stream)
                flush.fill_(1.0)
                a, b = plan.profile_gemm(d_pass, d_out, B=P, stream=stream)
            except q.QgmError as e:
                print(f"per-step profile unavailable: {e}", file=sys.stderr)
                ms[:] = 1e-9
                a, b = np.full(len(gemms), 1e-9), np.full(len(gemms), 1e-9)
            ms_split += a
            ms_prod += b
        ms /= reps
        ms_split /= reps
        ms_prod /= reps
        tc = [g for g in gemms if g["tc"]]
        tc_idx = [i for i, g in enumerate(gemms) if g["tc"]]
        g_flops = float(sum(step_flops[g["step"]] for g in tc))
        # a tensor-core step's time: its operand split pass (none for the
        # streamed operand of a step that converts it in the product kernel)
        # plus the product kernel
        g_ms_prod = float(ms_prod[tc_idx].sum()) if tc_idx else 0.0
        g_ms = g_ms_prod + (float(ms_split[tc_idx].sum()) if tc_idx else 0.0)
        ps = [s for s in range(info.n_steps) if kinds[s] != 3]
        ps_bytes = float(step_bytes[ps].sum())
        ps_ms = float(ms[[1 + s for s in ps]].sum())
        pass_ms = float(ms.sum())
        if tc and g_ms > 0:
            ach = g_flops / (g_ms / 1e3) / 1e12
            roof = {"bound": "tensor", "achieved": ach, "peak": pk["bf16_tflops"], "unit": "TFLOP/s",
                    "frac": ach / pk["bf16_tflops"], "traffic": NCU_TRAFFIC.get((args.workload, exec_hash())),
                    "kernel": f"k_gemm_tc with its operand split k_split (GEMM-shaped steps, "
                              f"split {'FP16' if args.precision == 'fp16' else 'BF16'} on tcgen05; algorithmic flops "
                              f"8*M*N*K per complex product, split terms not counted)",
                    "frac_sustained": ach / pk["bf16_tflops_sustained"], "peak_source": pk["source"] + " (bf16 burst)",
                    "algorithmic_flops_per_pass": g_flops, "kernel_ms_per_pass": g_ms,
                    "product_kernel_ms_per_pass": g_ms_prod,
                    "tensor_pipe_flops_per_algorithmic_flop": 3.0 if args.precision == "fp16" else 6.0,
                    "frac_ceiling": 1.0 / (3.0 if args.precision == "fp16" else 6.0)}
        else:
            ach = ps_bytes / (ps_ms / 1e3) / 1e9
            roof = {"bound": "hbm", "achieved": ach, "peak": pk["hbm_gbs"], "unit": "GB/s",
                    "frac": ach / pk["hbm_gbs"], "traffic": None, "kernel": "product-sum steps",
                    "algorithmic_bytes_per_pass": ps_bytes, "kernel_ms_per_pass": ps_ms,
                    "peak_source": pk["source"]}
        roof_steps = {
            "pass_ms_kernel_by_kernel": pass_ms,
            "gemm_tensor_core": {"steps": len(tc), "algorithmic_tflop": g_flops / 1e12, "ms": g_ms,
                                 "tflops": g_flops / (g_ms / 1e3) / 1e12 if g_ms else None,
                                 "frac_bf16_burst": (g_flops / (g_ms / 1e3) / 1e12) / pk["bf16_tflops"] if g_ms else None,
                                 "frac_bf16_sustained": (g_flops / (g_ms / 1e3) / 1e12) / pk["bf16_tflops_sustained"]
                                 if g_ms else None},
            "gemm_operand_split": {"ms": float(ms_split[tc_idx].sum()) if tc_idx else 0.0},
            "gemm_fp32_cores": {"steps": len(gemms) - len(tc),
                                "ms": float(ms_prod[[i for i, g in enumerate(gemms) if not g["tc"]]].sum())
                                if len(gemms) > len(tc) else 0.0},
            "product_sum": {"steps": len(ps), "algorithmic_gb": ps_bytes / 1e9, "ms": ps_ms,
                            "gbs": ps_bytes / (ps_ms / 1e3) / 1e9 if ps_ms else None,
                            "frac_hbm": ps_bytes / (ps_ms / 1e3) / 1e9 / pk["hbm_gbs"] if ps_ms else None},
            "per_gemm": [dict(g, split_ms=float(ms_split[i]), product_ms=float(ms_prod[i]),
                              tflops=float(step_flops[g["step"]] / ((ms_split[i] + ms_prod[i]) / 1e3) / 1e12)
                              if ms_split[i] + ms_prod[i] > 0 else None)
                         for i, g in enumerate(gemms)],
            "tuning": [t for t in plan.tuning()],
        }
        # the library's own count of its launches per call (grouped small
        # steps, split passes), times the timed calls
        launches = args.steps * int(plan.amplitudes_report(d_pass, d_out, B=P, stream=stream)["launches"])
    else:
        ms = np.zeros(info.n_steps + 2)
        for _ in range(reps):
            flush.fill_(1.0)
            ms += plan.profile(d_pass, d_out, B=P, stream=stream)
        ms /= reps
        k_ms = float(ms[0])
        peak = fp32_peak or 152 * 128 * 2 * 2.070e9 / 1e12
        ach = float(step_flops.sum()) / (k_ms / 1e3) / 1e12
        roof = {"bound": "alu", "achieved": ach, "peak": peak, "unit": "TFLOP/s", "frac": ach / peak,
                "traffic": None,
                "kernel": f"{'qgm_resident_plan (compiled for this plan)' if ex_kind == q.EXEC_COMPILED else 'k_resident'}"
                          f" (whole pass, {ex_chunk} bitstring(s) per CTA, {ex_smem} B shared memory)",
                "algorithmic_flops_per_pass": float(step_flops.sum()), "kernel_ms_per_pass": k_ms,
                "peak_source": "measured FP32 FMA microbenchmark (qgm_measure_fp32_peak)" if fp32_peak else
                               "derived: FP32 lanes x SMs x max SM clock"}
        launches = args.steps

    res = {
        "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps,
        "warmup": max(args.warmup, 3), "ms_per_step": t_ms / args.steps, "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None,
        "dtype": {"fp16": "c64 (GEMM steps split-fp16 x3)", "bf16": "c64 (GEMM steps split-bf16 x6)",
                  "fp32": "c64"}[args.precision],
        "data": "synthetic",
        "config": {"workload": args.workload, "grid": f"{rows}x{cols}", "depth": depth, "batch_per_gpu": B,
                   "bitstrings_per_step": amps_per_step, "seed": 0, "order": info.order_kind,
                   "max_clique": info.max_clique, "steps_per_pass": info.n_steps, "slices": info.n_slices,
                   "workspace_gb": info.workspace_bytes / 1e9, "parallelism": f"replicas{world}",
                   "executor": {1: "stepwise", 2: "resident", 3: "compiled resident"}.get(ex_kind), "chunk": ex_chunk,
                   "gemm_steps": info.n_gemm_steps, "gemm_steps_tensor_core": info.n_gemm_tc_steps,
                   "gemm_precision": args.precision, "autotune": not args.no_autotune,
                   "tc_convert": bool(args.tc_convert),
                   "l2": "flushed between timed steps (264 MB write, untimed); the pass's tensors exceed L2"},
        "error": err,
        "e2e": {"value": e2e, "unit": UNIT, "h2d_bytes_per_step": 8 * amps_per_step,
                "d2h_bytes_per_step": 16 * amps_per_step},
        "roofline": roof,
        "roofline_steps": roof_steps,
        "fp32_peak_tflops_measured": fp32_peak,
        "gpu_launches": launches,
        "clocks": clk.summary() if clk else None,
    }
    # ---- the same passes with each precision of the GEMM steps
    if not args.no_precisions:
        del plan
        torch.cuda.empty_cache()
        per = {}
        for name, prec in PRECISIONS:
            p2 = make_plan(prec)
            ks = max(2, args.steps // 2)
            t2, _ = timed(p2, ks, 1)
            per[name] = {"value": world * amps_per_step * ks / (t2 / 1e3), "ms_per_step": t2 / ks,
                         "gemm_steps_tensor_core": p2.info.n_gemm_tc_steps,
                         "error": error_measures(amplitudes_of(p2, ref[0]), ref[1], n) if ref is not None else None}
            del p2
            torch.cuda.empty_cache()
        res["precisions"] = per
        if per["c64"]["value"]:
            res["speedup_split_fp16_vs_c64"] = per["split_fp16"]["value"] / per["c64"]["value"]
            res["speedup_split_bf16_vs_c64"] = per["split_bf16"]["value"] / per["c64"]["value"]
    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        rate, sample, cores = cpu_oracle_sample(args.workload, c_py, bits)
        res["cpu_baseline"] = {"value": rate, "unit": UNIT, "cores": cores, "kind": "oracle", "sample": sample}
    if rank == 0:
        print(json.dumps(res), flush=True)
    if world > 1:
        dist.destroy_process_group()


if __name__ == "__main__":
    main()
