"""Benchmark of the multi-patch FC-SDNN operator: Euler RHS point-updates/s.

One step = one time step of Algorithm 1 on the workload (viscosity, filter, CFL
time step, five SSPRK-4 stages each followed by the boundary overwrite and the
inter-patch exchange), all patches batched (one launch per pass and length
class), captured once as a CUDA graph and replayed. A point-update is one active
(non-blanked) grid point receiving one RHS evaluation, so a step is 5 x active
points point-updates.

Before timing, fc_autotune times the candidate FFT stage orders and the warps per CTA of the
lines that run as transforms and keeps the fastest (--no-autotune: the cost model's
choices); on the default workload all lines are contracted and it has nothing to choose.

  python bench.py [--gpus N --steps K --warmup W --workload NAME --impl ours|reference]

N > 1 (torchrun): independent replicas, one per GPU (weak scaling); with --shard the
ranks share one workload instead (fc_partition + fc_shard: each rank advances its own
patches, the fringe values, window sums and the time step's minimum go through NCCL;
strong scaling, no graph, no per-patch or adjoint measurement).
--impl reference: the CPU oracle on the host cores, on a bounded sample of the
same workload, same metric and unit.
"""
import argparse
import json
import os
import statistics
import subprocess
import sys
import threading
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "Euler RHS point-updates/s"
UNIT = "point-updates/s"
DEFAULT_WORKLOAD = "cyl_m25_32"


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=10)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--workload", default=DEFAULT_WORKLOAD)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--sample-patches", type=int, default=1)
    ap.add_argument("--no-per-patch", action="store_true")
    ap.add_argument("--shard", action="store_true",
                    help="N > 1: split the workload's patches over the ranks (fc_shard) instead of replicas")
    ap.add_argument("--adjoint-steps", type=int, default=40,
                    help="steps of the adjoint cost measurement (one checkpoint segment by default)")
    ap.add_argument("--adjoint-checkpoint", type=int, default=40, help="checkpoint interval K of that measurement")
    ap.add_argument("--no-autotune", action="store_true",
                    help="keep the cost model's FFT stage orders and the default warps per CTA (skip fc_autotune)")
    return ap.parse_args()


# ---------------------------------------------------------------- CPU oracle on a bounded sample
def oracle_sample_workload(w, npatch, max_points=None):
    """A bounded sample of the workload: its npatch largest affine patches (of at most
    max_points points each, when given and some patch qualifies), each run as a stand-alone
    patch (sides made Dirichlet free stream, no hole), so the sample has the workload's
    line lengths and per-point work without inter-patch coupling."""
    import dataclasses
    from paper_2506_16076_gb300 import workloads as W
    aff = [p for p in w.patches if p.kind == W.AFFINE]
    aff.sort(key=lambda p: -p.npts)
    if max_points is not None and any(p.npts <= max_points for p in aff):
        aff = [p for p in aff if p.npts <= max_points]
    pts = [dataclasses.replace(p, side=(W.DIRICHLET,) * 4, hole=(0.0, 0.0, -1.0)) for p in aff[:npatch]]
    return W.Workload(w.name + "_sample", pts, w.params, w.freestream, w.init, w.steps, w.extra)


def oracle_bench(workload, steps, warmup, npatch, budget_s=None, max_points=None):
    """Time full oracle steps on the sample; returns (point-updates/s, sample description, seconds)."""
    from oracle import solver as S
    from paper_2506_16076_gb300 import workloads as W
    w = W.WORKLOADS[workload]()
    ws = oracle_sample_workload(w, npatch, max_points)
    sv = S.Solver(ws)
    st = W.initial_state(ws)
    active = sum(int((~g.blank).sum()) for g in sv.geos)
    for n in range(warmup):
        st = sv.step(st, n)
    t0 = time.perf_counter()
    done = 0
    for n in range(steps):
        st = sv.step(st, warmup + n)
        done += 1
        if budget_s and time.perf_counter() - t0 > budget_s:
            break
    el = time.perf_counter() - t0
    cap = "" if max_points is None else f" of at most {max_points} points"
    desc = (f"{len(ws.patches)} largest{cap} of the {len(w.patches)} patches of {workload} (stand-alone), "
            f"{active} active points, {done} full steps, long-double FC oracle")
    return active * 5 * done / el, desc, el, done


def oracle_single_patch(steps):
    """Single-thread oracle rate on the 128 x 128 shock tube (all of it, no sampling)."""
    from oracle import solver as S
    from paper_2506_16076_gb300 import workloads as W
    w = W.sod128()
    sv = S.Solver(w)
    st = S.smear_initial(sv, W.initial_state(w), 0.5)
    st = sv.step(st, 0)
    t0 = time.perf_counter()
    for n in range(steps):
        st = sv.step(st, 1 + n)
    el = time.perf_counter() - t0
    return 5 * w.total_points * steps / el, el


def oracle_adjoint_ratio():
    """Oracle adjoint / forward cost on the small cylinder under a Mach-2 stream at 2 degrees
    (the adjoint configuration's geometry and state at a size the oracle runs in seconds):
    one forward step with the viscosity and dt frozen, against one adjoint step (its
    forward recompute included) of the same step."""
    import dataclasses
    import math
    from oracle import adjoint as A, solver as S
    from paper_2506_16076_gb300 import workloads as W
    w0 = W.small_multipatch(W.ADIABATIC)
    a = math.radians(2.0)
    fs = (1.4, 2.0 * math.cos(a), 2.0 * math.sin(a), 1.0)
    w = W.Workload("small_m2", [dataclasses.replace(p, bc=(fs,) * 4) for p in w0.patches], w0.params, fs,
                   "freestream", 1)
    sv = S.Solver(w)
    st = sv.project(W.initial_state(w))
    mu = [0.0 * g.x for g in sv.geos]
    dt = 0.5 * sv.dt(st, mu)
    t0 = time.perf_counter()
    out = A.step_forward(sv, st, mu, dt, filt=True)[0][5]
    t1 = time.perf_counter()
    A.step_adjoint(sv, st, mu, dt, [0.0 * x + 1.0 for x in out], filt=True)
    t2 = time.perf_counter()
    return (t2 - t1) / (t1 - t0), t1 - t0, t2 - t1, w.total_points


def oracle_suite(workload, steps, warmup, npatch, budget_s, max_points=None, extras=True):
    r = {"sample": oracle_bench(workload, steps, warmup, npatch, budget_s, max_points)}
    if extras:
        r["sod128"] = oracle_single_patch(2)
        r["adjoint"] = oracle_adjoint_ratio()
    return r


def run_oracle_subprocess(workload, steps, warmup, npatch, budget_s, max_points=None, extras=False):
    """Run the oracle in a fresh process (spawned before any GPU work of that process), on one
    thread: the long-double numpy oracle does not parallelise, so the thread count is 1 and
    the math libraries are held to it."""
    env = dict(os.environ)
    for k in ("OMP_NUM_THREADS", "OPENBLAS_NUM_THREADS", "MKL_NUM_THREADS"):
        env[k] = "1"
    code = ("import json,sys; sys.path.insert(0, %r); import bench; "
            "r = bench.oracle_suite(%r, %d, %d, %d, %r, %r, %r); print(json.dumps(r))"
            % (ROOT, workload, steps, warmup, npatch, budget_s, max_points, extras))
    out = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, env=env, timeout=900)
    if out.returncode != 0:
        raise RuntimeError(out.stderr[-2000:])
    r = json.loads(out.stdout.strip().splitlines()[-1])
    v, desc, el, done = r["sample"]
    return v, desc, el, done, 1, r


# ---------------------------------------------------------------- clocks sampler
class Clocks:
    def __init__(self):
        self.lines = []
        self.proc = None

    def start(self):
        q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,clocks_event_reasons.hw_slowdown,"
             "clocks_event_reasons.hw_thermal_slowdown,clocks_event_reasons.sw_thermal_slowdown,"
             "clocks_event_reasons.sw_power_cap")
        try:
            self.proc = subprocess.Popen(["nvidia-smi", f"--query-gpu={q}", "--format=csv,noheader,nounits", "-lms",
                                          "200"], stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.th = threading.Thread(target=self._read, daemon=True)
            self.th.start()
        except OSError:
            self.proc = None

    def _read(self):
        for ln in self.proc.stdout:
            self.lines.append(ln.strip())

    def stop(self, dev):
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except subprocess.TimeoutExpired:
            self.proc.kill()
        sm, mx, reasons = [], None, set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for ln in self.lines:
            f = [x.strip() for x in ln.split(",")]
            if len(f) < 9 or f[0] != str(dev):
                continue
            try:
                sm.append(float(f[1]))
                mx = float(f[2])
            except ValueError:
                continue
            for k, nm in enumerate(names):
                if f[5 + k].lower() == "active":
                    reasons.add(nm)
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": mx, "reasons": sorted(reasons),
                "samples": len(sm)}


# ---------------------------------------------------------------- ranks
def combine_ranks(world, pu_step, steps, ms, ms_e2e, device, shared=False):
    """Whole-job rates: times are the maximum over ranks; work is the sum over ranks for
    independent replicas (weak scaling), or the one shared workload's when the ranks split
    it (shared, strong scaling). Returns (ms, ms_e2e, value, e2e)."""
    import torch
    import torch.distributed as dist
    t = torch.tensor([ms, ms_e2e], dtype=torch.float64, device=device)
    if world > 1:
        dist.all_reduce(t, op=dist.ReduceOp.MAX)
    ms, ms_e2e = t[0].item(), t[1].item()
    copies = 1 if shared else world
    return ms, ms_e2e, copies * pu_step * steps / (ms / 1e3), copies * pu_step / (ms_e2e / 1e3)


# ---------------------------------------------------------------- our arm
def peaks():
    p = {}
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as f:
            p = json.load(f)
    except OSError:
        pass
    return p


# the kernels and the host code that chooses their plans and launch shapes
KERNEL_SOURCES = ["fc_kernels.cu", "fc_line.cuh", "fc_internal.h", "fc_host.cpp", "fc_tables.h", "fc_mma.cuh", "fc_mma.cu",
                  "fc_mma_gen.cu", "fc_mma_adj.cu", "fc_mma_adj_gen.cu", "fc_point.cuh", "fc_split.cuh", "fc_mmtab.h"]

# operations that a line pass leaves to the FP64 pipe, per point and per point of a gradient round (fluxes
# or stage combination, the filter's pointwise maps, the lines' scale; a reciprocal counts as six)
FP64_OPS = {"cart_q1": (22, 8), "cart_q2": (22, 8), "filter_q1": (17, 0), "filter_q2": (17, 0)}


def kernel_sources_sha():
    import hashlib
    h = hashlib.sha256()
    for f in KERNEL_SOURCES:
        with open(os.path.join(ROOT, "paper_2506_16076_gb300", "csrc", f), "rb") as fh:
            h.update(fh.read())
    return h.hexdigest()


def measured_traffic(kernel, workload):
    """DRAM bytes (read + write) of one pass of `kernel` from the committed ncu summary
    profiles/traffic_<kernel>_<workload>.txt, or None when there is none or the kernel
    sources changed since it was captured."""
    path = os.path.join(ROOT, "profiles", f"traffic_{kernel}_{workload}.txt")
    try:
        kv = {}
        with open(path) as f:
            for ln in f:
                ln = ln.strip()
                if ln and not ln.startswith("#") and " " in ln:
                    k, v = ln.split(None, 1)
                    kv[k] = v.strip()
    except OSError:
        return None
    if kv.get("kernel_sources_sha256") != kernel_sources_sha():
        return None
    return int(kv["dram_bytes_read_per_pass"]) + int(kv["dram_bytes_write_per_pass"])


def main_ours(args):
    import torch
    import torch.distributed as dist
    from paper_2506_16076_gb300 import fcsdnn, workloads as W

    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    # the CPU baseline runs first, in its own process, before this process touches the GPU
    cpu = None
    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        try:
            v, desc, el, done, cores, r = run_oracle_subprocess(args.workload, 2, 0, args.sample_patches, 30.0,
                                                                extras=True)
            sod_v, sod_s = r["sod128"]
            ratio, f_s, a_s, npts = r["adjoint"]
            cpu = {"value": v, "unit": UNIT, "cores": cores, "kind": "oracle", "sample": desc + f", {el:.1f} s",
                   "threads": "1 (numpy long-double oracle; host cores: %d)" % (os.cpu_count() or 1),
                   "sod128_single_thread": {"value": sod_v, "unit": UNIT, "seconds": round(sod_s, 2),
                                            "sample": "128 x 128 shock tube, 2 full steps"},
                   "adjoint_forward_ratio": {"value": ratio, "forward_s": round(f_s, 2), "adjoint_s": round(a_s, 2),
                                             "sample": f"small O-grid + 2 x 2 cylinder, Mach 2 at 2 deg, {npts} "
                                                       "points, one filtered step, adiabatic wall"}}
        except Exception as ex:  # reported, not fatal
            cpu = {"value": None, "unit": UNIT, "cores": 1, "kind": "oracle", "sample": f"failed: {ex}"}
    if world > 1:
        dist.init_process_group("nccl")
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)

    w = W.WORKLOADS[args.workload]()
    t0 = time.perf_counter()
    ctx = fcsdnn.Context(w)
    init_s = time.perf_counter() - t0
    sharded = world > 1 and args.shard
    if sharded:
        from paper_2506_16076_gb300 import shard as SH
        ctx.shard(world, rank, SH.partition(w, world), SH.DistComm())
    tune = None
    if not args.no_autotune and not sharded:
        t0 = time.perf_counter()
        tune = ctx.autotune()
        tune["s"] = round(time.perf_counter() - t0, 2)
    e0 = torch.from_numpy(W.flatten(W.initial_state(w))).to(dev)
    e = e0.clone()
    dt = torch.zeros(1, dtype=torch.float64, device=dev)
    mu = torch.zeros(ctx.P, dtype=torch.float64, device=dev)
    stream = torch.cuda.Stream(device=dev)
    GRAPH, FILTER, PERPATCH = fcsdnn.STEP_GRAPH, fcsdnn.STEP_FILTER, fcsdnn.STEP_PER_PATCH
    if sharded:  # host-side exchanges between the stages: no captured graph
        GRAPH = 0

    def steps(k, flags, start):
        for n in range(start, start + k):
            ctx.rk_step(e, dt, mu, flags | (FILTER if n >= 1 else 0))

    def barrier():
        if world > 1:
            dist.barrier()

    with torch.cuda.stream(stream):
        steps(args.warmup, GRAPH, 0)
        n0 = args.warmup
        stream.synchronize()
        barrier()
        torch.cuda.synchronize()
        clocks = Clocks()
        clocks.start()
        l0 = ctx.launch_count()
        ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        ev0.record(stream)
        steps(args.steps, GRAPH, n0)
        ev1.record(stream)
        stream.synchronize()
        barrier()
        torch.cuda.synchronize()
        launches = ctx.launch_count() - l0
        ms = ev0.elapsed_time(ev1)
        ck = clocks.stop(local)
        n0 += args.steps
        status = ctx.sync_status(e)

        # per-patch schedule on the same GPU (baseline of the batched launch)
        ms_pp = None
        if not args.no_per_patch and not sharded:
            k_pp = max(1, min(args.steps, 3))
            ev0.record(stream)
            steps(k_pp, PERPATCH, n0)
            ev1.record(stream)
            stream.synchronize()
            ms_pp = ev0.elapsed_time(ev1) / k_pp
            n0 += k_pp

        # per-kernel durations, live, with CUDA events on the launching stream
        ctx.profile_reset()
        ctx.line_stats(reset=True)
        ctx.profile(True)
        steps(2, 0, n0)
        ctx.profile(False)
        prof = ctx.profile_read()
        skip = ctx.line_stats(reset=True)
        n0 += 2

        # adjoint / forward cost at the adjoint configuration's checkpoint interval: nadj filtered
        # steps recorded (mu, dt frozen for the adjoint, a checkpoint every K steps), then the
        # checkpointed reverse sweep (segment replays + adjoint steps); the drag functional's
        # parameter gradients are accumulated on the device as in a gradient run
        from paper_2506_16076_gb300 import adjoint as ADJ
        nadj, kadj = args.adjoint_steps, args.adjoint_checkpoint
        ms_fwd = ms_adj = None
        if not sharded:
            e_adj = e.clone()
            ev0.record(stream)
            eN, tr = ADJ.forward(ctx, e_adj, nadj, kadj, filter=True, first_filtered=0)
            ev1.record(stream)
            stream.synchronize()
            ms_fwd = ev0.elapsed_time(ev1)
            lam = torch.ones_like(eN)
            dparam = torch.zeros(2, dtype=torch.float64, device=dev)
            ev0.record(stream)
            lam0, _ = ADJ.backward(ctx, tr, lam, dparam)
            ev1.record(stream)
            stream.synchronize()
            ms_adj = ev0.elapsed_time(ev1)
            del tr, lam, lam0, eN, e_adj

        # end to end through the public API with host buffers: every step uploads its input
        # state from pinned host memory and reads its result back to pinned host memory.
        # Chained (the headline): a time march through host memory, step n+1 starts from the
        # host copy of step n's result (fc_rk_step_host: H2D, step, D2H in one call). Pipelined
        # (reported beside it): the steps' inputs are independent host states, so step n+1's
        # upload and step n's read-back run on two copy streams while the neighbouring steps
        # compute (device-side staging copies keep the step's own buffers, and with them its
        # captured graph, fixed).
        host = e.cpu().pin_memory()
        host_out = torch.empty_like(host).pin_memory()
        k_e2e = max(1, min(args.steps, 10))
        ctx.rk_step_host(host, dt, mu, GRAPH | FILTER)  # warm-up: captures the step on its device buffer
        n0 += 1
        ev0.record(stream)
        for n in range(n0, n0 + k_e2e):
            # one C-ABI call per step on the host buffer: upload, step, read-back, synchronise
            ctx.rk_step_host(host, dt, mu, GRAPH | FILTER)
        ev1.record(stream)
        stream.synchronize()
        ms_e2e_chain = ev0.elapsed_time(ev1) / k_e2e
        n0 += k_e2e

        h2d, d2h = torch.cuda.Stream(device=dev), torch.cuda.Stream(device=dev)
        stage_in, stage_out = torch.empty_like(e), torch.empty_like(e)
        Ev = torch.cuda.Event
        k_pipe = max(2, min(args.steps, 10))
        ev0.record(stream)
        in_ready, out_free = Ev(), Ev()
        h2d.wait_event(ev0)
        d2h.wait_event(ev0)
        with torch.cuda.stream(h2d):
            stage_in.copy_(host, non_blocking=True)
            in_ready.record(h2d)
        out_free.record(d2h)
        for n in range(n0, n0 + k_pipe):
            stream.wait_event(in_ready)
            e.copy_(stage_in)  # device-side staging copy into the step's own buffer
            consumed = Ev()
            consumed.record(stream)
            if n + 1 < n0 + k_pipe:
                in_ready = Ev()
                with torch.cuda.stream(h2d):
                    h2d.wait_event(consumed)
                    stage_in.copy_(host, non_blocking=True)
                    in_ready.record(h2d)
            ctx.rk_step(e, dt, mu, GRAPH | FILTER)
            stream.wait_event(out_free)
            stage_out.copy_(e)
            out_ready = Ev()
            out_ready.record(stream)
            out_free = Ev()
            with torch.cuda.stream(d2h):
                d2h.wait_event(out_ready)
                host_out.copy_(stage_out, non_blocking=True)
                out_free.record(d2h)
        stream.wait_event(out_free)
        ev1.record(stream)
        stream.synchronize()
        ms_e2e = ev0.elapsed_time(ev1) / k_pipe
        n0 += k_pipe

    pu_step = 5 * ctx.active
    ms, ms_e2e_pipe, value, e2e_pipe = combine_ranks(world, pu_step, args.steps, ms, ms_e2e, dev, sharded)
    _, ms_e2e_chain, _, e2e_chain = combine_ranks(world, pu_step, args.steps, ms, ms_e2e_chain, dev, sharded)
    probe = None
    try:
        probe = fcsdnn.probe_fp64()
    except Exception:  # reported as missing, not fatal
        pass
    if rank != 0:
        if world > 1:
            dist.destroy_process_group()
        return

    # roofline of the dominant line pass: what its kernels do on the three pipes that could bound it
    pk = peaks()
    dom = max((k for k in prof if k in FP64_OPS), key=lambda k: prof[k][0], default=None)
    roof = None
    if dom:
        _, nbytes, nl, npts = ctx.pass_stats(dom)
        products, transformed = ctx.pass_products(dom)
        tot_ms, cnt = prof[dom]
        # one pass launch group covers all its length classes
        passes = 2 * (5 if dom.startswith("cart") else 1)  # profiled 2 steps
        avg_s = tot_ms / 1e3 / passes
        # the gradient round is skipped on lines whose tile has mu == 0 everywhere
        skipped = {"cart_q1": skip[0], "cart_q2": skip[1]}.get(dom, 0) / passes
        viscous = 1.0 - skipped / max(nl, 1)
        rounds = (1.0 + viscous) / 2.0 if dom.startswith("cart") else 1.0
        ops, grad_ops = FP64_OPS[dom]
        fp64_ops = npts * (ops + grad_ops * viscous)
        sm_max = pk.get("sm_max_mhz", 2070.0)
        n_sm = torch.cuda.get_device_properties(dev).multi_processor_count
        pipes = {  # name: (work per pass, peak per second, unit, scale of the unit)
            "alu": (fp64_ops, n_sm * sm_max * 1e6 * 2, "T FP64 operations/s", 1e12),
            "tensor": (products * rounds, pk.get("bf16_tflops", 1900.0) * 1e12, "TFLOP/s", 1e12),
            "hbm": (nbytes, pk.get("hbm_gbs", 6787.9) * 1e9, "GB/s", 1e9)}
        rates = {k: {"work_per_pass": wk, "achieved": round(wk / avg_s / sc, 4), "peak": round(top / sc, 4), "unit": u,
                     "frac": round(wk / avg_s / top, 4)} for k, (wk, top, u, sc) in pipes.items()}
        bound = max(rates, key=lambda k: rates[k]["frac"])
        kname = f"k_mm_{dom}"  # the kernel that takes the pass's lines of contracted lengths
        roof = {"bound": bound, **{k: rates[bound][k] for k in ("achieved", "peak", "unit", "frac")}, "pipes": rates,
                "traffic": measured_traffic(kname, args.workload),
                "traffic_unit": "DRAM bytes per pass (all length-class launches), ncu", "kernel": kname,
                "algorithmic_bytes_per_pass": nbytes, "lines_per_pass": nl, "lines_as_transforms": transformed,
                "inviscid_lines_per_pass": skipped, "pass_ms": round(avg_s * 1e3, 3),
                "launches_per_pass": cnt // passes,
                "note": f"alu: FP64 pipe, {n_sm} SMs (device query) x 2 operations/clk x max SM clock {sm_max:.0f} MHz; "
                        "tensor: digit products at the measured bf16 rate (FP16 has the same; mma.sync does not reach it); "
                        "hbm: compulsory bytes at the measured copy rate. No pipe is full: latencies between a tile's "
                        "phases set the pace",
                "probe_TFLOPs": None if probe is None else {"dfma": round(probe[0] / 1e3, 4),
                                                            "dmma": round(probe[1] / 1e3, 4),
                                                            "source": "fc_probe_fp64, this run"}}
    out = {
        "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": ms / args.steps, "higher_is_better": True,
        "scaling": "strong" if sharded else "weak",
        "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "config": {"workload": args.workload, "points": ctx.P, "active_points": ctx.active,
                   "patches": len(w.patches), "schedule": "batched, one launch per pass and length class, CUDA graph",
                   "l2": "inputs larger than L2 (state %.2f GB)" % (32 * ctx.P / 1e9),
                   "parallelism": ("sharded patches, NCCL exchange" if sharded else "replicas") if world > 1
                   else "1 GPU", "init_s": round(init_s, 2),
                   "autotune": tune},
        "per_patch": None if ms_pp is None else {"value": world * pu_step / (ms_pp / 1e3), "ms_per_step": ms_pp,
                                                 "batched_speedup": ms_pp / (ms / args.steps)},
        "kernels_ms_per_step": {k: round(v[0] / 2, 3) for k, v in sorted(prof.items(), key=lambda x: -x[1][0])},
        "adjoint": None if ms_fwd is None else {
            "steps": nadj, "checkpoint_every": kadj, "filter": True, "forward_ms": ms_fwd, "adjoint_ms": ms_adj,
            "adjoint_forward_ratio": ms_adj / ms_fwd,
            "note": "forward = filtered steps with mu/dt recorded and checkpoints; adjoint = segment replays + "
                    "fc_adjoint_step per step with the parameter gradients accumulated"},
        "roofline": roof,
        "cpu_baseline": cpu,
        "e2e": {"value": e2e_chain, "unit": UNIT, "h2d_bytes_per_step": 32 * ctx.P,
                "d2h_bytes_per_step": 32 * ctx.P, "ms_per_step": ms_e2e_chain, "steps": k_e2e,
                "schedule": "chained time march of a pinned host state through fc_rk_step_host (one C-ABI call "
                            "per step: H2D, step, D2H, synchronise)",
                "independent_inputs_pipelined": {
                    "value": e2e_pipe, "ms_per_step": ms_e2e_pipe, "steps": k_pipe,
                    "schedule": "independent host inputs: step n+1's upload and step n's read-back on two copy "
                                "streams overlap the neighbouring steps' compute"}},
        "gpu_launches": launches,
        "clocks": ck,
        "state_status": int(status),
    }
    print(json.dumps(out))
    if world > 1:
        dist.destroy_process_group()


def main_reference(args):
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return
    # each step a bounded sample: patches small enough that the K + W oracle steps take about
    # two minutes at the slowest host rate seen for this oracle (3.5e4 point-updates/s, the
    # Arm cores, where long double is quad precision in software)
    max_points = max(4096, int(120.0 * 3.5e4 / 5.0 / max(1, args.steps + args.warmup)))
    v, desc, el, done, cores, _ = run_oracle_subprocess(args.workload, args.steps, args.warmup,
                                                        args.sample_patches, None, max_points)
    out = {"metric": METRIC, "value": v, "unit": UNIT, "n_gpus": args.gpus, "steps": done, "warmup": args.warmup,
           "ms_per_step": el / max(done, 1) * 1e3, "higher_is_better": True, "scaling": "weak",
           "vs_baseline": None, "dtype": "f64", "data": "synthetic", "impl": "reference",
           "config": {"workload": args.workload},
           "cpu_baseline": {"value": v, "unit": UNIT, "cores": cores, "kind": "oracle", "sample": desc},
           "e2e": {"value": v, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(out))


if __name__ == "__main__":
    a = parse()
    if a.impl == "reference":
        main_reference(a)
    else:
        main_ours(a)
