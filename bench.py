#!/usr/bin/env python
"""Benchmark: source-pixel visits per second of the per-source ELBO with its
gradient and Hessian, inside one trust-region Newton pass over a field.

One step = one Newton trust-region iteration on every source of the field,
colour class by colour class (sources of a class do not overlap, so they are
updated together; the background of each class reflects the classes before
it).  Each iteration evaluates L_s, its gradient and Hessian (the visits
counted), solves the FP64 trust-region subproblem and evaluates the trial
point.  Every timed step starts from the same parameters, so each one does
the full work.

Default workload: a field of five 2048 x 1489 images (one per band) with 600
sources, 30 % stars (the shape of the paper's synthetic study set).  Inputs
are seeded synthetic data.

    python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference]
"""
from __future__ import annotations

import argparse
import json
import math
import os
import subprocess
import sys
import tempfile
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

import fields  # noqa: E402

METRIC = "source-pixel visits/s (ELBO+grad+Hessian)"
UNIT = "visits/s"
# Algorithmic FP32 work of one visit in the derivative pixel kernel (value,
# 10 first and 52 second derivatives over the per-image natural coordinates,
# 48 galaxy + 3 star Gaussian components; FMA = 2 FLOP), counted on the
# direct formulation: every component's Hermite polynomials from its own
# offset and precision.  The kernel shares the offsets of the components of
# one PSF component and stages pixel-independent constants, and executes
# EXECUTED_FLOP_PER_VISIT; the roofline reports both fractions.  Both count
# every pair of components: in large patches the kernel skips the pairs that
# vanish exactly (about a fifth of them in blends), so frac_executed is an
# upper bound of the pipes' own utilisation there.
FLOP_PER_VISIT = 5320
EXECUTED_FLOP_PER_VISIT = 4723
FP32_LANES_PER_SM = 128
SEED = 1803_00113


def parse_args(argv=None):
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=10)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", choices=["ours", "reference"], default="ours")
    ap.add_argument("--workload", choices=["batched", "field", "serving", "first-order", "mcmc"],
                    default="batched")
    ap.add_argument("--no-field", action="store_true",
                    help="batched: skip the single-field run reported beside the headline")
    ap.add_argument("--no-serving", action="store_true",
                    help="skip the short serving run reported beside the headline")
    ap.add_argument("--derivs-reps", type=int, default=0,
                    help="derivs-only: time the derivative kernel over this many further calls")
    ap.add_argument("--derivs-only", action="store_true",
                    help="profiling case: plan the first colour class of a batched problem of "
                         "--sources sources (default 2000) and evaluate it twice")
    ap.add_argument("--mcmc-sources", type=int, default=16,
                    help="mcmc: sources of the field sampled (the brightest)")
    ap.add_argument("--rates", default="50,200,500,1000,2000",
                    help="serving: Poisson arrival rates (requests/s)")
    ap.add_argument("--serve-seconds", type=float, default=2.0,
                    help="serving: arrival window per rate")
    ap.add_argument("--pool", type=int, default=96, help="serving: distinct requests generated")
    ap.add_argument("--workers", type=int, default=0,
                    help="serving: worker threads (0: the server's default)")
    ap.add_argument("--serve-tile", type=int, default=128,
                    help="serving: pixels per tile of the pixel kernels")
    ap.add_argument("--fo-max-steps", type=int, default=3000,
                    help="first-order comparison: step cap of the L-BFGS subsolver")
    ap.add_argument("--sources", type=int, default=0, help="override the source count")
    ap.add_argument("--no-graph", action="store_true")
    ap.add_argument("--no-cache", action="store_true",
                    help="re-render neighbours for every background instead of caching renders")
    ap.add_argument("--no-plain", action="store_true")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--cpu-seconds", type=float, default=12.0)
    ap.add_argument("--no-autotune", action="store_true",
                    help="keep the default 256-pixel tiles instead of picking tile shapes per "
                         "patch-size bucket before timing")
    ap.add_argument("--tiles", default=None,
                    help="pixels per work item for the four patch-area buckets, comma-separated "
                         "(0 = default); replaces the autotuner")
    ap.add_argument("--plain-sample", type=int, default=600,
                    help="sources timed in the plain one-source-per-launch form")
    return ap.parse_args(argv)


def workload(name, n_sources, seed):
    if name == "field":
        n = n_sources or 600
        p = fields.single_field(seed=seed, n_sources=n)
        cfg = {"workload": "single field: 5 bands x 1 image of 2048x1489 px, "
                           f"{n} sources (30% stars), log-normal fluxes, one Newton "
                           "trust-region pass in colour classes",
               "bands": 5, "image_px": [2048, 1489], "sources": n}
    else:
        n = n_sources or 8192
        p = fields.batched(seed=seed, n_sources=n)
        cfg = {"workload": f"batched: {n} sources, patches 15..101 px, 1..6 images per band, "
                           "0..10 neighbours, one Newton trust-region pass in colour classes",
               "sources": n}
    return p, cfg


# ---------------------------------------------------------------------------
# distributed plumbing (one process per GPU; sources shard with no exchange)
# ---------------------------------------------------------------------------

def dist_info():
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return world, rank, local


def dist_init(world, backend):
    import torch.distributed as dist
    if world > 1 and not dist.is_initialized():
        dist.init_process_group(backend=backend)
    return dist


def barrier(world):
    if world > 1:
        import torch.distributed as dist
        dist.barrier()


def reduce_max(value, world, device="cpu"):
    """Maximum of a float over ranks (the job's time is its slowest rank)."""
    if world <= 1:
        return value
    import torch
    import torch.distributed as dist
    t = torch.tensor([float(value)], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def reduce_sum(value, world, device="cpu"):
    if world <= 1:
        return value
    import torch
    import torch.distributed as dist
    t = torch.tensor([float(value)], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.SUM)
    return float(t.item())


# ---------------------------------------------------------------------------
# clocks during the timed region
# ---------------------------------------------------------------------------

class ClockSampler:
    QUERY = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
             "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
             "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, index):
        self.index = index
        self.proc = None
        self.path = None
        self.n0 = 0

    def _lines(self):
        try:
            with open(self.path) as f:
                return sum(1 for _ in f)
        except OSError:
            return 0

    def _wait_for(self, n, timeout=5.0):
        t0 = time.time()
        while self._lines() < n and time.time() - t0 < timeout and self.proc.poll() is None:
            time.sleep(0.01)

    def start(self):
        """Starts sampling every 50 ms and returns once the first reading is
        in, so that the readings bracket the timed region that follows."""
        try:
            fd, self.path = tempfile.mkstemp(suffix=".csv")
            os.close(fd)
            self.proc = subprocess.Popen(
                ["nvidia-smi", f"--query-gpu={self.QUERY}", "--format=csv,noheader,nounits",
                 "-lms", "50", "-i", str(self.index)],
                stdout=open(self.path, "w"), stderr=subprocess.DEVNULL)
        except (OSError, FileNotFoundError):
            self.proc = None
            return
        self._wait_for(1)
        self.n0 = self._lines()

    def stop(self):
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        self._wait_for(self.n0 + 1)          # one reading after the timed region
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except subprocess.TimeoutExpired:
            self.proc.kill()
        rows = []
        for line in open(self.path):
            parts = [x.strip() for x in line.split(",")]
            if len(parts) >= 9:
                rows.append(parts)
        os.unlink(self.path)
        sm = [float(r[1]) for r in rows if r[1].replace(".", "").isdigit()]
        mx = [float(r[2]) for r in rows if r[2].replace(".", "").isdigit()]
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        reasons = sorted({names[k] for r in rows for k in range(4) if r[5 + k].lower() == "active"})
        return {"sm_mhz": float(np.median(sm)) if sm else None,
                "sm_max_mhz": max(mx) if mx else None, "samples": len(rows), "reasons": reasons}


# ---------------------------------------------------------------------------
# the CPU baseline: the oracle on a bounded sample of the same workload
# ---------------------------------------------------------------------------

def cpu_baseline(problem, seconds, order=None, threads=None):
    """The oracle's ELBO, gradient and Hessian of sources of the workload,
    in the given order, until `seconds` of CPU work (on `threads` threads,
    default all the host's cores)."""
    import torch
    import oracle
    order = list(range(problem.n_sources)) if order is None else order
    prev = torch.get_num_threads()
    if threads:
        torch.set_num_threads(threads)
    try:
        t_total, visits, used = 0.0, 0, []
        for s in order:
            t0 = time.perf_counter()
            oracle.elbo_grad_hess(problem, s)
            t_total += time.perf_counter() - t0
            visits += problem.visits([s])
            used.append(s)
            if t_total >= seconds:
                break
        cores = torch.get_num_threads()
    finally:
        torch.set_num_threads(prev)
    return {"value": visits / t_total, "unit": UNIT, "cores": cores,
            "kind": "oracle",
            "sample": f"FP64 oracle ELBO+gradient+Hessian of {len(used)} of the workload's "
                      f"{problem.n_sources} sources ({visits} visits, {t_total:.1f} s)",
            "seconds_per_source": t_total / len(used)}


def parse_tiles(text):
    """--tiles: four comma-separated non-negative pixels-per-item counts."""
    try:
        tiles = [int(t) for t in text.split(",")]
    except ValueError:
        tiles = []
    if len(tiles) != 4 or any(t < 0 for t in tiles):
        raise SystemExit("--tiles wants four non-negative integers, e.g. 128,256,0,0")
    return tiles


def derivs_source_hash(path):
    """Hash of the derivative kernel's source and build flags: pixel.cu up to
    the next kernel (its device helpers and derivs_kernel itself)."""
    import hashlib
    import re
    from paper_1803_00113_gb300 import build_lib
    text = open(path, "rb").read()
    cut = text.find(b"__global__ void __launch_bounds__(128) grad_kernel")
    text = text[:cut if cut > 0 else len(text)]
    # the code only: line comments and spacing do not change the kernel
    text = re.sub(rb"//[^\n]*", b"", text)
    text = re.sub(rb"\s+", b" ", text)
    # include paths name this checkout's location: leave them out
    flags = " ".join(f for f in build_lib.FLAGS + build_lib.FILE_FLAGS.get("pixel.cu", [])
                     if not f.startswith("-I")).encode()
    return hashlib.sha256(text + flags).hexdigest()[:16]


def traffic_per_launch(visits_per_launch):
    """DRAM bytes per derivative-kernel launch from the committed ncu summary,
    scaled by visits, when the summary was taken on the current kernel source."""
    import hashlib
    path = os.path.join(ROOT, "profiles", "derivs_kernel_dram.json")
    src = os.path.join(ROOT, "paper_1803_00113_gb300", "csrc", "pixel.cu")
    if not os.path.exists(path):
        return None
    d = json.load(open(path))
    if d.get("derivs_source_sha256_16") != derivs_source_hash(src):
        return None
    return d["dram_bytes_per_visit"] * visits_per_launch


# ---------------------------------------------------------------------------
# our implementation
# ---------------------------------------------------------------------------

class NewtonPass:
    """One Newton trust-region iteration on every source of a problem, colour
    class by colour class, as one captured CUDA graph (the bench's step).

    Every step starts from the same state: theta, the trust radii, the
    statuses and (with a render cache) the cached renders of theta, restored
    between steps outside the timed events, as the previous iteration of a
    fit leaves them (a fit keeps the cache current by committing the trial
    renders of accepted steps, which the step does)."""

    def __init__(self, cel, ctx, dp, classes, tiles, stream, graph=True):
        import torch
        self.cel, self.ctx, self.dp, self.stream = cel, ctx, dp, stream
        self.plans = [cel.Plan(ctx, dp, c, ppi_bucket=tiles) for c in classes]
        self.visits = sum(p.visits for p in self.plans)
        self.delta, self.status = cel.newton_state(dp)
        self.theta0 = dp.theta.clone()
        self.delta0, self.status0 = self.delta.clone(), self.status.clone()
        self.render_all()
        self.cache0 = dp.cache.clone() if dp.cache is not None else None
        self.half0 = dp.cache_half.clone() if dp.cache is not None else None
        self.graph = None
        # the library counts the kernels it launches: one eager step's worth
        self.reset()
        l0 = ctx.launches()
        self.step_eager()                         # also the warm-up before a capture
        self.n_launch = ctx.launches() - l0
        if graph:
            self.reset()
            # event timing of the derivative kernel is recorded into the graph
            # and so runs on every replay (read with reset=False after each)
            ctx.profile(True)
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=stream):
                self.step_eager()
            stream.synchronize()
            self.graph = g

    def render_all(self):
        if self.dp.cache is not None:
            for p in self.plans:
                self.cel.render_cache(p)

    def reset(self):
        self.dp.theta.copy_(self.theta0)
        self.delta.copy_(self.delta0)
        self.status.copy_(self.status0)
        if self.cache0 is not None:
            self.dp.cache.copy_(self.cache0)
            self.dp.cache_half.copy_(self.half0)

    def step_eager(self):
        for p in self.plans:
            self.cel.newton_step(p, self.delta, self.status)

    def step(self):
        if self.graph is not None:
            self.graph.replay()
        else:
            self.step_eager()

    def launches_per_step(self):
        return self.n_launch

    def close(self):
        for p in self.plans:
            p.close()


def time_steps(pas, steps, flush, timed_kinds=("derivs",)):
    """Times `steps` steps with CUDA events on the launching stream, L2
    flushed between steps (outside the events).  Returns per-step ms and the
    event-timed kernels of the kinds in timed_kinds, summed over the steps."""
    import torch
    ctx, stream = pas.ctx, pas.stream
    if pas.graph is None:
        ctx.profile(True, kinds=list(timed_kinds))
    by_kind = {k: [0.0, 0, 0] for k in pas.cel.KERNEL_KINDS}
    ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True))
          for _ in range(steps)]
    for k in range(steps):
        pas.reset()
        flush.zero_()
        ev[k][0].record(stream)
        pas.step()
        ev[k][1].record(stream)
        stream.synchronize()
        for kind, (ms, nl, nv) in ctx.profile_kernels(reset=pas.graph is None).items():
            if kind in timed_kinds:
                by_kind[kind][0] += ms
                by_kind[kind][1] += nl
                by_kind[kind][2] += nv
    if pas.graph is None:
        ctx.profile(False)
    return [a.elapsed_time(b) for a, b in ev], by_kind


def kernel_breakdown(pas, flush):
    """Every kernel kind of one eager step, event-timed (kept out of the
    timed region, where only the derivative kernel is timed)."""
    import torch
    pas.ctx.profile(True, kinds="all")
    pas.reset()
    flush.zero_()
    pas.step_eager()
    torch.cuda.synchronize()
    out = {k: {"ms": ms, "launches": nl} for k, (ms, nl, _) in
           pas.ctx.profile_kernels(reset=True).items() if nl}
    pas.ctx.profile(False)
    return out


def setup_problem(cel, problem, dev, stream, args, local):
    """Context, device problem (render cache where neighbours are dense),
    colour classes and tiles (autotuned unless given)."""
    ctx = cel.Context(problem.model, device=local, stream=stream)
    # cache renders where neighbours are dense (blends); in a sparse
    # field re-rendering the few neighbours is cheaper than the cache
    dense = problem.nbr_ptr[-1] >= 1.5 * problem.n_sources
    dp = cel.DeviceProblem(problem, dev, render_cache=dense and not args.no_cache)
    classes = cel.color_classes(problem)
    tiles = None
    if args.tiles:
        tiles = parse_tiles(args.tiles)
    elif not args.no_autotune:
        from paper_1803_00113_gb300.autotune import autotune
        tiles, _ = autotune(ctx, dp, range(problem.n_sources), reps=2, groups=classes)
        dp.set_theta(problem.theta)
    return ctx, dp, classes, tiles


def field_summary(cel, args, dev, stream, local, flush, rank):
    """The 600-source single field (the shape of the paper's study set): a
    short timed run of the same Newton pass, reported beside the headline."""
    import torch
    problem, cfg = workload("field", 0, SEED + 1 + rank)
    with torch.cuda.stream(stream):
        ctx, dp, classes, tiles = setup_problem(cel, problem, dev, stream, args, local)
        pas = NewtonPass(cel, ctx, dp, classes, tiles, stream, graph=not args.no_graph)
        for _ in range(3):
            pas.reset()
            pas.step()
        step_ms, by_kind = time_steps(pas, max(args.steps, 10), flush)
        breakdown = kernel_breakdown(pas, flush)
        pas.close()
    return {"workload": cfg["workload"], "visits_per_step": pas.visits,
            "value": pas.visits / (np.mean(step_ms) / 1e3), "unit": UNIT,
            "ms_per_step": float(np.mean(step_ms)), "colour_classes": len(classes),
            "tiles_per_area_bucket": tiles or [256, 256, 256, 256],
            "kernels_one_step": breakdown}


def run_ours(args):
    import torch
    world, rank, local = dist_info()
    dist_init(world, "nccl")
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    from paper_1803_00113_gb300 import build_lib
    build_lib.build()
    from paper_1803_00113_gb300 import celeste as cel

    if args.derivs_only:
        return derivs_only_case(cel, args)

    problem, cfg = workload(args.workload, args.sources, SEED + 1 + rank)
    stream = torch.cuda.Stream(dev)
    flush = torch.empty(256 * 1024 * 1024 // 4, dtype=torch.float32, device=dev)
    with torch.cuda.stream(stream):
        ctx, dp, classes, tiles = setup_problem(cel, problem, dev, stream, args, local)
        pas = NewtonPass(cel, ctx, dp, classes, tiles, stream, graph=not args.no_graph)
        visits = pas.visits
        for _ in range(max(args.warmup, 1)):
            pas.reset()
            pas.step()
        torch.cuda.synchronize(dev)

        # ---- timed region: K steps, L2 flushed between steps (outside the events)
        barrier(world)
        torch.cuda.synchronize(dev)
        clocks = ClockSampler(local)
        clocks.start()
        l0 = ctx.launches()
        step_ms, by_kind = time_steps(pas, args.steps, flush)
        torch.cuda.synchronize(dev)
        clk = clocks.stop()
        kern_ms, kern_launch, kern_visits = by_kind["derivs"]
        n_launch = ctx.launches() - l0
        if pas.graph is not None:
            # a replay launches the captured kernels: count them per step
            n_launch += args.steps * pas.launches_per_step()
        barrier(world)
        total_s = reduce_max(sum(step_ms) / 1e3, world, dev)
        all_visits = reduce_sum(visits * args.steps, world, dev)
        value = all_visits / total_s

        breakdown = kernel_breakdown(pas, flush)

        # ---- end to end through the public API, host buffers: every step
        # uploads the pixels and theta, renders the cache of the uploaded
        # theta (when the problem keeps one), runs the Newton pass and
        # reads theta back
        pin_pix = torch.from_numpy(problem.pixels).pin_memory()
        pin_theta = torch.from_numpy(problem.theta.copy()).pin_memory()
        out_theta = torch.empty_like(pin_theta).pin_memory()
        h2d = pin_pix.numel() * 4 + pin_theta.numel() * 8
        d2h = out_theta.numel() * 8
        barrier(world)
        torch.cuda.synchronize(dev)
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        for k in range(args.steps):
            dp.pixels.copy_(pin_pix, non_blocking=True)
            dp.theta.copy_(pin_theta, non_blocking=True)
            pas.delta.copy_(pas.delta0)
            pas.status.copy_(pas.status0)
            pas.render_all()
            pas.step()
            out_theta.copy_(dp.theta, non_blocking=True)
        e1.record(stream)
        torch.cuda.synchronize(dev)
        e2e_s = reduce_max(e0.elapsed_time(e1) / 1e3, world, dev)
        e2e_value = all_visits / e2e_s

        # ---- the plain one-source-per-launch form (same kernels)
        plain = None
        if not args.no_plain and rank == 0:
            order = [int(s) for c in classes for s in c]
            if len(order) > args.plain_sample:
                pick = np.linspace(0, len(order) - 1, args.plain_sample).round().astype(int)
                order = [order[k] for k in pick]
            single = {s: cel.Plan(ctx, dp, [s]) for s in order}
            pas.reset()
            for s in order[:20]:
                cel.newton_step(single[s], pas.delta, pas.status)
            torch.cuda.synchronize(dev)
            pas.reset()
            torch.cuda.synchronize(dev)
            t0 = time.perf_counter()
            for s in order:
                cel.newton_step(single[s], pas.delta, pas.status)
                stream.synchronize()
            plain_s = time.perf_counter() - t0
            pv = problem.visits(order)
            plain = {"value": pv / plain_s, "unit": UNIT, "sources_timed": len(order),
                     "ms_per_source": plain_s * 1e3 / len(order),
                     "form": "one source per launch sequence, host sync after each source"}
            for pl in single.values():
                pl.close()

        # ---- gradient-only pass vs gradient + Hessian (the paper's cost ratio):
        # whole calls, and the pixel kernels alone (the calls share the
        # neighbour-background kernel, which is the same work in both)
        big = max(pas.plans, key=lambda p: p.visits)
        ratio = {"visits": big.visits}
        for name, fn, kind in (("grad_hess", cel.elbo_grad_hess, "derivs"),
                               ("grad_only", cel.elbo_grad, "grad")):
            fn(big)
            torch.cuda.synchronize(dev)
            ctx.profile(True, kinds="all")
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record(stream)
            for _ in range(5):
                fn(big)
            b.record(stream)
            torch.cuda.synchronize(dev)
            kinds = ctx.profile_kernels(reset=True)
            ctx.profile(False)
            ratio[name + "_call_ms"] = a.elapsed_time(b) / 5
            ratio[name + "_pixel_kernel_ms"] = kinds[kind][0] / max(kinds[kind][1], 1)
            ratio[name + "_epilogue_ms"] = kinds["epilogue"][0] / max(kinds["epilogue"][1], 1)
        ratio["hess_over_grad_call"] = ratio["grad_hess_call_ms"] / ratio["grad_only_call_ms"]
        ratio["hess_over_grad_pixel_kernel"] = (ratio["grad_hess_pixel_kernel_ms"]
                                                / ratio["grad_only_pixel_kernel_ms"])

        # ---- the full-field ELBO (every pixel of every image, all KLs)
        fe = cel.FieldElbo(ctx, dp)
        fe()
        torch.cuda.synchronize(dev)
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record(stream)
        for _ in range(5):
            fe()
        b.record(stream)
        torch.cuda.synchronize(dev)
        field_elbo = {"ms": a.elapsed_time(b) / 5, "value": float(fe.out[0]),
                      "pixels": int(problem.pixels.size)}
        fe.close()
        pas.close()

    extra_field = None
    if args.workload == "batched" and not args.no_field:
        extra_field = field_summary(cel, args, dev, stream, local, flush, rank)
    serving = None
    if not args.no_serving and world == 1:
        serving = serving_summary(cel, args, local)
    differentiation = None
    if args.workload == "batched" and not args.no_field:
        differentiation = differentiation_summary(cel, dev, local)

    # ---- roofline of the derivative pixel kernel
    props = torch.cuda.get_device_properties(dev)
    sm_max = clk.get("sm_max_mhz") or 2070.0
    peak = props.multi_processor_count * FP32_LANES_PER_SM * 2 * sm_max * 1e6 / 1e12
    per_launch_visits = kern_visits / max(kern_launch, 1)
    avg_ms = kern_ms / max(kern_launch, 1)
    achieved = FLOP_PER_VISIT * per_launch_visits / (avg_ms / 1e3) / 1e12 if kern_launch else None
    traffic = traffic_per_launch(per_launch_visits)

    if rank != 0:
        return None
    line = {
        "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": float(np.mean(step_ms)),
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
        "dtype": "f32", "data": "synthetic (seeded fields shaped like the paper's study set)",
        "config": dict(cfg, l2="flushed between steps (256 MB write outside the timed events)",
                       graph=pas.graph is not None, visits_per_step=visits,
                       colour_classes=len(classes),
                       tiles_per_area_bucket=tiles or [256, 256, 256, 256],
                       tile_tuning=("given (--tiles)" if args.tiles else
                                    "composed: the step's colour-class plans, every kernel timed"
                                    if tiles else "default 256 pixels per item"),
                       render_cache=dp.cache is not None,
                       state_between_steps="theta, trust radii, statuses and the render cache "
                                           "of theta restored outside the timed events"),
        "step_ms_p50": float(np.percentile(step_ms, 50)),
        "step_ms_p99": float(np.percentile(step_ms, 99)),
        "grad_vs_hess": ratio,
        "kernels_one_step": breakdown,
        "full_field_elbo": field_elbo,
        "e2e": {"value": e2e_value, "unit": UNIT, "h2d_bytes_per_step": int(h2d),
                "d2h_bytes_per_step": int(d2h),
                "includes": "pixel and theta upload, render cache of the uploaded theta, the "
                            "Newton pass, theta download"},
        "gpu_launches": int(n_launch),
        "gpu_launches_per_step": pas.launches_per_step(),
        "clocks": clk,
        "roofline": {"bound": "alu", "achieved": achieved, "peak": peak, "unit": "TFLOP/s",
                     "frac": (achieved / peak) if achieved else None,
                     "traffic": traffic, "kernel": "derivs_kernel",
                     "kernel_ms_per_launch": avg_ms, "visits_per_launch": per_launch_visits,
                     "flop_per_visit": FLOP_PER_VISIT,
                     "frac_at_4200_flop_per_visit": (achieved / peak * 4200 / FLOP_PER_VISIT)
                     if achieved else None,
                     "executed_flop_per_visit": EXECUTED_FLOP_PER_VISIT,
                     "frac_executed": (achieved / peak * EXECUTED_FLOP_PER_VISIT / FLOP_PER_VISIT)
                     if achieved else None,
                     "peak_basis": f"{props.multi_processor_count} SMs x {FP32_LANES_PER_SM} FP32 "
                                   f"lanes x 2 FLOP x {sm_max:.0f} MHz (unit counts, maximum "
                                   "SM clock)"},
        "plain_per_source": plain,
    }
    if plain:
        line["vs_plain"] = value / plain["value"]
    if extra_field:
        line["single_field"] = extra_field
    if serving:
        line["serving"] = serving
    if differentiation:
        line["differentiation"] = differentiation
    if not args.no_cpu_baseline and world == 1:
        rng = np.random.default_rng(0)
        order = list(rng.permutation(problem.n_sources))
        line["cpu_baseline"] = cpu_baseline(problem, args.cpu_seconds, order)
        line["cpu_baseline"]["one_core"] = cpu_baseline(problem, args.cpu_seconds, order, threads=1)
    return line


def derivs_only_case(cel, args):
    """A small case for profiler captures of single kernels: a batched
    problem of --sources sources (default 2,000, whose pixels exceed L2),
    its first colour class planned, elbo_grad_hess called twice (a capture
    skips the first derivative-kernel launch and takes the second)."""
    n = args.sources or 2000
    p = fields.batched(seed=SEED + 3, n_sources=n)
    ctx = cel.Context(p.model)
    dp = cel.DeviceProblem(p)
    tiles = parse_tiles(args.tiles) if args.tiles else None
    plan = cel.Plan(ctx, dp, cel.color_classes(p)[0], ppi_bucket=tiles)
    for _ in range(2):
        cel.elbo_grad_hess(plan)
    ctx.synchronize()
    out = {"case": "derivs-only", "sources": n, "visits": plan.visits,
           "pixels_mb": p.pixels.nbytes / 1e6}
    if args.derivs_reps:
        # event-timed derivative kernel of further calls
        ctx.profile(True)
        for _ in range(args.derivs_reps):
            cel.elbo_grad_hess(plan)
        ms, nl, nv = ctx.profile_read(reset=True)
        ctx.profile(False)
        import torch
        props = torch.cuda.get_device_properties(torch.cuda.current_device())
        peak = props.multi_processor_count * FP32_LANES_PER_SM * 2 * 2070e6 / 1e12
        tf = FLOP_PER_VISIT * nv / (ms / 1e3) / 1e12
        out.update(derivs_ms_per_launch=ms / nl, visits_per_s=nv / (ms / 1e3),
                   frac=tf / peak, frac_at_4200_flop_per_visit=tf / peak * 4200 / FLOP_PER_VISIT)
    return out


# ---------------------------------------------------------------------------
# the reference arm: the FP64 oracle on the host cores
# ---------------------------------------------------------------------------

def run_reference_serving(args):
    """The oracle's region fit on single-source requests of the serving
    pool (the smallest requests; a bounded sample)."""
    import torch
    from oracle import newton as ON
    times = []
    k = 0
    for i in range(args.warmup + args.steps):
        q = fields.region_request(SEED + 5 + k, n_sources=1, side=32)
        k += 1
        t0 = time.perf_counter()
        ON.region_fit(q, max_passes=5, max_iter=50, pass_tol=1e-3)
        if i >= args.warmup:
            times.append(time.perf_counter() - t0)
    value = len(times) / sum(times)
    sample = (f"each step: FP64 oracle region fit of one 1-source, 32x32 px request "
              f"({args.steps} steps)")
    return {"impl": "reference", "metric": "region fits/s (Poisson arrivals, result back on the host)",
            "value": value, "unit": "fits/s", "n_gpus": 1, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": 1e3 * float(np.mean(times)),
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
            "data": "synthetic (seeded region requests)",
            "config": {"workload": "serving (oracle: smallest requests, one at a time)"},
            "cpu_baseline": {"value": value, "unit": "fits/s", "cores": torch.get_num_threads(),
                             "kind": "oracle", "sample": sample},
            "e2e": {"value": value, "unit": "fits/s", "h2d_bytes_per_step": 0,
                    "d2h_bytes_per_step": 0}}


def run_reference(args):
    world, rank, local = dist_info()
    if rank != 0:
        return None
    if args.workload == "serving":
        return run_reference_serving(args)
    import torch
    import oracle
    problem, cfg = workload(args.workload, args.sources, SEED + 1)
    rng = np.random.default_rng(0)
    order = list(rng.permutation(problem.n_sources))
    per_step = 1
    times, visits = [], 0
    k = 0
    for i in range(args.warmup + args.steps):
        srcs = [order[(k + j) % len(order)] for j in range(per_step)]
        k += per_step
        t0 = time.perf_counter()
        for s in srcs:
            oracle.elbo_grad_hess(problem, s)
        dt = time.perf_counter() - t0
        if i >= args.warmup:
            times.append(dt)
            visits += problem.visits(srcs)
    value = visits / sum(times)
    sample = (f"each step: FP64 oracle ELBO+gradient+Hessian of {per_step} sources of the "
              f"workload ({visits} visits over {args.steps} steps)")
    return {"impl": "reference", "metric": METRIC, "value": value, "unit": UNIT,
            "n_gpus": world, "steps": args.steps, "warmup": args.warmup,
            "ms_per_step": 1e3 * float(np.mean(times)), "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f64",
            "data": "synthetic (seeded fields shaped like the paper's study set)",
            "config": cfg,
            "cpu_baseline": {"value": value, "unit": UNIT, "cores": torch.get_num_threads(),
                             "kind": "oracle", "sample": sample},
            "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}


# ---------------------------------------------------------------------------
# serving: region fits submitted at Poisson arrival times
# ---------------------------------------------------------------------------

def _serve_run(cel, srv, pool, arrivals):
    """Submits pool requests (cycled) at the given arrival times; returns the
    per-request results (latency measured natively, submit -> ready)."""
    tickets = []
    t0 = time.perf_counter()
    for k, at in enumerate(arrivals):
        while True:
            dt = at - (time.perf_counter() - t0)
            if dt <= 0:
                break
            time.sleep(min(dt, 2e-3) if dt > 2e-3 else 0)
        while True:
            try:
                tickets.append(srv.submit(pool[k % len(pool)]))
                break
            except cel.CelesteError as e:
                if getattr(e, "code", 0) != cel.EAGAIN:
                    raise
                time.sleep(1e-3)
    out = []
    for t in tickets:
        r = None
        while r is None:
            r = srv.poll(t, wait_ms=200)
        if r["code"] != 0:
            raise RuntimeError(f"request failed with code {r['code']}")
        out.append(r)
    wall = time.perf_counter() - t0
    return out, wall


def differentiation_summary(cel, dev, local, reps=10):
    """Config 4: the autograd function over the hand-written adjoint on 1,024
    sources of the field generator (all in one plan): value + gradient via
    backward, and Hessian-vector products via double backward, event-timed."""
    import torch
    from paper_1803_00113_gb300.autograd import SourceObjective
    p = fields.single_field(seed=SEED + 4, n_sources=1024)
    ctx = cel.Context(p.model, device=local)
    dp = cel.DeviceProblem(p, dev)
    plan = cel.Plan(ctx, dp, list(range(p.n_sources)))
    obj = SourceObjective(plan)
    theta0 = torch.tensor(p.theta, dtype=torch.float64, device=dev)
    v = torch.ones_like(theta0)

    def grad_once():
        t = theta0.clone().requires_grad_(True)
        obj(t).sum().backward()
        return t.grad

    def hvp_once():
        return torch.autograd.functional.hvp(lambda t: obj(t).sum(), theta0, v)[1]

    out = {"workload": "1,024 sources of the single-field generator, one plan, neighbours "
                       "frozen; patch-level recomputation (nothing stored per pixel)",
           "visits_per_evaluation": plan.visits}
    for name, fn in (("value_and_gradient", grad_once), ("hessian_vector_product", hvp_once)):
        fn()
        torch.cuda.synchronize(dev)
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(reps):
            fn()
        b.record()
        torch.cuda.synchronize(dev)
        ms = a.elapsed_time(b) / reps
        out[name] = {"ms": ms, "visits_per_s": plan.visits / (ms / 1e3)}
    plan.close()
    ctx.close()
    return out


def serving_summary(cel, args, local, rates=(200.0, 2000.0), seconds=2.0):
    """A short serving run beside the headline: region requests at Poisson
    arrival rates of 200 and 2,000 requests/s for `seconds` each; per rate the
    fit latency (submit -> result ready) percentiles and the throughput."""
    reqs = [fields.region_request(SEED + 5 + k) for k in range(args.pool)]
    pool = [cel.Server.prepare(q) for q in reqs]
    rng = np.random.default_rng(SEED + 5)
    srv = cel.Server(reqs[0].model, device=local, workers=args.workers,
                     pixels_per_item=args.serve_tile)
    t0 = time.perf_counter()
    _serve_run(cel, srv, pool[:8], np.zeros(8))          # warm-up: graphs, buffers
    per_rate = {}
    for rate in rates:
        n = max(int(rate * seconds), 20)
        res, wall = _serve_run(cel, srv, pool, np.cumsum(rng.exponential(1.0 / rate, n)))
        lat = np.array([r["latency_s"] for r in res]) * 1e3
        per_rate[str(int(rate))] = {
            "requests": n, "fit_latency_ms_p50": float(np.percentile(lat, 50)),
            "fit_latency_ms_p99": float(np.percentile(lat, 99)), "fits_per_s": n / wall,
            "mean_batch": float(np.mean([r["batch_requests"] for r in res]))}
    srv.close()
    return {"workload": "region requests: 1..64 sources, 32..512 px, 5 bands, 1..4 images per "
                        f"band, Poisson arrivals for {seconds:g} s per rate, fits of <= 5 passes "
                        "x <= 50 Newton iterations",
            "rates": per_rate, "seconds": time.perf_counter() - t0}


def run_serving(args):
    import torch
    world, rank, local = dist_info()
    if rank != 0:
        return None
    torch.cuda.set_device(local)
    from paper_1803_00113_gb300 import build_lib
    build_lib.build()
    from paper_1803_00113_gb300 import celeste as cel
    reqs = [fields.region_request(SEED + 5 + k) for k in range(args.pool)]
    pool = [cel.Server.prepare(q) for q in reqs]
    model = reqs[0].model
    mean_in = float(np.mean([q.bytes_in for q in pool]))
    mean_out = float(np.mean([q.n_sources * (27 * 8 + 4) for q in reqs]))
    rng = np.random.default_rng(SEED + 5)
    rates = [float(r) for r in args.rates.split(",")]

    def arrivals(rate, n):
        return np.cumsum(rng.exponential(1.0 / rate, n))

    srv = cel.Server(model, device=local, workers=args.workers, pixels_per_item=args.serve_tile)
    _serve_run(cel, srv, pool[:8], np.zeros(8))          # warm-up: graphs, buffers
    clocks = ClockSampler(local)
    clocks.start()
    per_rate = {}
    for rate in rates:
        n = max(int(rate * args.serve_seconds), 20)
        res, wall = _serve_run(cel, srv, pool, arrivals(rate, n))
        lat = np.array([r["latency_s"] for r in res]) * 1e3
        per_rate[str(int(rate))] = {
            "requests": n, "p50_ms": float(np.percentile(lat, 50)),
            "p99_ms": float(np.percentile(lat, 99)), "throughput": n / wall,
            "mean_batch": float(np.mean([r["batch_requests"] for r in res])),
            "mean_passes": float(np.mean([r["passes"] for r in res]))}
    clk = clocks.stop()
    st = srv.stats()
    srv.close()
    # the plain form: one request at a time, each its own fit, saturated
    plain_srv = cel.Server(model, device=local, workers=1, max_batch=1,
                           pixels_per_item=args.serve_tile)
    _serve_run(cel, plain_srv, pool[:4], np.zeros(4))
    n_plain = min(len(pool), 48)
    res, wall = _serve_run(cel, plain_srv, pool[:n_plain], np.zeros(n_plain))
    plain_srv.close()
    plain = {"throughput": n_plain / wall,
             "p50_ms_saturated": float(np.percentile([r["latency_s"] * 1e3 for r in res], 50)),
             "form": "one request per fit, one request in flight (saturated queue)"}
    best = max(per_rate.values(), key=lambda d: d["throughput"])
    top = per_rate[str(int(rates[-1]))]
    return {"metric": "region fits/s (Poisson arrivals, result back on the host)",
            "value": best["throughput"], "unit": "fits/s", "n_gpus": 1,
            "steps": len(rates), "warmup": 1, "ms_per_step": top["p50_ms"],
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f32",
            "data": "synthetic (seeded region requests: 1..64 sources, 32..512 px, 5 bands, "
                    "1..4 images per band)",
            "config": {"workload": "serving: Poisson arrivals at "
                                   f"{args.rates} requests/s, {args.serve_seconds:g} s each, "
                                   f"fits of <= 5 passes x <= 50 Newton iterations",
                       "pool": args.pool, "workers": args.workers or 2,
                       "pixels_per_tile": args.serve_tile,
                       "l2": "inputs stream in per request (not reused)"},
            "latency": per_rate,
            "plain_per_request": plain, "vs_plain": best["throughput"] / plain["throughput"],
            "e2e": {"value": best["throughput"], "unit": "fits/s",
                    "h2d_bytes_per_step": int(mean_in), "d2h_bytes_per_step": int(mean_out)},
            "gpu_launches": int(st["launches"]), "clocks": clk}


# ---------------------------------------------------------------------------
# Newton trust region vs a first-order subsolver (the paper's claim)
# ---------------------------------------------------------------------------

def run_first_order(args):
    """Both subsolvers on the same per-source problems: the largest colour
    class of the field, neighbours frozen at their start values.  Newton
    runs until every source stops; L-BFGS (m = 10, Armijo backtracking) runs
    until every source is within 1e-6 (1 + |L|) of the Newton optimum, or
    until it stops, or for at most --fo-max-steps steps."""
    import torch
    world, rank, local = dist_info()
    if rank != 0:
        return None
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    from paper_1803_00113_gb300 import build_lib
    build_lib.build()
    from paper_1803_00113_gb300 import celeste as cel
    problem, cfg = workload("field", args.sources, SEED + 1)
    ctx = cel.Context(problem.model, device=local)
    dp = cel.DeviceProblem(problem, dev)
    cls = max(cel.color_classes(problem), key=len)
    plan = cel.Plan(ctx, dp, cls)
    srcs = torch.as_tensor(plan.sources, dtype=torch.long, device=dev)

    def timed(fn):
        torch.cuda.synchronize(dev)
        t0 = time.perf_counter()
        out = fn()
        torch.cuda.synchronize(dev)
        return out, time.perf_counter() - t0

    # Newton: iterations per source until it stops
    step_ms = []

    def newton():
        delta, status = cel.newton_state(dp)
        its = torch.zeros(plan.n, dtype=torch.int32, device=dev)
        for k in range(50):
            live = (status[srcs] != cel.ST_CONVERGED) & (status[srcs] != cel.ST_FAILED)
            its += live.int()
            if not bool(live.any()):
                break
            t0 = time.perf_counter()
            cel.newton_step(plan, delta, status)
            torch.cuda.synchronize(dev)
            step_ms.append((time.perf_counter() - t0) * 1e3)
        return its
    newton()                                              # warm-up (kernels, torch ops)
    step_ms.clear()
    dp.set_theta(problem.theta)
    n_its, t_newton = timed(newton)
    best = cel.elbo(plan)[1].clone()
    dp.set_theta(problem.theta)
    lb = cel.Lbfgs(plan, m=10)
    target = best - 1e-6 * (1 + best.abs())

    def first_order():
        status = torch.zeros(problem.n_sources, dtype=torch.int32, device=dev)
        steps = 0
        for steps in range(1, args.fo_max_steps + 1):
            lb.step(status, target)
            if steps % 50 == 0:
                reached = lb.counts()[2]
                done = (reached > 0) | (status[srcs] == cel.ST_CONVERGED)
                if bool(done.all()):
                    break
        return steps
    lb.step(torch.zeros(problem.n_sources, dtype=torch.int32, device=dev), target)   # warm-up
    lb.counts()
    dp.set_theta(problem.theta)
    lb.reset()
    steps, t_fo = timed(first_order)
    iters, fevals, reached = [t.cpu().numpy() for t in lb.counts()]
    n_its = n_its.cpu().numpy()
    ok = reached > 0
    q = lambda a, f: float(np.percentile(a, f)) if len(a) else None
    return {"metric": "time to the Newton optimum, L-BFGS over Newton trust region",
            "value": t_fo / t_newton, "unit": "x", "n_gpus": 1, "steps": 1, "warmup": 1,
            "ms_per_step": t_newton * 1e3, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "f32 pixels, f64 subsolvers",
            "data": "synthetic (seeded field shaped like the paper's study set)",
            "config": dict(cfg, workload="first-order comparison on the largest colour class "
                                         f"of the field ({plan.n} sources)"),
            "newton": {"seconds": t_newton, "step_ms": [round(x, 3) for x in step_ms],
                       "iterations_p50": q(n_its, 50),
                       "iterations_p90": q(n_its, 90), "iterations_max": int(n_its.max())},
            "lbfgs": {"seconds": t_fo, "steps": int(steps), "reached_fraction": float(ok.mean()),
                      "gradient_evals_to_target_p50": q(reached[ok], 50),
                      "gradient_evals_to_target_p90": q(reached[ok], 90),
                      "gradient_evals_to_target_max": int(reached[ok].max()) if ok.any() else None,
                      "trial_evals_total_p50": q(fevals, 50), "history": 10},
            "e2e": None, "gpu_launches": int(ctx.launches())}


# ---------------------------------------------------------------------------
# the MCMC consumer: AIS + slice sampling per source (the paper's settings)
# ---------------------------------------------------------------------------

def run_mcmc(args):
    """AIS (T = 200, N' = 25 per type) and B' = 25 slice-sampling sweeps for
    the brightest sources of the field, neighbours fixed: all sources'
    chains in lock step, every sampler round one batched log-likelihood
    call; the plain form runs one source at a time."""
    import torch
    world, rank, local = dist_info()
    if rank != 0:
        return None
    torch.cuda.set_device(local)
    from paper_1803_00113_gb300 import build_lib
    build_lib.build()
    from paper_1803_00113_gb300 import mcmc
    problem, cfg = workload("field", args.sources, SEED + 1)
    bright = [int(s) for s in np.argsort(-problem.truth["logr"])[:args.mcmc_sources]]
    mcmc.type_posteriors(problem, bright[:1], n_chains=4, T=2, B=1)     # warm-up
    # one at a time (the plain form) and all together (chains batched)
    t0 = time.perf_counter()
    single_calls = 0
    for s in bright[:2]:
        single_calls += mcmc.type_posterior(problem, s, n_chains=25, T=200, B=25, seed=s)["calls"]
    single_s = (time.perf_counter() - t0) / 2
    t0 = time.perf_counter()
    res, calls = mcmc.type_posteriors(problem, bright, n_chains=25, T=200, B=25, seed=1)
    total = time.perf_counter() - t0
    visits = calls * 50 * problem.visits(bright)
    correct = sum(int((r["p_star"] > 0.5) == bool(problem.truth["is_star"][r["source"]]))
                  for r in res)
    per = bright
    return {"metric": "source posteriors/s (AIS T=200 x 25 chains per type + 25 sweeps)",
            "value": len(per) / total, "unit": "sources/s", "n_gpus": 1, "steps": 1,
            "warmup": 1, "ms_per_step": 1e3 * total, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f32 pixels, f64 sums",
            "data": "synthetic (seeded field shaped like the paper's study set)",
            "config": dict(cfg, workload=f"MCMC (AIS + slice sampling) of the {len(per)} brightest "
                                         "field sources, neighbours fixed"),
            "loglik_calls_per_s": calls / total, "visits_per_s": visits / total,
            "sources_batched": len(per), "type_correct": correct,
            "plain_one_source_at_a_time": {"seconds_per_source": single_s,
                                            "loglik_calls": single_calls},
            "vs_plain": single_s / (total / len(per)),
            "e2e": None, "gpu_launches": None}


def main(argv=None):
    args = parse_args(argv)
    if args.impl == "reference":
        line = run_reference(args)
    elif args.workload == "mcmc":
        line = run_mcmc(args)
    elif args.workload == "first-order":
        line = run_first_order(args)
    elif args.workload == "serving":
        line = run_serving(args)
    else:
        line = run_ours(args)
    if line is not None:
        print(json.dumps(line), flush=True)
    world = dist_info()[0]
    if world > 1:
        import torch.distributed as dist
        if dist.is_initialized():
            dist.destroy_process_group()


if __name__ == "__main__":
    main()
