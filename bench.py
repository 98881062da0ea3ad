#!/usr/bin/env python3
"""Benchmark of BMMC permutations on GB300: effective bandwidth 2*N*e / time.

Default workload (one "step"): arrays of 2^28 elements at 4, 8 and 16 bytes
per element, and for each element size the permutation set
    bit reversal, half swap (2^14 x 2^14 transpose), 16 random bit
    permutations, 16 random tiled-only BMMCs, 64 random dense BMMCs
(dense BMMCs with a random complement c).  Each permutation runs once per
step through the library's C ABI on device-resident buffers; every array is
larger than L2, so no flush is needed between steps.

Reported beside the headline number: per-class bandwidth, a same-run
cudaMemcpyAsync device-to-device copy of the same bytes, the dominant
kernel's roofline against the measured HBM peak, the end-to-end figure with
host buffers, the SM clocks sampled during the timed region, and the CPU
oracle timed on a bounded sample (baseline only).

    python bench.py [--gpus N] [--steps K] [--warmup W] [--impl reference]

With N > 1 the script runs under torchrun, one process per GPU, each GPU
running the full per-GPU workload (independent arrays: replicas, weak
scaling); the value is the total bytes of all ranks over the slowest rank.
"""

import argparse
import hashlib
import json
import os
import statistics
import subprocess
import sys
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = ("effective GB/s (2·N·bytes/s) vs GB300 HBM peak & D2D copy; "
          "batched/served p50/p99")
FALLBACK_HBM_GBS = 6800.0
# The path copies elements as opaque 4-, 8- and 16-byte blobs.
DTYPE = "opaque 4/8/16-byte elements"
PROFILE_TRAFFIC = os.path.join(ROOT, "profiles", "bmmc_tiled_pass_traffic.md")
KERNEL_SOURCES = [os.path.join(ROOT, "paper_2306_07795_gb300", "csrc", f)
                  for f in ("kernels.cu", "tile_body.cuh", "pass_desc.h", "plan.cpp")]


def parse_args():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=5)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", choices=["ours", "reference"], default="ours")
    ap.add_argument("--n", type=int, default=28)
    ap.add_argument("--elem", type=str, default="4,8,16")
    ap.add_argument("--dense", type=int, default=64)
    ap.add_argument("--bp", type=int, default=16)
    ap.add_argument("--tiled", type=int, default=16)
    ap.add_argument("--strategy", choices=["paper", "single"], default="paper")
    ap.add_argument("--cta-tile", type=int, default=0,
                    help="log2 bytes per thread block of the headline plans (0 = default)")
    ap.add_argument("--load", choices=["cp", "tma"], default="cp",
                    help="tile loads of the headline plans: 16-byte cp.async copies or "
                         "tensor copies (BMMC_PLAN_TMA_LOAD)")
    ap.add_argument("--e2e-steps", type=int, default=2)
    ap.add_argument("--no-e2e", action="store_true")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-extras", action="store_true")
    ap.add_argument("--no-batched", action="store_true")
    ap.add_argument("--no-serving", action="store_true")
    ap.add_argument("--no-autograd", action="store_true")
    ap.add_argument("--serving-seconds", type=float, default=10.0)
    ap.add_argument("--batched-count", type=int, default=4096,
                    help="arrays in the batched workload (4096 in the configuration)")
    ap.add_argument("--no-small", action="store_true",
                    help="skip the n=20 configuration and the sorting network")
    return ap.parse_args()


# ---------------------------------------------------------------------------
# Distributed setup (replicas; no collective on the data path)
# ---------------------------------------------------------------------------

def dist_setup():
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return world, rank, local


def dist_init(world, local):
    import torch
    torch.cuda.set_device(local)
    if world > 1:
        import torch.distributed as dist
        os.environ.setdefault("MASTER_ADDR", "127.0.0.1")
        dist.init_process_group("nccl", device_id=torch.device("cuda", local))


def barrier(world):
    if world > 1:
        import torch.distributed as dist
        dist.barrier()


def _reduce_device():
    import torch.distributed as dist
    return "cuda" if dist.get_backend() == "nccl" else "cpu"


def allreduce_max(world, value):
    """Max over ranks (the slowest rank's time)."""
    if world == 1:
        return value
    import torch
    import torch.distributed as dist
    t = torch.tensor([value], dtype=torch.float64, device=_reduce_device())
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def allreduce_sum(world, value):
    """Sum over ranks (the bytes all replicas moved)."""
    if world == 1:
        return value
    import torch
    import torch.distributed as dist
    t = torch.tensor([value], dtype=torch.float64, device=_reduce_device())
    dist.all_reduce(t, op=dist.ReduceOp.SUM)
    return float(t.item())


# ---------------------------------------------------------------------------
# Workload
# ---------------------------------------------------------------------------

def lib_invertible(n):
    """Invertibility test for rejection sampling: the library's own
    validation (bmmc_plan_create returns BMMC_ERR_SINGULAR)."""
    import paper_2306_07795_gb300 as bm

    def test(rows):
        try:
            h = bm.bmmc_plan_create(n, rows, 0, 4)
        except bm.BmmcError as err:
            if err.code == bm.BMMC_ERR_SINGULAR:
                return False
            raise
        bm.bmmc_plan_destroy(h)
        return True
    return test


def workload(n, elems, n_bp, n_tiled, n_dense, seed_base=0):
    """List of (class, e, rows, c) for one step."""
    import workloads as wl
    inv = lib_invertible(n)
    out = []
    for e in elems:
        k = 8 - {4: 2, 8: 3, 16: 4}[e]
        out.append(("bit_reverse", e, wl.bit_reverse(n), 0))
        out.append(("half_swap", e, wl.half_swap(n), 0))
        for s in range(n_bp):
            out.append(("bp", e, wl.random_bp(n, seed_base + 1 + s), 0))
        for s in range(n_tiled):
            rows, c = wl.tiled_only_bmmc(n, k, seed_base + 1 + s, inv)
            out.append(("tiled_only", e, rows, c))
        for s in range(n_dense):
            rows, c = wl.dense_bmmc(n, seed_base + 1 + s, inv)
            out.append(("dense", e, rows, c))
    return out


# ---------------------------------------------------------------------------
# Clock sampling during the timed region
# ---------------------------------------------------------------------------

CLOCK_QUERY = ("index,clocks.sm,clocks.max.sm,power.draw,"
               "clocks_event_reasons.active,clocks_event_reasons.hw_slowdown,"
               "clocks_event_reasons.hw_thermal_slowdown,"
               "clocks_event_reasons.sw_thermal_slowdown,"
               "clocks_event_reasons.sw_power_cap")


def clock_sampler_start(device_index):
    import torch
    sel = []
    try:
        uuid = str(torch.cuda.get_device_properties(device_index).uuid)
        if uuid:
            sel = ["-i", uuid if uuid.startswith("GPU-") else "GPU-" + uuid]
    except Exception:
        sel = []
    try:
        return subprocess.Popen(
            ["nvidia-smi", "--query-gpu=" + CLOCK_QUERY,
             "--format=csv,noheader,nounits", "-lms", "200"] + sel,
            stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
    except (OSError, FileNotFoundError):
        return None


def clock_sampler_stop(proc):
    if proc is None:
        return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["unavailable"]}
    time.sleep(0.25)
    proc.terminate()
    try:
        out, _ = proc.communicate(timeout=5)
    except subprocess.TimeoutExpired:
        proc.kill()
        out, _ = proc.communicate()
    sm, smax, power = [], [], []
    flags = {"hw_slowdown": 0, "hw_thermal_slowdown": 0,
             "sw_thermal_slowdown": 0, "sw_power_cap": 0}
    names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown",
             "sw_power_cap"]
    for line in out.splitlines():
        parts = [p.strip() for p in line.split(",")]
        if len(parts) < 9:
            continue
        try:
            sm.append(float(parts[1]))
            smax.append(float(parts[2]))
            power.append(float(parts[3]))
        except ValueError:
            continue
        for nm, val in zip(names, parts[5:9]):
            if val.lower().startswith("active"):
                flags[nm] += 1
    reasons = [nm for nm in names if flags[nm]]
    return {"sm_mhz": statistics.median(sm) if sm else None,
            "sm_max_mhz": max(smax) if smax else None,
            "power_w_max": max(power) if power else None,
            "samples": len(sm), "reasons": reasons}


# ---------------------------------------------------------------------------
# Roofline helpers
# ---------------------------------------------------------------------------

def measured_hbm_peak():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    try:
        with open(path) as f:
            peaks = json.load(f)
        return float(peaks["hbm_gbs"]), "measured"
    except (OSError, KeyError, ValueError):
        return FALLBACK_HBM_GBS, "fallback"


def kernel_source_sha():
    h = hashlib.sha256()
    for p in KERNEL_SOURCES:
        with open(p, "rb") as f:
            h.update(f.read())
    return h.hexdigest()[:16]


def profiled_traffic(kernel_name):
    """DRAM bytes per launch from the committed ncu summary, if it was taken
    on the current kernel sources for this kernel; else None."""
    try:
        with open(PROFILE_TRAFFIC) as f:
            text = f.read()
    except OSError:
        return None, None
    fields = {}
    for line in text.splitlines():
        if ":" in line and line.startswith("- "):
            key, val = line[2:].split(":", 1)
            fields[key.strip()] = val.strip().strip("`")
    if fields.get("source_sha") != kernel_source_sha():
        return None, "stale"
    if fields.get("kernel") != kernel_name:
        return None, "other kernel"
    try:
        return float(fields["dram_bytes_per_launch"]), fields.get("workload")
    except (KeyError, ValueError):
        return None, None


# What the strategies run: with the default segments every matrix is one launch.
STRATEGY = {"paper": "paper, two-pass plans as one launch", "single": "single"}


def workload_config(args, world):
    """The `config` object of both arms' JSON lines (the same workload)."""
    elems = [int(v) for v in args.elem.split(",")]
    N = 1 << args.n
    count = len(elems) * (2 + args.bp + args.tiled + args.dense)
    return {
        "workload": "n=%d BMMC permutation set per elem size: bit-reversal, "
                    "half-swap, %d random BP, %d random tiled-only, %d random "
                    "dense (random c)" % (args.n, args.bp, args.tiled, args.dense),
        "n": args.n, "elem_bytes": elems, "strategy": STRATEGY[args.strategy],
        "tile_load": "tensor copies (TMA)" if args.load == "tma" else "16-byte cp.async",
        "permutations_per_step": count,
        "l2": "inputs larger than L2 (%d-%d MiB per array), no flush"
              % (N * min(elems) >> 20, N * max(elems) >> 20),
        "parallelism": "replicas" if world > 1 else "single GPU"}


# ---------------------------------------------------------------------------
# CPU baseline / reference arm: the oracle on the host cores
# ---------------------------------------------------------------------------

# Array size (log2 elements) of the oracle's timed sample.
ORACLE_N = 28


def oracle_sample(n, n_dense=4):
    """The CPU-baseline sample of the n = 28 configuration at 4-byte
    elements: bit-reversal, half-swap and the first n_dense dense random
    BMMCs of the benchmark's own set (seeds 1..n_dense, random c)."""
    import workloads as wl
    from oracle import f2
    inv = lambda rows: f2.is_invertible(rows, len(rows))  # noqa: E731
    items = [("bit_reverse", 4, wl.bit_reverse(n), 0),
             ("half_swap", 4, wl.half_swap(n), 0)]
    for sd in range(1, n_dense + 1):
        rows, c = wl.dense_bmmc(n, sd, inv)
        items.append(("dense", 4, rows, c))
    return items


def run_oracle_step(n, items, inp, out, threads=True):
    """Run every permutation of `items` once through the oracle's C loop
    (into the preallocated `out`); returns the effective bytes 2 N e."""
    import oracle
    moved = 0
    for cls, e, rows, c in items:
        oracle.apply_into(n, rows, c, inp, out, elem_bytes=e, threads=threads)
        moved += 2 * (1 << n) * e
    return moved


def oracle_sample_text():
    return ("the oracle's C loop out[A x + c] = in[x] (OpenMP over x) on the "
            "n = %d configuration at 4-byte elements (%d MiB arrays): "
            "bit-reversal, half-swap and dense random BMMCs seeds 1-4"
            % (ORACLE_N, (4 << ORACLE_N) >> 20))


def cpu_model():
    """The host CPU's model name (lscpu), or the platform's processor string."""
    try:
        out = subprocess.run(["lscpu"], capture_output=True, text=True, timeout=10).stdout
        for line in out.splitlines():
            if line.strip().lower().startswith("model name"):
                return line.split(":", 1)[1].strip()
    except (OSError, subprocess.SubprocessError):
        pass
    import platform
    return platform.processor() or platform.machine()


def cpu_baseline():
    """The oracle on the host cores: all cores on the n = 28 sample, one
    core on part of it, and the n = 20 configuration in full."""
    import numpy as np
    import oracle
    import workloads as wl
    n = ORACLE_N
    items = oracle_sample(n)
    inp = wl.payload(n, 4)
    out = np.empty_like(inp)
    run_oracle_step(n, items[:1], inp, out)  # first touch of both arrays
    t0 = time.perf_counter()
    moved = run_oracle_step(n, items, inp, out)
    dt = time.perf_counter() - t0
    res = {"value": round(moved / dt / 1e9, 3), "unit": "GB/s",
           "cores": oracle.num_threads(), "kind": "oracle",
           "sample": "%s, all cores, %.1f s" % (oracle_sample_text(), dt),
           "cpu_model": cpu_model(), "nproc": os.cpu_count()}
    one = items[:1] + items[2:3]
    t0 = time.perf_counter()
    moved = run_oracle_step(n, one, inp, out, threads=False)
    dt = time.perf_counter() - t0
    res["single_thread"] = {"value": round(moved / dt / 1e9, 3), "unit": "GB/s", "cores": 1,
                            "sample": "bit-reversal and dense seed 1 of the same sample "
                                      "on one core, %.1f s" % dt}
    del inp, out
    # the n = 20 configuration in full: int32 iota, bit-reversal + 16 dense
    from oracle import f2
    inv = lambda rows: f2.is_invertible(rows, len(rows))  # noqa: E731
    c1 = [("bit_reverse", 4, wl.bit_reverse(20), 0)] + \
        [("dense", 4) + tuple(wl.dense_bmmc(20, sd, inv)) for sd in range(1, 17)]
    iota = np.arange(1 << 20, dtype=np.uint32)
    out20 = np.empty_like(iota)
    for threads, key in ((True, "n20_config"), (False, "n20_config_single_thread")):
        t0 = time.perf_counter()
        moved = run_oracle_step(20, c1, iota, out20, threads=threads)
        res[key] = {"value": round(moved / (time.perf_counter() - t0) / 1e9, 3),
                    "unit": "GB/s", "cores": oracle.num_threads() if threads else 1,
                    "sample": "all 17 permutations of the n = 20 configuration"}
    return res


def reference_arm(args):
    """The oracle, as it stands, on the host cores: each step runs the
    n = 28 sample once on all cores (rank 0 only)."""
    world, rank, local = dist_setup()
    if rank != 0:
        return 0
    import numpy as np
    import oracle
    import workloads as wl
    n = ORACLE_N
    items = oracle_sample(n)
    inp = wl.payload(n, 4)
    out = np.empty_like(inp)
    for _ in range(args.warmup):
        run_oracle_step(n, items, inp, out)
    t0 = time.perf_counter()
    moved = 0
    for _ in range(args.steps):
        moved += run_oracle_step(n, items, inp, out)
    dt = time.perf_counter() - t0
    value = moved / dt / 1e9
    sample = "%s, all cores, per step" % oracle_sample_text()
    line = {
        "impl": "reference", "metric": METRIC, "value": value, "unit": "GB/s",
        "n_gpus": args.gpus, "steps": args.steps, "warmup": args.warmup,
        "ms_per_step": dt * 1e3 / max(1, args.steps), "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": DTYPE,
        "data": "synthetic",
        "config": workload_config(args, args.gpus),
        "cpu_baseline": {"value": value, "unit": "GB/s",
                         "cores": oracle.num_threads(), "kind": "oracle",
                         "sample": sample, "cpu_model": cpu_model(),
                         "nproc": os.cpu_count()},
        "e2e": {"value": value, "unit": "GB/s", "h2d_bytes_per_step": 0,
                "d2h_bytes_per_step": 0},
    }
    print(json.dumps(line))
    return 0


# ---------------------------------------------------------------------------
# Batched, differentiable and served forms (reported beside the headline)
# ---------------------------------------------------------------------------

def _percentile(values, q):
    v = sorted(values)
    k = (len(v) - 1) * q
    lo = int(k)
    hi = min(lo + 1, len(v) - 1)
    return v[lo] + (v[hi] - v[lo]) * (k - lo)


def bench_batched(dev, stream, count=4096, seed=7, replays=20, warmup=3):
    """4096 int32 arrays, n uniform in 10..24, each with its own dense BMMC:
    one batch (persistent launches, tile options chosen by the autotuner)
    captured in a CUDA graph, against one plain launch per array."""
    import torch
    import paper_2306_07795_gb300 as bm
    from paper_2306_07795_gb300.autotune import tune_batch
    from paper_2306_07795_gb300.batch import Batch
    import workloads as wl

    ns = wl.batched_sizes(count=count, lo=10, hi=24, seed=seed)
    mats = [wl.dense_bmmc(n, seed * 100003 + i, lib_invertible(n)) for i, n in enumerate(ns)]
    sizes = [(1 << n) * 4 for n in ns]
    offs, total = [], 0
    for s in sizes:
        offs.append(total)
        total += (s + 255) // 256 * 256
    gen = torch.Generator(device=dev).manual_seed(seed)
    xin = torch.randint(-2**31, 2**31 - 1, (total // 4,), dtype=torch.int32, device=dev,
                        generator=gen)
    xout = torch.empty_like(xin)
    ins = [xin[o // 4:(o + s) // 4] for o, s in zip(offs, sizes)]
    outs = [xout[o // 4:(o + s) // 4] for o, s in zip(offs, sizes)]
    moved = sum(2 * s for s in sizes)

    def plans_for(flags, seg, tile):
        return [bm.Plan(n, rows, c, 4, flags=flags, seg_bits=seg, cta_tile_log2=tile)
                for n, (rows, c) in zip(ns, mats)]

    def time_graph(batch):
        graph = batch.capture()
        for _ in range(warmup):
            graph.replay()
        evs = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True))
               for _ in range(replays)]
        s = torch.cuda.current_stream(dev)
        for a, b in evs:
            a.record(s)
            graph.replay()
            b.record(s)
        torch.cuda.synchronize(dev)
        ms = [a.elapsed_time(b) for a, b in evs]
        del graph
        return ms

    out = {"arrays": count, "elem_bytes": 4, "bytes_moved_per_replay": moved,
           "n_range": [10, 24]}
    # autotuner: tile options for the whole batch, paper strategy
    best, trials = tune_batch(lambda seg, tile: Batch(plans_for(bm.BMMC_PLAN_PAPER, seg, tile),
                                                      ins, outs), dev)
    out["autotune"] = {"chosen": {"seg_bits": best[0], "cta_tile_log2": best[1]},
                       "trials": trials}
    plans = plans_for(bm.BMMC_PLAN_PAPER, *best)
    batch = Batch(plans, ins, outs)
    ms = time_graph(batch)
    med = statistics.median(ms)
    out["graph"] = {"launches_per_replay": batch.num_launches,
                    "gbs": round(moved / (med / 1e3) / 1e9, 1),
                    "replay_ms_p50": round(_percentile(ms, 0.5), 3),
                    "replay_ms_p99": round(_percentile(ms, 0.99), 3)}
    ws_need = batch.workspace.numel() if batch.workspace is not None else 0
    del batch
    # plain: one bmmc_execute per array, in order, on one stream
    ws = torch.empty(max(p.workspace_bytes for p in plans) or 16, dtype=torch.uint8,
                     device=dev)
    for p, x, y in zip(plans, ins, outs):
        p(x, out=y, stream=stream, workspace=ws)
    plain_ms = []
    for _ in range(3):
        a = torch.cuda.Event(enable_timing=True)
        b = torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize(dev)
        a.record(stream)
        for p, x, y in zip(plans, ins, outs):
            p(x, out=y, stream=stream, workspace=ws)
        b.record(stream)
        torch.cuda.synchronize(dev)
        plain_ms.append(a.elapsed_time(b))
    pm = statistics.median(plain_ms)
    out["plain_launches"] = {"launches": sum(p.num_launches for p in plans),
                             "gbs": round(moved / (pm / 1e3) / 1e9, 1),
                             "ms": round(pm, 3)}
    out["speedup_vs_plain"] = round(pm / med, 3)
    out["workspace_bytes"] = ws_need
    del ws
    # single-pass strategy (beyond the paper): one launch, no workspace
    sp = Batch(plans_for(bm.BMMC_PLAN_SINGLE_PASS, *best), ins, outs)
    ms = time_graph(sp)
    med1 = statistics.median(ms)
    out["graph_single_pass"] = {"launches_per_replay": sp.num_launches,
                                "gbs": round(moved / (med1 / 1e3) / 1e9, 1),
                                "replay_ms_p50": round(_percentile(ms, 0.5), 3),
                                "replay_ms_p99": round(_percentile(ms, 0.99), 3)}
    del sp, xin, xout, ins, outs
    torch.cuda.empty_cache()
    return out


def bench_autograd(dev, iters=20):
    """[64, 2^20] fp32 through the differentiable permutation: forward and
    backward (the inverse BMMC) per iteration, against a D2D copy."""
    import torch
    import paper_2306_07795_gb300 as bm
    from paper_2306_07795_gb300.autograd import bmmc_permute
    import workloads as wl

    n = 20
    rows, c = wl.dense_bmmc(n, 3, lib_invertible(n))
    out = {"shape": [64, 1 << n], "dtype": "float32"}
    gen = torch.Generator(device=dev).manual_seed(3)
    x = torch.randn(64, 1 << n, device=dev, generator=gen).requires_grad_(True)
    w = torch.randn(64, 1 << n, device=dev, generator=gen)
    nbytes = x.numel() * 4
    for name, flags in (("paper", bm.BMMC_PLAN_PAPER), ("single_pass", bm.BMMC_PLAN_SINGLE_PASS)):
        plan = bm.Plan(n, rows, c, 4, flags=flags)
        for _ in range(3):
            x.grad = None
            bmmc_permute(x, plan).backward(w)
        s = torch.cuda.current_stream(dev)
        a = torch.cuda.Event(enable_timing=True)
        b = torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize(dev)
        a.record(s)
        for _ in range(iters):
            x.grad = None
            bmmc_permute(x, plan).backward(w)
        b.record(s)
        torch.cuda.synchronize(dev)
        ms = a.elapsed_time(b) / iters
        out[name] = {"fwd_bwd_ms": round(ms, 4),
                     "gbs": round(2 * 2 * nbytes / (ms / 1e3) / 1e9, 1)}
        # the same step captured in a CUDA graph (no Python or autograd-engine
        # time between the launches)
        x.grad = None
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            bmmc_permute(x, plan).backward(w)
        gms = _time_ms(graph.replay, dev, iters)
        out[name]["graph_fwd_bwd_ms"] = round(gms, 4)
        out[name]["graph_gbs"] = round(2 * 2 * nbytes / (gms / 1e3) / 1e9, 1)
        del graph
        x.grad = None
    y = torch.empty_like(w)
    y.copy_(w)
    a = torch.cuda.Event(enable_timing=True)
    b = torch.cuda.Event(enable_timing=True)
    a.record()
    for _ in range(iters):
        y.copy_(w)
    b.record()
    torch.cuda.synchronize(dev)
    d2d = a.elapsed_time(b) / iters
    out["two_d2d_copies_ms"] = round(2 * d2d, 4)
    for name in ("paper", "single_pass"):
        out[name]["frac_of_2x_d2d"] = round(2 * d2d / out[name]["fwd_bwd_ms"], 4)
        out[name]["graph_frac_of_2x_d2d"] = round(2 * d2d / out[name]["graph_fwd_bwd_ms"], 4)
    return out


def _time_ms(fn, dev, reps, warmup=3):
    import torch
    s = torch.cuda.current_stream(dev)
    for _ in range(warmup):
        fn()
    a = torch.cuda.Event(enable_timing=True)
    b = torch.cuda.Event(enable_timing=True)
    torch.cuda.synchronize(dev)
    a.record(s)
    for _ in range(reps):
        fn()
    b.record(s)
    torch.cuda.synchronize(dev)
    return a.elapsed_time(b) / reps


def bench_n20(dev, reps=50):
    """The n = 20 configuration (int32 iota; bit-reversal and 16 dense BMMCs,
    seeds 1..16): 4 MiB arrays, resident in L2 between launches, so this is
    an L2 figure, not an HBM one."""
    import torch
    import paper_2306_07795_gb300 as bm
    import workloads as wl
    n = 20
    mats = [(wl.bit_reverse(n), 0)] + [wl.dense_bmmc(n, s, lib_invertible(n))
                                       for s in range(1, 17)]
    x = torch.arange(1 << n, dtype=torch.int32, device=dev)
    y = torch.empty_like(x)
    ws = torch.empty((1 << n) * 4, dtype=torch.uint8, device=dev)
    out = {"permutations": len(mats), "bytes_per_permutation": 2 * (1 << n) * 4,
           "l2_resident": True}
    for name, flags in (("paper", bm.BMMC_PLAN_PAPER), ("single_pass", bm.BMMC_PLAN_SINGLE_PASS)):
        plans = [bm.Plan(n, rows, c, 4, flags=flags) for rows, c in mats]

        def run():
            for p in plans:
                p(x, out=y, workspace=ws)
        ms = _time_ms(run, dev, reps) / len(plans)
        run()
        torch.cuda.synchronize(dev)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            run()
        gms = _time_ms(graph.replay, dev, reps) / len(plans)
        out[name] = {"us_per_permutation": round(ms * 1e3, 2),
                     "gbs": round(2 * (1 << n) * 4 / (ms / 1e3) / 1e9, 1),
                     "graph_us_per_permutation": round(gms * 1e3, 2),
                     "graph_gbs": round(2 * (1 << n) * 4 / (gms / 1e3) / 1e9, 1),
                     "launches": sum(p.num_launches for p in plans)}
        del graph
    return out


def bench_sorting(dev):
    """The Sec. 6.1 sorting network on float32 keys: fused passes (many
    comparator stages per pass, include/bmmc_sort.h) and one
    permute-and-compare pass per stage, beside torch.sort of the same keys."""
    import torch
    from paper_2306_07795_gb300.sorting import SortingNetwork
    out = {}
    for n in (20, 24):
        x = torch.randn(1 << n, device=dev)
        want = torch.sort(x).values
        ref = _time_ms(lambda: torch.sort(x), dev, 5)
        res = {"stages": n * (n + 1) // 2, "torch_sort_ms": round(ref, 3)}
        for name, net in (("fused", SortingNetwork(n)),
                          ("stagewise", SortingNetwork(n, fused=False))):
            ms = _time_ms(lambda: net(x), dev, 5)
            graph, gout = net.capture(x)
            gms = _time_ms(graph.replay, dev, 10)
            passes = net.num_passes(torch.float32)
            res[name] = {"passes": passes, "ms": round(ms, 3), "graph_ms": round(gms, 3),
                         "pass_gbs": round(passes * 2 * x.numel() * 4 / (gms / 1e3) / 1e9, 1),
                         "vs_torch_sort": round(ref / gms, 3)}
            graph.replay()
            torch.cuda.synchronize(dev)
            assert torch.equal(gout, want)
            del graph, gout
        out["n%d" % n] = res
    return out


def bench_serving(dev, seconds=10.0, rate=2000.0, seed=11, budget=40 * 10**9, streams=4):
    """Poisson request stream; continuous-admission server vs a plain loop."""
    import torch
    from paper_2306_07795_gb300 import serving
    import workloads as wl

    specs = wl.serving_requests(rate=rate, seconds=seconds, seed=seed)
    mats = []
    for s in specs:
        if s["kind"] == "bp":
            mats.append((wl.random_bp(s["n"], s["seed"]), 0))
        else:
            mats.append(wl.dense_bmmc(s["n"], s["seed"], lib_invertible(s["n"])))
    gen = torch.Generator(device=dev).manual_seed(seed)
    pool = torch.randint(-2**31, 2**31 - 1, ((1 << 27) * 8 // 4,), dtype=torch.int32,
                         device=dev, generator=gen)

    # For the repeated-matrix extra: 4 matrices per (n, kind), reused.
    reuse = {}
    for s, m in zip(specs, mats):
        lst = reuse.setdefault((s["n"], s["kind"]), [])
        if len(lst) < 4:
            lst.append(m)

    def requests(speedup=1.0, limit_s=None, repeated=False):
        out = []
        for i, (s, (rows, c)) in enumerate(zip(specs, mats)):
            t = s["arrival"] / speedup
            if limit_s is not None and t >= limit_s:
                break
            if repeated:
                lst = reuse[(s["n"], s["kind"])]
                rows, c = lst[i % len(lst)]
            x = pool[: (1 << s["n"]) * s["e"] // 4]
            out.append(serving.Request(i, t, s["n"], s["e"], rows, c, x))
        return out

    def rounded(d):
        for f in ("throughput_req_s", "effective_gbs", "p50_ms", "p99_ms", "mean_ms",
                  "makespan_s", "submit_late_p99_ms"):
            d[f] = round(d[f], 4)
        return d

    def compare(flags, speedup=1.0, limit_s=None, repeated=False, large_log2=None):
        out = {}
        for mode, key in (("continuous", "server"), ("plain", "plain")):
            srv = serving.Server(dev, mode=mode, streams=streams, budget_bytes=budget,
                                 flags=flags, large_log2=large_log2 if mode != "plain" else 0)
            reqs = serving.drive(srv, requests(speedup, limit_s, repeated))
            out[key] = rounded(serving.summarize(reqs))
            out[key]["stats"] = srv.stats()
            srv.close()
            del srv, reqs
            torch.cuda.empty_cache()
        out["p99_ratio_plain_over_server"] = round(out["plain"]["p99_ms"]
                                                   / out["server"]["p99_ms"], 3)
        out["throughput_ratio_server_over_plain"] = round(
            out["server"]["throughput_req_s"] / out["plain"]["throughput_req_s"], 3)
        return out

    import paper_2306_07795_gb300 as bm
    res = {"requests": len(specs), "rate_per_s": rate, "seconds": seconds,
           "budget_bytes": budget, "streams": streams, "strategy": STRATEGY["paper"],
           "server_large_log2": 28}
    # The latency floor with no queueing: each request's HBM traffic (2 N e
    # per launch) at the measured peak; its 99th percentile bounds p99 from
    # below at a rate that never queues.
    peak, _ = measured_hbm_peak()
    ideal = []
    for s_, (rows, c) in zip(specs, mats):
        launches = bm.Plan(s_["n"], rows, c, s_["e"]).num_launches
        ideal.append(launches * 2 * (1 << s_["n"]) * s_["e"] / (peak * 1e9) * 1e3)
    res["ideal_service_ms"] = {"p50": round(_percentile(ideal, 0.5), 4),
                               "p99": round(_percentile(ideal, 0.99), 4),
                               "max": round(max(ideal), 4),
                               "peak_gbs": peak}
    res.update(compare(bm.BMMC_PLAN_PAPER))
    res["single_pass_plans"] = compare(bm.BMMC_PLAN_SINGLE_PASS)
    # Extra: the server without its high-priority stream for large requests
    res["extra_no_priority_stream"] = {"large_log2": 0}
    res["extra_no_priority_stream"].update(compare(bm.BMMC_PLAN_PAPER, large_log2=0))
    # Extra, beyond the configured 2000 requests/s: the same request mix with
    # arrival times compressed, 2 s per rate.
    res["extra_rate_sweep"] = []
    for fast in (2.0, 4.0, 6.0, 8.0, 10.0):
        row = {"rate_per_s": rate * fast}
        row.update(compare(bm.BMMC_PLAN_PAPER, speedup=fast, limit_s=2.0))
        res["extra_rate_sweep"].append(row)
    # Extra: the configured stream for 2 s, but with the matrices drawn from 4
    # per (n, kind), so that the server's plan cache hits (the plain loop
    # still plans every request).
    res["extra_repeated_matrices"] = {"rate_per_s": rate, "matrices_per_size_and_kind": 4}
    res["extra_repeated_matrices"].update(compare(bm.BMMC_PLAN_PAPER, limit_s=2.0,
                                                  repeated=True))
    del pool
    torch.cuda.empty_cache()
    return res


# ---------------------------------------------------------------------------
# Our arm
# ---------------------------------------------------------------------------

def main():
    args = parse_args()
    if args.impl == "reference":
        return reference_arm(args)
    import torch
    import paper_2306_07795_gb300 as bm

    world, rank, local = dist_setup()
    dist_init(world, local)
    dev = torch.device("cuda", local)
    stream = torch.cuda.current_stream(dev)
    elems = [int(v) for v in args.elem.split(",")]
    n = args.n
    N = 1 << n
    flags = bm.BMMC_PLAN_SINGLE_PASS if args.strategy == "single" else bm.BMMC_PLAN_PAPER
    if args.load == "tma":
        flags |= bm.BMMC_PLAN_TMA_LOAD

    # ---- plans and device buffers (outside the timed region) --------------
    import workloads as wl
    items = workload(n, elems, args.bp, args.tiled, args.dense, seed_base=1000 * rank)
    plans = [bm.Plan(n, rows, c, e, flags=flags, cta_tile_log2=args.cta_tile)
             for (_, e, rows, c) in items]
    bufs = {}
    for e in elems:
        x = wl.payload_torch(n, e, seed=rank, device=dev)
        y = torch.empty_like(x)
        ws = torch.empty(N * e, dtype=torch.uint8, device=dev)
        bufs[e] = (x, y, ws)
    torch.cuda.synchronize(dev)

    def run(i):
        cls, e, rows, c = items[i]
        x, y, ws = bufs[e]
        plans[i](x, out=y, stream=stream, workspace=ws)

    # ---- timed region ------------------------------------------------------
    K, W = args.steps, args.warmup
    per_item = [[torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)]
                for _ in range(len(items) * K)]
    t_start = torch.cuda.Event(enable_timing=True)
    t_end = torch.cuda.Event(enable_timing=True)
    # The clock sampler starts first; the warm-up steps then run right up to
    # the timed region, so its first launch does not meet an idle GPU.
    sampler = clock_sampler_start(local)
    time.sleep(0.3)
    for _ in range(W):
        for i in range(len(items)):
            run(i)
    torch.cuda.synchronize(dev)
    barrier(world)
    torch.cuda.synchronize(dev)
    wall0 = time.perf_counter()
    t_start.record(stream)
    for k in range(K):
        for i in range(len(items)):
            ev = per_item[k * len(items) + i]
            ev[0].record(stream)
            run(i)
            ev[1].record(stream)
    t_end.record(stream)
    torch.cuda.synchronize(dev)
    wall1 = time.perf_counter()
    clocks = clock_sampler_stop(sampler)
    barrier(world)
    elapsed_ms = t_start.elapsed_time(t_end)
    elapsed_ms = allreduce_max(world, elapsed_ms)

    bytes_per_step = sum(2 * N * e for (_, e, _, _) in items)
    total_bytes = allreduce_sum(world, float(bytes_per_step * K))
    value = total_bytes / (elapsed_ms / 1e3) / 1e9
    launches_per_step = sum(p.num_launches for p in plans)

    # per class / element size; per kernel instantiation (one per elem size)
    durs = [0.0] * len(items)
    step_durs = [[0.0] * K for _ in range(len(items))]
    for k in range(K):
        for i in range(len(items)):
            ev = per_item[k * len(items) + i]
            step_durs[i][k] = ev[0].elapsed_time(ev[1])
            durs[i] += step_durs[i][k] / K
    # The timed region's first launch follows the idle gap of the barrier and
    # synchronisation before it, and runs slower than the same launch in the
    # later steps; the per-class breakdown takes the median over the steps.
    first_launch_gbs = 2 * N * items[0][1] / (step_durs[0][0] / 1e3) / 1e9
    by_class = {}
    class_steps = {}
    kernel_time = {}
    kernel_launches = {}
    kernel_bytes = {}
    for i, (cls, e, rows, c) in enumerate(items):
        key = "%s_e%d" % (cls, e)
        b = 2 * N * e
        d = by_class.setdefault(key, {"bytes": 0, "ms": 0.0, "count": 0,
                                      "launches": plans[i].num_launches})
        d["bytes"] += b
        d["ms"] += durs[i]
        d["count"] += 1
        cs = class_steps.setdefault(key, [0.0] * K)
        for k in range(K):
            cs[k] += step_durs[i][k]
        kname = "%s<%d>" % ("bmmc_tiled_pass_tma" if args.load == "tma" else "bmmc_tiled_pass",
                            {4: 2, 8: 3, 16: 4}[e])
        kernel_time[kname] = kernel_time.get(kname, 0.0) + durs[i]
        kernel_launches[kname] = kernel_launches.get(kname, 0) + plans[i].num_launches
        kernel_bytes[kname] = kernel_bytes.get(kname, 0) + b * plans[i].num_launches

    # ---- same-run D2D copy baseline ---------------------------------------
    d2d = {}
    for e in elems:
        x, y, _ = bufs[e]
        for _ in range(3):
            y.copy_(x)
        evs = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True))
               for _ in range(10)]
        for a, b in evs:
            a.record(stream)
            y.copy_(x)
            b.record(stream)
        torch.cuda.synchronize(dev)
        ms = statistics.median(a.elapsed_time(b) for a, b in evs)
        d2d[e] = 2 * N * e / (ms / 1e3) / 1e9
    breakdown = {}
    for key, d in sorted(by_class.items()):
        e = int(key.rsplit("_e", 1)[1])
        gbs = d["bytes"] / (statistics.median(class_steps[key]) / 1e3) / 1e9
        breakdown[key] = {"gbs": round(gbs, 1), "frac_of_d2d": round(gbs / d2d[e], 4),
                          "launches": d["launches"], "count": d["count"]}

    # ---- roofline of the dominant kernel ----------------------------------
    dom = max(kernel_time, key=kernel_time.get)
    avg_launch_ms = kernel_time[dom] / kernel_launches[dom]
    bytes_per_launch = kernel_bytes[dom] / kernel_launches[dom]
    achieved = bytes_per_launch / (avg_launch_ms / 1e3) / 1e9
    peak, peak_src = measured_hbm_peak()
    traffic, traffic_note = profiled_traffic(dom)
    step_ms_sum = sum(kernel_time.values())
    roofline = {"bound": "hbm", "kernel": dom, "achieved": round(achieved, 1),
                "peak": peak, "peak_source": peak_src, "unit": "GB/s",
                "frac": round(achieved / peak, 4), "traffic": traffic,
                "algorithmic_bytes_per_launch": bytes_per_launch,
                "avg_launch_ms": round(avg_launch_ms, 4),
                "share_of_step": round(kernel_time[dom] / step_ms_sum, 4)}
    if traffic_note and traffic is None:
        roofline["traffic_note"] = traffic_note
    # every kernel instantiation of the step against the same peak
    kernels = {}
    for k in sorted(kernel_time):
        ms_l = kernel_time[k] / kernel_launches[k]
        a = kernel_bytes[k] / kernel_launches[k] / (ms_l / 1e3) / 1e9
        kernels[k] = {"achieved_gbs": round(a, 1), "frac_of_peak": round(a / peak, 4),
                      "launches_per_step": kernel_launches[k],
                      "share_of_step": round(kernel_time[k] / step_ms_sum, 4)}

    extras = {"kernels": kernels}
    # ---- single-pass strategy on the dense set (beyond the paper) ---------
    if not args.no_extras and args.strategy == "paper":
        sp = {}
        for e in elems:
            dense = [(rows, c) for (cls, ee, rows, c) in items if cls == "dense" and ee == e]
            if not dense:
                continue
            sp_plans = [bm.Plan(n, rows, c, e, flags=bm.BMMC_PLAN_SINGLE_PASS)
                        for rows, c in dense[:16]]
            x, y, ws = bufs[e]
            for p in sp_plans:
                p(x, out=y, stream=stream)
            a = torch.cuda.Event(enable_timing=True)
            b = torch.cuda.Event(enable_timing=True)
            torch.cuda.synchronize(dev)
            a.record(stream)
            for _ in range(2):
                for p in sp_plans:
                    p(x, out=y, stream=stream)
            b.record(stream)
            torch.cuda.synchronize(dev)
            gbs = 2 * len(sp_plans) * 2 * N * e / (a.elapsed_time(b) / 1e3) / 1e9
            sp["dense_e%d" % e] = {"gbs": round(gbs, 1), "frac_of_d2d": round(gbs / d2d[e], 4),
                                   "passes": 1, "count": len(sp_plans)}
        extras["single_pass_dense"] = sp

    # The legs below report the other configurations beside the headline; a
    # leg that raises is recorded as an error in its place, so that it cannot
    # take the headline line down with it.
    def leg(key, fn, *a, **kw):
        try:
            extras[key] = fn(*a, **kw)
        except Exception as exc:  # reported in the JSON line
            extras[key] = {"error": "%s: %s" % (type(exc).__name__, exc)}
            print("bench leg %s failed: %r" % (key, exc), file=sys.stderr)
        torch.cuda.synchronize(dev)
        torch.cuda.empty_cache()

    # The L2-resident legs run before the end-to-end leg's large staging
    # allocations (after those, the same replays measured 10-25 % slower).
    if not args.no_small:
        leg("n20_config", bench_n20, dev)
        leg("sorting_network", bench_sorting, dev)

    # ---- end to end through the public API with host buffers --------------
    e2e = None
    if not args.no_e2e:
        host = {}
        for e in elems:
            x, y, _ = bufs[e]
            hin = torch.empty(x.numel(), dtype=x.dtype, pin_memory=True)
            hin.copy_(x)
            hout = torch.empty_like(hin, pin_memory=True)
            host[e] = (hin, hout)
        torch.cuda.synchronize(dev)

        # Every permutation is one bmmc_execute_host call (upload, passes,
        # download on one stream).  Consecutive calls rotate over three
        # streams, each with its own staging buffers, so the upload of one
        # permutation, the kernels of the previous one and the download of the
        # one before that run at once (the host link is full duplex).
        NS = 3
        sets = {e: [bufs[e]] + [tuple(torch.empty_like(t) for t in bufs[e])
                                for _ in range(NS - 1)] for e in elems}
        streams = [torch.cuda.Stream(device=dev) for _ in range(NS)]

        def e2e_step():
            for i, (cls, e, rows, c) in enumerate(items):
                j = i % NS
                x, y, ws = sets[e][j]
                hin, hout = host[e]
                plans[i].execute_host(hin, hout, x, y, stream=streams[j], workspace=ws)

        # The host link alone: the same copies on the same streams with no
        # kernel (the download reads back the buffer the upload filled).  This
        # is the ceiling of the end-to-end number.
        def link_step():
            for i, (cls, e, rows, c) in enumerate(items):
                j = i % NS
                x, y, ws = sets[e][j]
                hin, hout = host[e]
                with torch.cuda.stream(streams[j]):
                    x.copy_(hin, non_blocking=True)
                    hout.copy_(x, non_blocking=True)

        def timed(step, reps):
            cur = torch.cuda.current_stream(dev)
            a = torch.cuda.Event(enable_timing=True)
            b = torch.cuda.Event(enable_timing=True)
            torch.cuda.synchronize(dev)
            a.record(cur)
            for st in streams:
                st.wait_stream(cur)
            for _ in range(reps):
                step()
            for st in streams:
                cur.wait_stream(st)
            b.record(cur)
            torch.cuda.synchronize(dev)
            return a.elapsed_time(b)

        e2e_step()
        torch.cuda.synchronize(dev)
        barrier(world)
        ms = timed(e2e_step, args.e2e_steps)
        link_ms = timed(link_step, 1)
        del sets
        barrier(world)
        ms = allreduce_max(world, ms)
        link_ms = allreduce_max(world, link_ms)
        e2e_bytes = allreduce_sum(world, float(bytes_per_step * args.e2e_steps))
        hbytes = sum(N * e for (_, e, _, _) in items)
        link_gbs = bytes_per_step * world / (link_ms / 1e3) / 1e9
        e2e = {"value": round(e2e_bytes / (ms / 1e3) / 1e9, 1), "unit": "GB/s",
               "h2d_bytes_per_step": hbytes, "d2h_bytes_per_step": hbytes,
               "steps": args.e2e_steps, "warmup": 1, "entry_point": "bmmc_execute_host",
               "copies_only_gbs": round(link_gbs, 1),
               "frac_of_copies_only": round(e2e_bytes / (ms / 1e3) / 1e9 / link_gbs, 4)}
        del host

    del bufs
    torch.cuda.empty_cache()

    if not args.no_autograd:
        leg("autograd", bench_autograd, dev)
    if not args.no_batched:
        leg("batched", bench_batched, dev, stream, count=args.batched_count)
    if not args.no_serving:
        leg("serving", bench_serving, dev, seconds=args.serving_seconds)

    cpu = None
    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        cpu = cpu_baseline()

    if rank == 0:
        line = {
            "metric": METRIC, "value": round(value, 1), "unit": "GB/s",
            "n_gpus": world, "steps": K, "warmup": W,
            "ms_per_step": round(elapsed_ms / K, 3), "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": DTYPE,
            "data": "synthetic",
            "config": workload_config(args, world),
            "roofline": roofline,
            "cpu_baseline": cpu,
            "e2e": e2e,
            "gpu_launches": launches_per_step * K,
            "clocks": clocks,
            "d2d_copy_gbs": {str(e): round(v, 1) for e, v in d2d.items()},
            "frac_of_d2d": round(value / (sum(d2d[e] * sum(1 for it in items if it[1] == e) * e
                                              for e in elems)
                                          / sum(it[1] for it in items)), 4),
            "breakdown": breakdown,
            "breakdown_stat": "per class, the median over the timed steps of its summed "
                              "launch times",
            "first_launch_after_idle": {"item": "%s_e%d" % (items[0][0], items[0][1]),
                                        "gbs": round(first_launch_gbs, 1)},
            "wall_s_timed": round(wall1 - wall0, 3),
        }
        line.update(extras)
        print(json.dumps(line))
    if world > 1:
        import torch.distributed as dist
        dist.destroy_process_group()
    return 0


if __name__ == "__main__":
    sys.exit(main())
