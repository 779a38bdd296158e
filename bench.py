"""Benchmark: incremental max-flow updates/s on the R-MAT scale-20 workload.

One step = one whole pass of the hot path over one batch: apply the batch and
repair the preflow (the batch part of Alg. 5), then the backward-BFS / worklist /
discharge / remove-invalid loop until no active vertex remains, then the
value.  The graph is R-MAT scale 20 (2^20 vertices, 16 x 2^20 draws,
a/b/c/d = 0.57/0.19/0.19/0.05, self-loops dropped, duplicates merged, caps
U[1,1000]); batches are mixed (40% increase, 40% decrease, 10% insert, 10%
delete) of --batch updates.  The residual state (~0.6 GB) is larger than the
129 MB L2, so no flush is needed between steps.

  python bench.py [--gpus N] [--steps K] [--warmup W] [--batch B] [--impl ours|reference]

With N > 1 every rank runs its own replica on its own GPU: push-relabel on
one graph needs an exchange at every sweep and a global BFS, so the path does
not shard, and replicas need no collective on the data path.  Rank 0 reports
the aggregate (the units of all ranks over the slowest rank's timed region).
Launched as `python bench.py --gpus N` without torchrun, the script starts the
N ranks itself through torch.distributed.run.  --impl reference times the CPU
oracle (Dinic recomputed from scratch after each batch) on rank 0 only.

Besides the headline workload the default run measures the other shapes of
the metric in a `configs` block: the small Erdos-Renyi graph (n=4096,
m=32768, batches of 256), R-MAT 20 with batches of 1K and 100K, the 2048x2048
segmentation grid with its window batches, and 64 uneven instances in one
batched launch; each with kernel latency, the static re-solve and their ratio.
"""
from __future__ import annotations

import argparse
import json
import os
import subprocess
import sys
import threading
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

METRIC = "dynamic maxflow updates/s & p50/p99 batch latency vs static re-solve; HBM GB/s"
UNIT = "updates/s"
HBM_FALLBACK_GBS = 6800.0
HBM_NOMINAL_GBS = 7900.0           # the part's nominal HBM3e bandwidth, for context beside the measured copy


def _peaks():
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as f:
            return json.load(f), "measured"
    except Exception:
        return {"hbm_gbs": HBM_FALLBACK_GBS}, "fallback"


def measured_traffic(workload: str, batch: int):
    """DRAM bytes per launch from the committed ncu summary, if the kernel is unchanged since.

    The summary records a digest of the kernel's code (comments and whitespace
    left out) at capture time; when the code differs now, the counters no
    longer describe this kernel and the traffic is reported as null.
    """
    import hashlib
    if workload != "rmat20" or batch != 10000:
        return None
    path = os.path.join(ROOT, "profiles", "mf_solve_kernel_rmat20_traffic.md")
    try:
        txt = open(path).read()
        want = txt.split("kernel_code_sha256:")[1].split()[0]
        val = int(txt.split("traffic_bytes_per_launch:")[1].split()[0])
    except (OSError, IndexError, ValueError):
        return None
    h = hashlib.sha256()
    for f in ("solver.cu", "mf_internal.h"):
        with open(os.path.join(ROOT, "paper_2511_01235_gb300", "csrc", f)) as fh:
            h.update(code_only(fh.read()).encode())
    return val if h.hexdigest() == want else None


def code_only(src: str) -> str:
    """C/C++ source without its comments, one space per run of whitespace: an
    edit to a comment leaves the digest of the code unchanged."""
    out, i, n = [], 0, len(src)
    while i < n:
        c = src[i]
        if c in "\"'":                                   # a literal, copied whole
            j = i + 1
            while j < n and src[j] != c:
                j += 2 if src[j] == "\\" else 1
            out.append(src[i:j + 1])
            i = j + 1
        elif src.startswith("//", i):
            j = src.find("\n", i)
            i = n if j < 0 else j
        elif src.startswith("/*", i):
            j = src.find("*/", i + 2)
            out.append(" ")
            i = n if j < 0 else j + 2
        else:
            out.append(c)
            i += 1
    return " ".join("".join(out).split())


class ClockSampler:
    """SM clocks and throttle reasons, sampled during the timed region: through
    NVML (read-only queries, every 5 ms, from a thread) where libnvidia-ml loads,
    else nvidia-smi's own loop (every 100 ms)."""

    Q = ("clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.hw_slowdown,"
         "clocks_event_reasons.hw_thermal_slowdown,clocks_event_reasons.sw_thermal_slowdown,"
         "clocks_event_reasons.sw_power_cap")
    # NVML clock event reason bits (nvml.h): the four that mark a throttled run
    REASON_BITS = {"sw_power_cap": 0x4, "hw_slowdown": 0x8, "sw_thermal_slowdown": 0x20,
                   "hw_thermal_slowdown": 0x40}

    def __init__(self, index: int):
        self.index = index
        self.proc = None
        self.lines = []
        self.samples = []            # NVML: (sm MHz, max MHz, reason bits)
        self.nvml = None
        self.stop_evt = threading.Event()

    def _nvml_open(self):
        import ctypes
        lib = ctypes.CDLL("libnvidia-ml.so.1")
        if lib.nvmlInit_v2() != 0:
            return None
        h = ctypes.c_void_p()
        if lib.nvmlDeviceGetHandleByIndex_v2(ctypes.c_uint(self.index), ctypes.byref(h)) != 0:
            return None
        reasons = getattr(lib, "nvmlDeviceGetCurrentClocksEventReasons", None) or \
            getattr(lib, "nvmlDeviceGetCurrentClocksThrottleReasons")
        return lib, h, reasons

    def _nvml_loop(self):
        import ctypes
        lib, h, reasons = self.nvml
        clk, mx, bits = ctypes.c_uint(), ctypes.c_uint(), ctypes.c_ulonglong()
        while not self.stop_evt.is_set():
            if (lib.nvmlDeviceGetClockInfo(h, 1, ctypes.byref(clk)) == 0 and
                    lib.nvmlDeviceGetMaxClockInfo(h, 1, ctypes.byref(mx)) == 0 and reasons(h, ctypes.byref(bits)) == 0):
                self.samples.append((clk.value, mx.value, bits.value))
            self.stop_evt.wait(0.005)

    def start(self):
        try:
            self.nvml = self._nvml_open()
        except Exception:
            self.nvml = None
        if self.nvml is not None:
            self.t = threading.Thread(target=self._nvml_loop, daemon=True)
            self.t.start()
            return
        try:
            self.proc = subprocess.Popen(["nvidia-smi", "-i", str(self.index), f"--query-gpu={self.Q}",
                                          "--format=csv,noheader,nounits", "-lms", "100"],
                                         stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.t = threading.Thread(target=self._read, daemon=True)
            self.t.start()
        except Exception:
            self.proc = None

    def _read(self):
        for line in self.proc.stdout:
            self.lines.append(line.strip())

    def stop(self):
        if self.nvml is not None:
            self.stop_evt.set()
            self.t.join(timeout=5)
            sm = [x[0] for x in self.samples]
            mx = [x[1] for x in self.samples]
            reasons = {nm for nm, bit in self.REASON_BITS.items() for x in self.samples if x[2] & bit}
            return {"sm_mhz": float(np.median(sm)) if sm else None, "sm_max_mhz": max(mx) if mx else None,
                    "reasons": sorted(reasons), "samples": len(sm), "source": "nvml, every 5 ms"}
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except Exception:
            self.proc.kill()
        sm, mx, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for ln in self.lines:
            parts = [p.strip() for p in ln.split(",")]
            if len(parts) < 7:
                continue
            try:
                sm.append(float(parts[0]))
                mx.append(float(parts[1]))
            except ValueError:
                continue
            for nm, val in zip(names, parts[3:7]):
                if val.lower() in ("active", "1", "yes"):
                    reasons.add(nm)
        return {"sm_mhz": float(np.median(sm)) if sm else None, "sm_max_mhz": max(mx) if mx else None,
                "reasons": sorted(reasons), "samples": len(sm), "source": "nvidia-smi, every 100 ms"}


class Workload:
    """A graph plus a deterministic stream of update batches."""

    def __init__(self, args):
        from paper_2511_01235_gb300 import workloads as W
        self.kind = args.workload
        self.grid = None
        if self.kind.startswith("rmat"):
            scale = int(self.kind[4:] or 20)
            self.g = W.rmat(scale, 16, 0.57, 0.19, 0.19, seed=2 if scale == 20 else 10 + scale, cap_lo=1,
                            cap_hi=1000)
            self.ins_hi = 1000
        elif self.kind == "er_small":
            self.g = W.er_small()
            self.ins_hi = 100
        elif self.kind.startswith("grid"):
            side = int(self.kind[4:] or 2048)
            self.grid = W.GridSegmentation(side=side, seed=3)
            self.g = self.grid.graph()
            self.ins_hi = 1000
        else:
            raise SystemExit(f"unknown workload {self.kind}")
        self.es = W.EdgeSet(self.g.n, self.g.src, self.g.dst, self.g.cap)
        self.rng = np.random.default_rng(1234)
        self.k = 0

    def batches(self, count, B):
        from paper_2511_01235_gb300 import workloads as W
        out = []
        for _ in range(count):
            if self.grid is not None:
                b = self.grid.window_batch(self.k % 30)
            else:
                b = W.mixed_batch(self.es, B, self.rng, ins_cap_hi=self.ins_hi)
            self.es.apply(b.u, b.v, b.cap)
            self.k += 1
            out.append(b)
        return out

    def describe(self):
        if self.kind.startswith("rmat"):
            return (f"{self.kind}: R-MAT scale {self.kind[4:] or 20}, edge factor 16, a/b/c=0.57/0.19/0.19, "
                    f"caps U[1,1000], mixed batches 40/40/10/10")
        if self.kind == "er_small":
            return "er_small: Erdos-Renyi n=4096 m=32768 caps U[1,100], mixed batches 40/40/10/10"
        return (f"{self.kind}: {self.grid.side}x{self.grid.side} 4-connected segmentation grid, "
                f"t-links re-drawn in a 256x256 window shifting 8 px per batch")


def aggregate_over_ranks(tot_ms: float, units_per_rank: int, device=None):
    """Whole-job throughput of independent replicas: the units of all ranks over
    the slowest rank's timed region (max over ranks).  Returns (value, max_ms, world)."""
    ws = 1
    try:
        import torch.distributed as dist
        if dist.is_available() and dist.is_initialized():
            import torch
            ws = dist.get_world_size()
            t = torch.tensor([float(tot_ms)], dtype=torch.float64, device=device)
            dist.all_reduce(t, op=dist.ReduceOp.MAX)
            tot_ms = float(t.item())
    except ImportError:
        pass
    return ws * units_per_rank / (tot_ms / 1e3), tot_ms, ws


def dist_env():
    ws = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return ws, rank, local


def run_reference(args):
    """The CPU oracle timed on this host: Dinic from scratch on the updated graph, per batch."""
    import oracle
    ws, rank, _ = dist_env()
    if rank != 0:
        return
    wl = Workload(args)
    g = wl.g
    # a bounded sample: one warm-up batch, then at most 12 timed batches and ~60 s of oracle time
    # (Dinic from scratch takes seconds per batch on the large graphs)
    warm = min(args.warmup, 1)
    batches = wl.batches(warm + min(args.steps, 12), args.batch)
    args.batch = batches[0].size
    es2 = W_edgeset(g)
    times = []
    for i, b in enumerate(batches):
        es2.apply(b.u, b.v, b.cap)
        u, v, c = es2.coo()
        t0 = time.perf_counter()
        oracle.maxflow(g.n, u, v, c, g.s, g.t)
        dt = time.perf_counter() - t0
        if i >= warm:
            times.append(dt)
            if sum(times) > 60.0:
                break
    tot = sum(times)
    val = args.batch * len(times) / tot
    line = {"impl": "reference", "metric": METRIC, "value": val, "unit": UNIT, "n_gpus": args.gpus,
            "steps": len(times), "warmup": warm, "ms_per_step": 1e3 * tot / len(times),
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "int64",
            "data": "synthetic", "config": config_of(args, g, wl, ws),
            "cpu_baseline": {"value": val, "unit": UNIT, "cores": 1, "kind": "oracle",
                             "sample": f"{len(times)} batches of {args.batch} "
                                       f"(of {args.steps} asked; bounded to ~60 s); "
                                       "Dinic recomputed from scratch per batch"},
            "e2e": {"value": val, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)


def W_edgeset(g):
    from paper_2511_01235_gb300 import workloads as W
    return W.EdgeSet(g.n, g.src, g.dst, g.cap)


def config_of(args, g, wl, world=1):
    return {"workload": wl.describe(),
            "n": int(g.n), "m_merged": int(g.m), "s": int(g.s), "t": int(g.t), "batch": args.batch,
            "l2": "inputs larger than L2 (residual state of R-MAT 20 / grid 2048 ~0.6 GB vs 129 MB L2)",
            "parallelism": f"replicas x{world}"}


def replica_command(argv, n, port):
    """The torch.distributed.run command that starts n ranks of this script, one per local GPU."""
    return [sys.executable, "-m", "torch.distributed.run", "--nnodes=1", f"--nproc-per-node={n}",
            "--master-addr=127.0.0.1", f"--master-port={port}", os.path.abspath(__file__)] + list(argv)


def launch_replicas(argv, n):
    """Start n replicas of this script (one process per GPU) and return their exit status.
    Refuses cleanly when the host has fewer than n GPUs."""
    import socket
    import torch
    have = torch.cuda.device_count() if torch.cuda.is_available() else 0
    if have < n:
        sys.stderr.write(f"bench.py: --gpus {n} needs {n} GPUs on this host, found {have}\n")
        return 2
    sk = socket.socket()
    sk.bind(("127.0.0.1", 0))
    port = sk.getsockname()[1]
    sk.close()
    return subprocess.call(replica_command(argv, n, port))


def cpu_baseline_sample(g, batches, budget_s=20.0):
    import oracle
    es2 = W_edgeset(g)
    times = []
    t_start = time.perf_counter()
    for b in batches:
        es2.apply(b.u, b.v, b.cap)
        u, v, c = es2.coo()
        t0 = time.perf_counter()
        oracle.maxflow(g.n, u, v, c, g.s, g.t)
        times.append(time.perf_counter() - t0)
        if time.perf_counter() - t_start > budget_s:
            break
    return times


def cpu_baseline_batched(gs):
    """The oracle on every instance (Dinic from scratch), spread over all host
    cores by a thread pool: ctypes releases the GIL during each call, so the
    threads run in parallel.  Returns (instances/s, threads, values)."""
    from concurrent.futures import ThreadPoolExecutor

    import oracle
    oracle.maxflow(2, [0], [1], [1], 0, 1)          # build and load once, before the threads
    threads = os.cpu_count() or 1
    t0 = time.perf_counter()
    with ThreadPoolExecutor(threads) as ex:
        vals = list(ex.map(lambda g: oracle.maxflow(g.n, g.src, g.dst, g.cap, g.s, g.t).value, gs))
    return len(gs) / (time.perf_counter() - t0), threads, vals


def _phase_rates(S, totals):
    """Add the last call's per-phase algorithmic bytes and device time to totals."""
    st = S.stats()
    for ph, bk, mk in (("bfs", "bytes_bfs", "ms_bfs"), ("discharge", "bytes_discharge", "ms_discharge"),
                       ("fix", "bytes_fix", "ms_fix"), ("apply", "bytes_apply", "ms_apply")):
        t = totals.setdefault(ph, [0.0, 0.0])
        t[0] += st[bk]
        t[1] += st[mk]
    return st


def phase_roofline(totals, hbm):
    """Per phase: algorithmic bytes over the phase's device time (hook timestamps), against the peak."""
    out = {}
    for ph, (b, ms) in totals.items():
        gbs = b / (ms * 1e-3) / 1e9 if ms > 0 else 0.0
        out[ph] = {"bytes": int(b), "ms": float(ms), "gbs": gbs, "frac": gbs / hbm}
    return out


def dynamic_config(name, S, es, batch_fn, steps, warm, static_reps, check_each, hbm, describe):
    """Incremental updates on S (kernel device time per update), then the static re-solve of the
    final graph; the oracle checks the final value (and every batch's with check_each)."""
    import oracle
    import torch
    batches = []
    for _ in range(warm + steps):
        b = batch_fn(es)
        es.apply(b.u, b.v, b.cap)
        batches.append((b, es.copy() if check_each else None))
    kms, totals, checked, equal = [], {}, 0, True
    detail = []
    for k, (b, es_k) in enumerate(batches):
        S.update(torch.from_numpy(b.u).cuda(), torch.from_numpy(b.v).cuda(), torch.from_numpy(b.cap).cuda())
        if k < warm:
            continue
        st = _phase_rates(S, totals)
        kms.append(st["ms_update"])
        detail.append([round(st["ms_update"], 3), st["iterations"], st["bfs_levels"], st["barriers"]])
        if check_each:
            u, v, c = es_k.coo()
            equal &= S.query()[0] == oracle.maxflow(es_k.n, u, v, c, S.s, S.t).value
            checked += 1
    value = S.query()[0]
    if not check_each:
        u, v, c = es.coo()
        equal &= value == oracle.maxflow(es.n, u, v, c, S.s, S.t).value
        checked += 1
    static_ms = []
    for _ in range(static_reps):
        S.resolve_static()
        static_ms.append(S.stats()["ms_update"])
        equal &= S.query()[0] == value
    kp50 = float(np.percentile(kms, 50))
    sms = float(np.median(static_ms))
    B = int(batches[0][0].size)
    return {"workload": describe, "batch": B, "steps": steps, "warmup": warm,
            "kernel_ms": {"p50": kp50, "p99": float(np.percentile(kms, 99)), "mean": float(np.mean(kms))},
            "updates_per_s": B * len(kms) / (sum(kms) / 1e3),
            "static_resolve_ms": sms, "speedup_vs_static": sms / kp50 if kp50 > 0 else None,
            "phases": phase_roofline(totals, hbm),
            "flow_check": {"batches_checked": checked, "equal": bool(equal)},
            "steps_detail": {"cols": ["kernel_ms", "iterations", "bfs_levels", "barriers"], "rows": detail}}


def run_configs(S, es_main, hbm):
    """The other shapes of the metric, each with kernel latency, static re-solve and their ratio."""
    import torch
    from paper_2511_01235_gb300 import native
    from paper_2511_01235_gb300 import workloads as W
    out = {}
    t0 = time.perf_counter()
    # small Erdos-Renyi: n=4096, m=32768, caps U[1,100]; 10 batches of 256 (40/40/10/10), every one checked
    g = W.er_small()
    C1 = native.Solver(g.n, g.src, g.dst, g.cap, g.s, g.t, stream=torch.cuda.current_stream())
    rng = np.random.default_rng(11)
    out["er_small"] = dynamic_config(
        "er_small", C1, W.EdgeSet(g.n, g.src, g.dst, g.cap),
        lambda es: W.mixed_batch(es, 256, rng, ins_cap_hi=100), 10, 3, 3, True, hbm,
        "Erdos-Renyi n=4096 m=32768 caps U[1,100], s=0, t=4095; batches of 256 (40/40/10/10)")
    C1.close()
    # R-MAT 20 with small (1K) and large (100K) batches, on clones of the headline state
    for B, steps in ((1000, 10), (100000, 4)):
        C = S.clone()
        rng = np.random.default_rng(2000 + B)
        out[f"rmat20_{B // 1000}k"] = dynamic_config(
            f"rmat20_{B // 1000}k", C, es_main.copy(), lambda es, B=B: W.mixed_batch(es, B, rng, ins_cap_hi=1000),
            steps, 2, 2, False, hbm, f"R-MAT scale 20 (the headline graph and state); batches of {B} (40/40/10/10)")
        C.close()
    # segmentation grid 2048x2048: t-links re-drawn in a 256x256 window shifting 8 px per batch
    grid = W.GridSegmentation(side=2048, seed=3)
    g = grid.graph()
    G = native.Solver(g.n, g.src, g.dst, g.cap, g.s, g.t, stream=torch.cuda.current_stream())
    ks = iter(range(30))
    out["grid2048"] = dynamic_config(
        "grid2048", G, W.EdgeSet(g.n, g.src, g.dst, g.cap), lambda es: grid.window_batch(next(ks)), 3, 1, 2, False,
        hbm, "2048x2048 4-connected segmentation grid (n=4,194,306), t-links re-drawn in a 256x256 window "
             "shifting 8 px per batch (131,072 updates)")
    G.close()
    out["batched64"] = batched_summary()
    out["serving"] = serving_summary()
    out["wall_s"] = time.perf_counter() - t0
    return out


SERVING_SMALL = ["--workload", "serving:18,18,19,19,20", "--steps", "60", "--warmup", "3", "--budget-gb", "1.5"]


def serving_summary():
    """A small serving run (five R-MAT graphs of scales 18-20 under a 1.5 GB budget, 60 Poisson
    requests) in a child process of this script; the full one is --workload serving."""
    import subprocess
    cmd = [sys.executable, os.path.abspath(__file__)] + SERVING_SMALL
    t0 = time.perf_counter()
    try:
        r = subprocess.run(cmd, capture_output=True, text=True, timeout=600, cwd=ROOT)
    except subprocess.TimeoutExpired:
        return {"error": "timed out after 600 s", "command": " ".join(SERVING_SMALL)}
    lines = [ln for ln in r.stdout.splitlines() if ln.startswith("{")]
    if r.returncode != 0 or not lines:
        return {"error": f"exit {r.returncode}: {r.stderr.strip().splitlines()[-1:]}", "command": " ".join(SERVING_SMALL)}
    d = json.loads(lines[-1])
    return {"command": "bench.py " + " ".join(SERVING_SMALL), "workload": d["config"]["workload"],
            "updates_per_s": d["value"], "latency_ms": d["latency_ms"], "states_gb": d["config"]["states_gb"],
            "budget_gb": d["config"]["budget_gb"], "evictions": d["serving"].get("evictions"),
            "flow_check": d["flow_check"], "gpu_launches": d["gpu_launches"],
            "offered_rate_per_s": d["config"]["rate_per_s"], "calibration": d["calibration"],
            "wall_s": time.perf_counter() - t0}


def batched_summary():
    """64 uneven instances in one persistent launch (default configuration, no autotuning)."""
    import torch
    from paper_2511_01235_gb300 import autotune, native
    from paper_2511_01235_gb300 import workloads as W
    gs = W.batched_instances(count=64, seed=4)
    S = [native.Solver(g.n, g.src, g.dst, g.cap, g.s, g.t, stream=torch.cuda.current_stream()) for g in gs]
    vals = [s.query()[0] for s in S]
    cfg = autotune.DEFAULT
    autotune.apply_config(S, cfg)
    native.maxflow_solve_batched(S, None, group_blocks=cfg["group_blocks"])
    ms = [native.maxflow_solve_batched(S, None, group_blocks=cfg["group_blocks"]) for _ in range(3)]
    same = [s.query()[0] for s in S] == vals
    one = 0.0
    for s in S:
        s.resolve_static()
        one += s.stats()["ms_update"]
    cpu_rate, cpu_threads, cpu_vals = cpu_baseline_batched(gs)
    for s in S:
        s.close()
    best = float(np.median(ms))
    return {"workload": "64 instances, n log-uniform in [1e3, 2e5], ER / layered DAG / geometric, caps U[1,500]",
            "instances_per_s": len(gs) / (best / 1e3), "ms_per_batched_solve": best, "one_by_one_ms": one,
            "speedup_vs_one_by_one": one / best, "config": {k: (list(v) if isinstance(v, tuple) else v)
                                                            for k, v in cfg.items()},
            "cpu_baseline": {"value": cpu_rate, "unit": "instances/s", "cores": cpu_threads, "kind": "oracle",
                             "sample": f"all {len(gs)} instances, one per thread"},
            "flow_check": {"instances": len(gs), "equal": bool(same and cpu_vals == vals)}}


def scheduler_comparison(S, wl, count):
    """The learned schedule against the paper's fixed one and the library default on the same
    held-out batches (sizes log-uniform in [1K, 100K], the headline mix), each on its own clone
    of one state.  Device time per call from CUDA events on the solver's stream: the learned
    path pays for its features and forward pass."""
    import math

    import torch
    from paper_2511_01235_gb300 import scheduler as SCH
    from paper_2511_01235_gb300 import workloads as W
    if not os.path.exists(SCH.DEFAULT_WEIGHTS):
        return None
    mlp = SCH.load()
    rng = np.random.default_rng(4321)
    es = wl.es.copy()
    sizes = [int(x) for x in np.exp(rng.uniform(math.log(1000), math.log(100_000), size=count))]
    batches = []
    for B in sizes:
        b = W.mixed_batch(es, B, rng, ins_cap_hi=wl.ins_hi)
        es.apply(b.u, b.v, b.cap)
        batches.append(b)
    out = {"batches": len(batches), "sizes": sizes}
    picks = []
    C = S.clone()               # once through untimed: the first arm would pay for the first use of batches and sizes
    for b in batches:
        C.update(b.u, b.v, b.cap)
    C.close()
    for key in ("learned", "paper", "default"):
        C = S.clone()
        ts = []
        for b in batches:
            e0 = torch.cuda.Event(enable_timing=True)
            e1 = torch.cuda.Event(enable_timing=True)
            e0.record(C.stream)
            if key == "learned":
                picks.append(C.update_scheduled(b.u, b.v, b.cap, mlp))
            else:
                C.run_action(b.u, b.v, b.cap, SCH.ACTION_PAPER if key == "paper" else SCH.ACTION_DEFAULT)
            e1.record(C.stream)
            e1.synchronize()
            ts.append(e0.elapsed_time(e1))
        out[key + "_ms_total"] = float(np.sum(ts))
        out[key + "_ms_mean"] = float(np.mean(ts))
        out[key + "_value"] = int(C.query()[0])
        C.close()
    out["learned_vs_default"] = out["learned_ms_total"] / out["default_ms_total"]
    out["learned_vs_paper"] = out["learned_ms_total"] / out["paper_ms_total"]
    out["learned_picks"] = np.bincount(picks, minlength=len(native_actions())).tolist()
    out["values_equal"] = len({out["learned_value"], out["paper_value"], out["default_value"]}) == 1
    out["note"] = ("device ms per update call (CUDA events), host batches; paper = 1 round, K = avg degree, "
                   "Alg. 3; default = the library's adaptive schedule")
    return out


def native_actions():
    from paper_2511_01235_gb300 import native
    return native.maxflow_sched_actions()


def run_batched(args):
    """Many uneven instances in one persistent launch (64 graphs of 1K-200K vertices)."""
    import torch
    from paper_2511_01235_gb300 import autotune, native
    from paper_2511_01235_gb300 import workloads as W
    torch.cuda.set_device(0)
    native.load()
    gs = W.batched_instances(count=64, seed=4)
    S = [native.Solver(g.n, g.src, g.dst, g.cap, g.s, g.t) for g in gs]
    ref_values = [s.query()[0] for s in S]
    best, best_ms, trials = autotune.tune(S, passes=2, reps=2)
    for _ in range(args.warmup):
        native.maxflow_solve_batched(S, None, group_blocks=best["group_blocks"])
    clk = ClockSampler(0)
    clk.start()
    l0 = native.kernel_launches()
    ms = [native.maxflow_solve_batched(S, None, group_blocks=best["group_blocks"]) for _ in range(args.steps)]
    launches = native.kernel_launches() - l0
    clocks = clk.stop()
    assert [s.query()[0] for s in S] == ref_values
    # one by one, each instance alone on the whole GPU (same settings)
    one = []
    for _ in range(2):
        t = 0.0
        for s in S:
            s.resolve_static()
            t += s.stats()["ms_update"]
        one.append(t)
    # default configuration, batched
    autotune.apply_config(S, autotune.DEFAULT)
    ms_default = min(native.maxflow_solve_batched(S, None, group_blocks=autotune.DEFAULT["group_blocks"])
                     for _ in range(3))
    autotune.apply_config(S, best)
    # one mixed batch of 1% of the edges per instance, batched
    rng = np.random.default_rng(44)
    batches = []
    for g in gs:
        es = W.EdgeSet(g.n, g.src, g.dst, g.cap)
        b = W.mixed_batch(es, max(1, es.m // 100), rng, ins_cap_hi=500)
        batches.append((torch.from_numpy(b.u).cuda(), torch.from_numpy(b.v).cuda(), torch.from_numpy(b.cap).cuda()))
    upd_ms = native.maxflow_solve_batched(S, batches, group_blocks=best["group_blocks"])
    n_upd = int(sum(int(b[0].numel()) for b in batches))
    cpu_rate, cpu_threads, cpu_vals = cpu_baseline_batched(gs)
    tot = float(np.sum(ms))
    value = len(S) * args.steps / (tot / 1e3)
    line = {"metric": "batched static max-flow solves (64 uneven instances, one persistent launch)",
            "value": value, "unit": "instances/s", "n_gpus": 1, "steps": args.steps, "warmup": args.warmup,
            "ms_per_step": tot / args.steps, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
            "dtype": "int64", "data": "synthetic",
            "config": {"workload": "64 instances, n log-uniform in [1e3, 2e5], ER (avg out-degree 8) / layered DAG "
                                   "(16 layers) / random geometric (avg degree 8), caps U[1,500], seed 4",
                       "vertices_total": int(sum(g.n for g in gs)), "edges_total": int(sum(g.m for g in gs)),
                       "autotuned": {k: (list(v) if isinstance(v, tuple) else v) for k, v in best.items()},
                       "l2": "working set of all instances ~0.3 GB, larger than L2"},
            "one_by_one_ms": float(min(one)), "batched_default_ms": ms_default,
            "speedup_vs_one_by_one": float(min(one)) / (tot / args.steps),
            "mixed_update_1pct": {"updates": n_upd, "ms": upd_ms, "updates_per_s": n_upd / (upd_ms / 1e3)},
            "autotune_trials": len(trials), "gpu_launches": launches, "clocks": clocks,
            "cpu_baseline": {"value": cpu_rate, "unit": "instances/s", "cores": cpu_threads, "kind": "oracle",
                             "sample": f"all {len(gs)} instances, Dinic from scratch, one instance per thread "
                                       f"on a pool of {cpu_threads} threads"},
            "flow_check": {"instances": len(gs), "equal": bool(cpu_vals == ref_values)}}
    print(json.dumps(line), flush=True)
    for s in S:
        s.close()


def _serving_worker(job):
    """One serving graph and its batch sequence (runs in a spawned process, no CUDA)."""
    scale, gseed, sizes, bseed = job
    from paper_2511_01235_gb300 import serving as SV
    from paper_2511_01235_gb300 import workloads as W
    g = W.rmat(scale, 16, 0.57, 0.19, 0.19, seed=gseed, cap_hi=1000)
    return g, SV.graph_batches(g, sizes, bseed)


def step_records(lat_ms, kernel_ms, detail, barriers, alg_bytes, batch: int):
    """One record per timed batch: latency (CUDA events around the call), the
    kernel's own time, updates/s, the solve's counters and the algorithmic
    bytes with their rate.  detail rows: kernel ms, iterations, BFS levels,
    pushes, relabels."""
    out = []
    for k, lt in enumerate(lat_ms):
        row = detail[k]
        km = float(kernel_ms[k])
        out.append({"step": k, "batch": int(batch), "latency_ms": float(lt), "kernel_ms": km,
                    "updates_per_s": batch / (float(lt) / 1e3) if lt > 0 else None,
                    "iterations": int(row[1]), "bfs_levels": int(row[2]), "pushes": int(row[3]),
                    "relabels": int(row[4]), "barriers": int(barriers[k]), "alg_bytes": float(alg_bytes[k]),
                    "alg_gbs": float(alg_bytes[k]) / (km * 1e6) if km > 0 else None})
    return out


def write_jsonl(path: str, records):
    with open(path, "w") as f:
        for r in records:
            f.write(json.dumps(r) + "\n")


def service_time(cal_wall_s: float, cal_sizes, timed_sizes):
    """(calibration mean per request, expected service time of a timed request), in seconds.

    The calibration serves its requests one at a time in cal_wall_s.  A timed
    request is taken to cost the longer of the calibration's mean per request
    and its mean per update times the timed requests' mean size: the
    calibration sample's sizes need not match the timed mix, and the per-request
    mean of a sample of small requests would offer more load than the server
    sustains."""
    per_req = cal_wall_s / max(1, len(cal_sizes))
    per_upd = cal_wall_s / max(1, int(sum(cal_sizes)))
    mean_size = float(np.mean(timed_sizes)) if len(timed_sizes) else 0.0
    return per_req, max(per_req, per_upd * mean_size)


def run_serving(args):
    """Serving: 16 R-MAT graphs (scales 18x4, 19x3, 20x3, 21x3, 22x3) under a device-memory
    budget, Poisson arrivals of mixed batches (sizes log-uniform in [10, 100K]), continuous
    batching.  A step is one request."""
    import multiprocessing as mp
    from paper_2511_01235_gb300 import serving as SV
    ws, rank, _ = dist_env()
    if ws > 1 and rank != 0:
        return
    spec = args.workload.split(":", 1)
    scales = SV.SERVING_SCALES if len(spec) == 1 else tuple(int(x) for x in spec[1].split(","))
    n_cal = max(args.warmup, 1) * len(scales)
    n_req = n_cal + args.steps
    plan = SV.plan_requests(len(scales), n_req, 1.0, seed=77, size_lo=10, size_hi=100_000)
    jobs = [(sc, 10 + k, [b for gi, b, _ in plan if gi == k], (77, k)) for k, sc in enumerate(scales)]
    t0 = time.perf_counter()
    with mp.get_context("spawn").Pool(min(len(jobs), os.cpu_count() or 1)) as pool:   # before any CUDA call
        res = pool.map(_serving_worker, jobs, chunksize=1)
    gen_s = time.perf_counter() - t0
    graphs = [r[0] for r in res]
    reqs = SV.assemble(plan, [r[1] for r in res])
    del res
    import torch
    from paper_2511_01235_gb300 import native
    torch.cuda.set_device(0)
    native.load()
    budget = int(args.budget_gb * 2**30)
    t0 = time.perf_counter()
    srv = SV.Server(graphs, budget, group_blocks=args.group_blocks)
    init_s = time.perf_counter() - t0
    state_gb = sum(srv.bytes) / 2**30
    # warm-up and calibration: the first requests one at a time, all arrived at 0
    cal = reqs[:n_cal]
    for r in cal:
        r.arrival = 0.0
    srv.max_per_tick = 1
    cst = srv.run(cal)
    per_req_s, mean_s = service_time(cst.wall_s, [r.size for r in cal], [r.size for r in reqs[n_cal:]])
    rate = args.utilization / mean_s
    srv.max_per_tick = None
    srv.stats = SV.ServeStats()
    timed = SV.retime(reqs[n_cal:], rate, seed=78)
    clk = ClockSampler(0)
    clk.start()
    l0 = native.kernel_launches()
    st = srv.run(timed)
    launches = native.kernel_launches() - l0
    clocks = clk.stop()
    sm = st.summary()
    # the oracle on the smallest graph's final state; the exact alone-vs-mix check is a GPU test
    import oracle
    g0 = graphs[0]
    es = W_edgeset(g0)
    for r in reqs:
        if r.graph == 0:
            es.apply(r.u, r.v, r.cap)
    u, v, c = es.coo()
    tq = time.perf_counter()
    want = oracle.maxflow(g0.n, u, v, c, g0.s, g0.t).value
    oracle_s = time.perf_counter() - tq
    got = srv.solvers[0].query()[0]
    last0 = [r for r in reqs if r.graph == 0][-1]
    peaks, peak_src = _peaks()
    hbm = float(peaks.get("hbm_gbs", HBM_FALLBACK_GBS))
    line = {"metric": "serving: dynamic maxflow updates/s and p50/p99 request latency (arrival to result)",
            "value": sm["updates_per_s"], "unit": UNIT, "n_gpus": 1, "steps": args.steps, "warmup": args.warmup,
            "ms_per_step": 1e3 * st.wall_s / max(1, st.instances), "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "int64", "data": "synthetic",
            "config": {"workload": f"{len(scales)} R-MAT graphs, scales {list(scales)}, edge factor 16, "
                                   f"a/b/c=0.57/0.19/0.19, caps U[1,1000], seeds 10..{9 + len(scales)}; "
                                   "Poisson arrivals, mixed batches 40/40/10/10, sizes log-uniform in [10, 100K]",
                       "budget_gb": args.budget_gb, "states_gb": state_gb, "rate_per_s": rate,
                       "target_utilization": args.utilization, "group_blocks": args.group_blocks,
                       "l2": "states of several GB, larger than L2"},
            "latency_ms": {"p50": sm["p50_ms"], "p99": sm["p99_ms"], "mean": sm["mean_ms"]},
            "serving": sm, "calibration": {"requests": len(cal), "mean_wall_ms": 1e3 * per_req_s,
                                           "updates": int(sum(r.size for r in cal)),
                                           "service_ms_per_timed_request": 1e3 * mean_s},
            "flow_check": {"graph": 0, "requests": sum(1 for r in reqs if r.graph == 0), "gpu": int(got),
                           "oracle": int(want), "equal": bool(got == want)},
            "gpu_launches": launches,
            "roofline": {"bound": "hbm", "achieved": sm["alg_gbs"], "peak": hbm, "unit": "GB/s",
                         "frac": sm["alg_gbs"] / hbm, "traffic": None, "kernel": "mf_multi_kernel",
                         "peak_source": f"{peak_src} hbm_gbs (copy)",
                         "frac_of_nominal": sm["alg_gbs"] / HBM_NOMINAL_GBS},
            "cpu_baseline": {"value": last0.size / oracle_s, "unit": UNIT, "cores": 1, "kind": "oracle",
                             "sample": f"one request ({last0.size} updates) on graph 0 (scale {scales[0]}): "
                                       "Dinic from scratch on the updated graph, single thread"},
            "e2e": {"value": sm["updates_per_s"], "unit": UNIT,
                    "h2d_bytes_per_step": int(12 * np.mean([r.size for r in timed])), "d2h_bytes_per_step": 8,
                    "note": "serving is end to end: host batches in, values out, arrival to result"},
            "arena": srv.arena.stats() if srv.arena is not None else None,
            "clocks": clocks, "gen_s": gen_s, "init_s": init_s}
    print(json.dumps(line), flush=True)
    srv.close()


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=100)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--batch", type=int, default=10000)
    ap.add_argument("--workload", default="rmat20")
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-configs", action="store_true", help="headline workload only (no configs block)")
    ap.add_argument("--log-jsonl", default=None,
                    help="write one JSON record per timed batch (latency, kernel time, iterations, bytes, GB/s)")
    ap.add_argument("--static-reps", type=int, default=3)
    ap.add_argument("--quick", action="store_true", help="timed steps only (for profiling runs)")
    ap.add_argument("--sched-steps", type=int, default=30, help="held-out batches for the learned-vs-fixed schedule comparison")
    ap.add_argument("--budget-gb", type=float, default=8.0, help="serving: device-memory budget of the states")
    ap.add_argument("--utilization", type=float, default=0.7, help="serving: offered load vs one-at-a-time service")
    ap.add_argument("--group-blocks", type=int, default=8, help="serving: CTAs per instance in a launch")
    args = ap.parse_args()
    if args.impl == "reference":
        return run_reference(args)
    if args.gpus > 1 and "WORLD_SIZE" not in os.environ:
        return launch_replicas(sys.argv[1:], args.gpus)
    if args.workload == "batched64":
        return run_batched(args)
    if args.workload.startswith("serving"):
        return run_serving(args)

    import torch
    from paper_2511_01235_gb300 import native

    ws, rank, local = dist_env()
    if ws != args.gpus:
        sys.stderr.write(f"bench.py: --gpus {args.gpus} but WORLD_SIZE is {ws}\n")
        return 2
    if ws > 1:
        import torch.distributed as dist
        torch.cuda.set_device(local)
        dist.init_process_group("nccl")
    else:
        torch.cuda.set_device(0)
    dev = torch.cuda.current_device()
    native.load()

    wl = Workload(args)
    g = wl.g
    nb = args.warmup + args.steps
    batches = wl.batches(nb, args.batch)
    args.batch = batches[0].size
    dev_batches = [(torch.from_numpy(b.u).cuda(), torch.from_numpy(b.v).cuda(), torch.from_numpy(b.cap).cuda())
                   for b in batches]
    stream = torch.cuda.current_stream()
    t0 = time.perf_counter()
    S = native.Solver(g.n, g.src, g.dst, g.cap, g.s, g.t, stream=stream)
    init_s = time.perf_counter() - t0
    static_value = S.query()[0]

    # ---- device-resident timed region ----
    for i in range(args.warmup):
        S.update(*dev_batches[i])
    torch.cuda.synchronize()
    if ws > 1:
        torch.distributed.barrier()
    clk = ClockSampler(dev)
    clk.start()
    evs = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(args.steps)]
    lat = []
    kbytes, kms, detail, barriers, phase_tot = [], [], [], [], {}
    torch.cuda.synchronize()
    l0 = native.kernel_launches()
    t_wall = time.perf_counter()
    for k in range(args.steps):
        a, b = evs[k]
        a.record(stream)
        S.update(*dev_batches[args.warmup + k])
        b.record(stream)
        st = S.stats()
        for ph, bk, mk in (("bfs", "bytes_bfs", "ms_bfs"), ("discharge", "bytes_discharge", "ms_discharge"),
                           ("fix", "bytes_fix", "ms_fix"), ("apply", "bytes_apply", "ms_apply")):
            t = phase_tot.setdefault(ph, [0.0, 0.0])
            t[0] += st[bk]
            t[1] += st[mk]
        barriers.append(st["barriers"])
        kbytes.append(st["bytes_bfs"] + st["bytes_discharge"] + st["bytes_fix"] + st["bytes_worklist"]
                      + st["bytes_apply"])
        kms.append(st["ms_last"])
        detail.append([round(st["ms_last"], 3), st["iterations"], st["bfs_levels"], st["pushes"], st["relabels"]])
    torch.cuda.synchronize()
    wall = time.perf_counter() - t_wall
    launches = native.kernel_launches() - l0
    clocks = clk.stop()
    lat = np.array([a.elapsed_time(b) for a, b in evs])
    if args.log_jsonl and rank == 0:
        write_jsonl(args.log_jsonl, step_records(lat, kms, detail, barriers, kbytes, args.batch))
    tot_ms = float(lat.sum())
    value, tot_ms, _ = aggregate_over_ranks(tot_ms, args.batch * args.steps, device="cuda" if ws > 1 else None)
    final_value = S.query()[0]
    last_stats = S.stats()

    if args.quick:
        args.no_cpu_baseline = True
        args.static_reps = 0
    # ---- end-to-end through the public API with host buffers ----
    e2e_b = wl.batches(0 if args.quick else min(args.steps, 10), args.batch)
    pinned = []
    for b in e2e_b:
        tu = torch.from_numpy(b.u).pin_memory()
        tv = torch.from_numpy(b.v).pin_memory()
        tc = torch.from_numpy(b.cap).pin_memory()
        pinned.append((tu, tv, tc))
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    for tu, tv, tc in pinned:
        native.maxflow_update(S.h, tu.numpy(), tv.numpy(), tc.numpy())
        native.maxflow_query(S.h, S.n)
    e2e_s = time.perf_counter() - t0
    e2e_val = ws * args.batch * len(pinned) / e2e_s if pinned else None
    es_state = wl.es.copy()            # the graph S holds now (the comparisons below run on clones)

    # ---- learned schedule vs the fixed ones on one held-out stream of mixed sizes (clones of one state) ----
    sched = None
    if not args.quick and args.sched_steps > 0:
        sched = scheduler_comparison(S, wl, args.sched_steps)

    # ---- dynamic push-pull (Sec. 5.2.2, O2) vs the default update, same batches on clones ----
    pushpull = None
    if not args.quick and args.sched_steps > 0:
        pb = wl.batches(min(args.sched_steps, 4), args.batch)
        pushpull = {}
        for key in ("update", "push_pull"):
            C = S.clone()
            dms = []
            for b in pb:
                (C.update if key == "update" else C.update_pp)(b.u, b.v, b.cap)
                dms.append(C.stats()["ms_update"])
            pushpull[key + "_device_ms_mean"] = float(np.mean(dms))
            pushpull[key + "_value"] = int(C.query()[0])
            C.close()
        pushpull["batches"] = len(pb)

    # ---- static re-solve comparator (same updated graph) ----
    static_ms = []
    for _ in range(args.static_reps):
        S.resolve_static()
        static_ms.append(S.stats()["ms_last"])
    static_stats = S.stats()

    peaks, peak_src = _peaks()
    hbm = float(peaks.get("hbm_gbs", HBM_FALLBACK_GBS))
    configs = None
    if ws == 1 and not args.quick and not args.no_configs:
        configs = run_configs(S, es_state, hbm)
    if rank == 0:
        avg_bytes = float(np.mean(kbytes))
        avg_ms = float(np.mean(kms))
        achieved = avg_bytes / (avg_ms * 1e-3) / 1e9 if avg_ms > 0 else 0.0
        cpu = None
        if not args.no_cpu_baseline and ws == 1:
            times = cpu_baseline_sample(g, batches[: 8])
            cpu = {"value": args.batch * len(times) / sum(times), "unit": UNIT, "cores": 1, "kind": "oracle",
                   "sample": f"{len(times)} batches of {args.batch} on {os.cpu_count()} host cores "
                             f"(Dinic recomputed from scratch per batch, single thread)"}
        p50 = float(np.percentile(lat, 50))
        p99 = float(np.percentile(lat, 99))
        kp50 = float(np.percentile(kms, 50))
        line = {
            "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": ws, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": tot_ms / args.steps, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "int64", "data": "synthetic",
            "config": config_of(args, g, wl, ws),
            "latency_ms": {"p50": p50, "p99": p99, "mean": float(lat.mean())},
            "kernel_ms": {"p50": kp50, "mean": float(np.mean(kms))},
            "static_resolve_ms": float(np.median(static_ms)) if static_ms else None,
            # both sides device time of the solve kernel (the latency above also holds the call's host work)
            "speedup_vs_static": float(np.median(static_ms)) / kp50 if static_ms and kp50 > 0 else None,
            "flow_value": {"static": int(static_value), "final": int(final_value)},
            "init_s": init_s,
            "gpu_launches": launches,
            "roofline": {"bound": "hbm", "achieved": achieved, "peak": hbm, "unit": "GB/s",
                         "frac": achieved / hbm, "traffic": measured_traffic(args.workload, args.batch),
                         "kernel": "mf_solve_kernel", "peak_source": f"{peak_src} hbm_gbs (copy)",
                         "algorithmic_bytes_per_launch": avg_bytes, "avg_launch_ms": avg_ms,
                         "frac_of_nominal": achieved / HBM_NOMINAL_GBS,
                         "phases": phase_roofline(phase_tot, hbm)},
            "barriers_per_update": float(np.mean(barriers)),
            "configs": configs,
            "cpu_baseline": cpu,
            "e2e": {"value": e2e_val, "unit": UNIT, "h2d_bytes_per_step": 12 * args.batch,
                    "d2h_bytes_per_step": 2048 + 8},
            "clocks": clocks,
            "last_update_stats": {k: last_stats[k] for k in ("iterations", "bfs_levels", "pushes", "relabels",
                                                             "steep_fixes", "active_first", "ms_bfs", "ms_discharge",
                                                             "ms_fix", "ms_worklist", "ms_apply", "grid_blocks",
                                                             "kernel_cycles")},
            "scheduler": sched,
            "push_pull": pushpull,
            "static_stats": {k: static_stats[k] for k in ("iterations", "bfs_levels", "pushes", "relabels",
                                                          "ms_bfs", "ms_discharge", "ms_fix", "ms_worklist")},
            "wall_s_timed": wall,
            "steps_detail": {"cols": ["kernel_ms", "iterations", "bfs_levels", "pushes", "relabels"],
                             "rows": detail},
        }
        print(json.dumps(line), flush=True)
    S.close()
    if ws > 1:
        torch.distributed.destroy_process_group()


if __name__ == "__main__":
    sys.exit(main() or 0)
