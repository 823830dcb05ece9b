"""Benchmark of the lattice Boltzmann hot path on GB300.

Workload: the porous-medium lattice of the paper's method (1024 x 1024,
random discs at porosity 0.7, Zou-He density inlet 1.001 / outlet 1.0,
tau = 0.8, periodic in y), FP32 population storage.  A step is one
iteration of the update through the C ABI (lb_iteration(ctx, 1)); thermo
runs every 100 iterations as in the paper's scripts.

value: MLUPS over all nodes, whole job, inputs resident in HBM; the L2 is
flushed (a write of a buffer twice its size, then a read of another) before
every timed step and each step is timed by CUDA events on the library's
stream.  e2e: the same metric through the public API with host buffers:
every step uploads the state snapshot from pinned memory, iterates once
(producing the node fields, output command) and downloads density and
velocity to pinned memory; two contexts on two streams take alternate steps
so that one step's upload overlaps the other's download (the one-context
rate is reported beside it).
--impl reference times the FP64 CPU oracle on the same workload.

Multi-GPU (torchrun), --mode:
  replicas (default): every rank advances its own replica of the lattice
    (independent units, no collective on the data path): weak scaling;
  split: the lattice is split into N y slabs (processors command), one per
    rank, with a halo exchange over NCCL after every iteration: strong
    scaling of the one lattice;
  batch: the 256 lattices of the batched workload are shared out over the
    ranks by longest-processing-time bin packing (node counts), each rank
    advancing its share in one launch per iteration: strong scaling.
"""
from __future__ import annotations

import argparse
import hashlib
import json
import os
import subprocess
import sys
import threading
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "D2Q9 MLUPS and % of HBM roofline; 16-bit-storage & batched vs plain FP32 at ≤1e-5"
WORKLOAD = "porous 1024x1024 (random discs r 8-24 seed 1, porosity 0.7, Zou-He rho 1.001/1.0, tau 0.8)"
BYTES_PER_FLUID_NODE = {"fp32": 72, "fp16": 36, "bf16": 36}
THERMO_EVERY = 100  # iterations between two thermo records of the timed run
# measured against the FP64 oracle on this workload after its stated 10 000
# iterations (tests/long_parity.py); the target for 16-bit storage is 2e-3
ACCURACY_16 = {"fp16": "rel. u 7.3e-4 after 10 000 iterations: meets 2e-3",
               "bf16": "rel. u 6.4e-3 after 10 000 iterations: misses 2e-3 (8-bit significand)"}


def peaks():
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as fh:
            d = json.load(fh)
        return float(d["hbm_gbs"]), "measured"
    except Exception:
        return 6800.0, "fallback"


def kernel_source_hash() -> str:
    """Hash of the code (line comments and blank lines dropped) of the
    sources the streaming kernel is compiled from."""
    h = hashlib.sha256()
    for name in ("k_fluid.cu", "lbarith.cuh", "lbcollide.cuh", "lbdev.cuh", "lbint.h", "lbpdl.cuh", "lbsolute.cuh"):
        with open(os.path.join(ROOT, "paper_1202_0442_gb300", "csrc", name)) as fh:
            for line in fh:
                code = line.split("//", 1)[0].rstrip()
                if code:
                    h.update(code.encode() + b"\n")
    return h.hexdigest()[:16]


def recorded_traffic(kernel: str, storage: str, workload: str):
    """DRAM bytes (read + write) of one launch of the fused kernel on this
    workload, from the committed ncu capture (profiles/traffic.json); None
    when there is none or it was taken on different kernel source."""
    path = os.path.join(ROOT, "profiles", "traffic.json")
    try:
        with open(path) as fh:
            d = json.load(fh)
    except Exception:
        return None
    e = d.get(f"{kernel}/{storage}@{workload}")
    if not e or e.get("source_hash") != kernel_source_hash():
        return None
    return e["dram_bytes_read"] + e["dram_bytes_write"]


class ClockSampler:
    """nvidia-smi clocks and throttle reasons during the timed region."""
    Q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
         "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
         "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, index: int):
        self.index = index
        self.proc = None
        self.lines = []

    def start(self):
        try:
            self.proc = subprocess.Popen(["nvidia-smi", f"--query-gpu={self.Q}", "--format=csv,noheader,nounits",
                                          "-i", str(self.index), "-lms", "100"],
                                         stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.t = threading.Thread(target=self._read, daemon=True)
            self.t.start()
            # the timed region is short: let the first sample land before it
            t0 = time.time()
            while not self.lines and time.time() - t0 < 2.0:
                time.sleep(0.01)
            self.n0 = len(self.lines)
        except Exception:
            self.proc = None

    def _read(self):
        for line in self.proc.stdout:
            self.lines.append(line.strip())

    def stop(self):
        if not self.proc:
            return None
        # and one more right after it
        try:
            one = subprocess.run(["nvidia-smi", f"--query-gpu={self.Q}", "--format=csv,noheader,nounits",
                                  "-i", str(self.index)], capture_output=True, text=True, timeout=10)
            self.lines.extend(x.strip() for x in one.stdout.splitlines() if x.strip())
        except Exception:
            pass
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except Exception:
            self.proc.kill()
        self.t.join(timeout=2)
        sm, mx, reasons = [], None, set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for ln in self.lines:
            p = [x.strip() for x in ln.split(",")]
            if len(p) < 9:
                continue
            try:
                sm.append(float(p[1]))
                mx = float(p[2])
            except ValueError:
                continue
            for k, nm in enumerate(names):
                if p[5 + k].lower().startswith("active"):
                    reasons.add(nm)
        if not sm:
            return None
        return {"sm_mhz": float(np.median(sm)), "sm_max_mhz": mx, "reasons": sorted(reasons),
                "samples": len(sm)}


class NvmlSampler:
    """SM clock and clock-event reasons read through NVML (ctypes, read-only
    queries) every 2 ms on a thread while the timed region runs; the
    GPU is found by its PCI address, so the CUDA and NVML numberings need
    not agree."""
    # clock-event reason bits of the NVML API
    REASONS = {0x4: "sw_power_cap", 0x8: "hw_slowdown", 0x20: "sw_thermal_slowdown",
               0x40: "hw_thermal_slowdown", 0x80: "hw_power_brake_slowdown"}

    def __init__(self, device: int):
        import ctypes
        import torch
        self.C = ctypes
        self.nv = ctypes.CDLL("libnvidia-ml.so.1")
        if self.nv.nvmlInit_v2() != 0:
            raise RuntimeError("nvmlInit failed")
        pr = torch.cuda.get_device_properties(device)
        bus = f"{pr.pci_domain_id:08x}:{pr.pci_bus_id:02x}:{pr.pci_device_id:02x}.0".encode()
        self.h = ctypes.c_void_p()
        if self.nv.nvmlDeviceGetHandleByPciBusId_v2(bus, ctypes.byref(self.h)) != 0:
            raise RuntimeError("no NVML handle for " + bus.decode())
        self.reasons_fn = getattr(self.nv, "nvmlDeviceGetCurrentClocksEventReasons", None) or \
            self.nv.nvmlDeviceGetCurrentClocksThrottleReasons
        mx = ctypes.c_uint()
        self.nv.nvmlDeviceGetMaxClockInfo(self.h, 1, ctypes.byref(mx))  # NVML_CLOCK_SM
        self.max_mhz = float(mx.value)
        self.samples = []
        self.run = False
        self._one()  # fails here, not in the thread, if a query is refused

    def _one(self):
        C = self.C
        mhz, rs = C.c_uint(), C.c_ulonglong()
        if self.nv.nvmlDeviceGetClockInfo(self.h, 1, C.byref(mhz)) != 0:
            raise RuntimeError("clock query failed")
        self.reasons_fn(self.h, C.byref(rs))
        self.samples.append((float(mhz.value), int(rs.value)))

    def _loop(self):
        while self.run:
            try:
                self._one()
            except Exception:
                return
            time.sleep(0.002)

    def start(self):
        self.samples = []
        self.run = True
        self.t = threading.Thread(target=self._loop, daemon=True)
        self.t.start()
        t0 = time.time()
        while not self.samples and time.time() - t0 < 1.0:
            time.sleep(0.0005)

    def stop(self):
        self.run = False
        self.t.join(timeout=2)
        try:
            self._one()
        except Exception:
            pass
        self.nv.nvmlShutdown()
        if not self.samples:
            return None
        reasons = sorted({nm for _, r in self.samples for bit, nm in self.REASONS.items() if r & bit})
        return {"sm_mhz": float(np.median([m for m, _ in self.samples])), "sm_max_mhz": self.max_mhz,
                "reasons": reasons, "samples": len(self.samples), "source": "nvml, every 2 ms"}


def clock_sampler(device: int):
    """NVML sampler where the driver's library loads, else nvidia-smi."""
    try:
        return NvmlSampler(device)
    except Exception:
        return ClockSampler(device)


def dist_setup(args):
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    if world > 1:
        import torch
        import torch.distributed as dist
        backend = "nccl" if torch.cuda.is_available() else "gloo"
        if torch.cuda.is_available():
            torch.cuda.set_device(local)
        dist.init_process_group(backend)
        return world, rank, local, dist
    return 1, 0, 0, None


def max_over_ranks(x: float, dist, world: int) -> float:
    if dist is None or world == 1:
        return x
    import torch
    dev = torch.device("cuda", torch.cuda.current_device()) if torch.cuda.is_available() else torch.device("cpu")
    t = torch.tensor([x], dtype=torch.float64, device=dev)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def lpt_partition(sizes, nbins: int):
    """Longest-processing-time bin packing: items (by size, largest first)
    go to the bin with the least load so far; returns the item indices of
    each bin.  Its largest load is at most 4/3 of the best possible."""
    bins = [[] for _ in range(nbins)]
    load = [0] * nbins
    for k in sorted(range(len(sizes)), key=lambda k: (-sizes[k], k)):
        b = min(range(nbins), key=lambda j: (load[j], j))
        bins[b].append(k)
        load[b] += sizes[k]
    return bins


def run_split(args, world, rank, local, dist):
    """One lattice in `world` y slabs, one per rank, halo rows exchanged
    over NCCL after every iteration; value = the lattice's nodes per
    max-over-ranks step time (strong scaling)."""
    import torch
    from paper_1202_0442_gb300 import build, halo, lb2d, synth
    torch.cuda.set_device(local)
    if local == 0:
        build.build()
    if dist is not None:
        dist.barrier()
    dev = torch.device("cuda", local)
    stream = torch.cuda.current_stream(dev)
    w = synth.porous()
    lt = lb2d.from_workload(w, args.storage, h_max=2e-3, device=local, stream=stream.cuda_stream,
                            slab=(world, rank))
    lt.thermo(1 << 30)
    ex = halo.SlabExchange(lt, dist, rank, world, dev)
    l2 = torch.cuda.get_device_properties(dev).L2_cache_size
    flush_w = torch.empty(2 * l2 // 4, dtype=torch.float32, device=dev)
    flush_r = torch.ones(2 * l2 // 4, dtype=torch.float32, device=dev)
    sink = torch.zeros(1, dtype=torch.float32, device=dev)

    def step():
        lt.iteration(1)
        # one rank: the single slab refills its own ghost rows inside the
        # iteration (it is its own neighbour)
        if world > 1:
            ex()

    for _ in range(args.warmup):
        step()
    torch.cuda.synchronize()
    if dist is not None:
        dist.barrier()
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    tot = 0.0
    for _ in range(args.steps):
        flush_w.fill_(1.0)
        sink.add_(flush_r.sum())
        a.record(stream)
        step()
        b.record(stream)
        torch.cuda.synchronize()
        tot += a.elapsed_time(b)
    ms = max_over_ranks(tot / args.steps, dist, world)
    if rank == 0:
        print(json.dumps({
            "metric": METRIC, "value": w.nodes / (ms * 1e-3) / 1e6, "unit": "MLUPS", "n_gpus": world,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": ms, "higher_is_better": True,
            "scaling": "strong", "vs_baseline": None, "dtype": "f32" if args.storage == "fp32" else args.storage,
            "data": "synthetic",
            "config": {"workload": WORKLOAD, "mode": "split", "parallelism": f"{world} y slabs",
                       "halo_bytes_per_rank_step": ex.bytes_per_iteration if world > 1 else 0,
                       "l2": "flushed before every timed step"}}), flush=True)
    return 0


def run_batch_split(args, world, rank, local, dist):
    """The 256-lattice batch shared out over the ranks by LPT bin packing of
    the node counts; each rank advances its share in one persistent launch
    per iteration (graph-captured); value = all nodes per max-over-ranks
    iteration time (strong scaling)."""
    import torch
    from paper_1202_0442_gb300 import build, lb2d, synth
    torch.cuda.set_device(local)
    if local == 0:
        build.build()
    if dist is not None:
        dist.barrier()
    dev = torch.device("cuda", local)
    stream = torch.cuda.current_stream(dev)
    ws = synth.batch()
    share = lpt_partition([x.nodes for x in ws], world)[rank]
    kw = {"h_max": 5e-3, "rounding": "stochastic"} if args.storage != "fp32" else {"precise": True}
    lats = [lb2d.from_workload(ws[k], args.storage, device=local, stream=stream.cuda_stream, **kw) for k in share]
    for x in lats:
        x.thermo(1 << 30)
    bt = lb2d.Batch(lats)
    bt.autotune(None)
    bt.iteration(max(args.warmup, 20), use_graph=True)
    torch.cuda.synchronize()
    if dist is not None:
        dist.barrier()
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    a.record(stream)
    bt.iteration(args.steps, use_graph=True)
    b.record(stream)
    torch.cuda.synchronize()
    ms = max_over_ranks(a.elapsed_time(b) / args.steps, dist, world)
    nodes = sum(x.nodes for x in ws)
    if rank == 0:
        print(json.dumps({
            "metric": METRIC, "value": nodes / (ms * 1e-3) / 1e6, "unit": "MLUPS", "n_gpus": world,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": ms, "higher_is_better": True,
            "scaling": "strong", "vs_baseline": None, "dtype": "f32" if args.storage == "fp32" else args.storage,
            "data": "synthetic",
            "config": {"workload": f"{len(ws)} periodic porous lattices, sides 64-512 ({nodes} nodes)",
                       "mode": "batch", "parallelism": f"LPT bin packing over {world} ranks",
                       "nodes_rank0": sum(ws[k].nodes for k in share),
                       "l2": "state 1.4 GB > L2, iterations back to back"}}), flush=True)
    return 0


def oracle_rate(w, seconds: float, max_steps: int):
    """Time the FP64 oracle on workload w: single-threaded MLUPS."""
    from oracle.drive import oracle_from_workload
    o = oracle_from_workload(w)
    t0 = time.perf_counter()
    o.step(1)
    one = time.perf_counter() - t0
    n = int(max(1, min(max_steps, seconds / max(one, 1e-9))))
    t0 = time.perf_counter()
    o.step(n)
    dt = time.perf_counter() - t0
    return w.nodes * n / dt / 1e6, n, dt


def run_reference(args, world, rank, dist):
    from paper_1202_0442_gb300 import synth
    if rank != 0:
        return 0
    w = synth.porous()
    from oracle.drive import oracle_from_workload
    o = oracle_from_workload(w)
    o.step(args.warmup)
    t0 = time.perf_counter()
    o.step(args.steps)
    dt = time.perf_counter() - t0
    v = w.nodes * args.steps / dt / 1e6
    line = {"impl": "reference", "metric": METRIC, "value": v, "unit": "MLUPS", "n_gpus": args.gpus,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": dt * 1e3 / args.steps,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
            "data": "synthetic", "config": {"workload": WORKLOAD, "impl": "FP64 CPU oracle (single thread)"},
            "cpu_baseline": {"value": v, "unit": "MLUPS", "cores": 1, "kind": "oracle",
                             "sample": f"full 1024x1024 lattice, {args.steps} timed iterations"},
            "e2e": {"value": v, "unit": "MLUPS", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)
    return 0


def time_steps(lt, steps, flush, stream):
    """Per-step CUDA-event times (ms) of lt.iteration(1), L2 flushed before
    each step."""
    import torch
    ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(steps)]
    for k in range(steps):
        flush()
        ev[k][0].record(stream)
        lt.iteration(1)
        ev[k][1].record(stream)
    torch.cuda.synchronize()
    return np.array([a.elapsed_time(b) for a, b in ev])


def variants(args, local, stream, flush, value_fp32):
    """16-bit storage on the same workload, and the 256-lattice batch in one
    launch per two iterations against one launch per lattice and iteration."""
    import torch
    from paper_1202_0442_gb300 import lb2d, synth
    out = {}
    w = synth.porous()
    for st in ("fp16", "bf16"):
        lt = lb2d.from_workload(w, st, h_max=2e-3, device=local, stream=stream.cuda_stream,
                                rounding="stochastic")
        lt.thermo(100)
        time_steps(lt, 5, flush, stream)
        t = time_steps(lt, min(args.steps, 60), flush, stream)
        v = w.nodes / (t.mean() * 1e-3) / 1e6
        out[st] = {"value": v, "unit": "MLUPS", "speedup_vs_fp32": v / value_fp32,
                   "rounding": "stochastic", "accuracy": ACCURACY_16[st],
                   "kernel_ms": float(np.median(t))}
        del lt
    # the benchmark lattice with iterations back to back, as a run of the
    # method executes them: the 75 MB state stays in L2 between iterations
    # and consecutive launches overlap (programmatic dependent launch), so
    # this is the production rate, not a DRAM roofline figure
    lt = lb2d.from_workload(w, "fp32", device=local, stream=stream.cuda_stream)
    lt.thermo(1 << 30)
    lt.iteration(20)
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    n = 400
    a.record(stream)
    lt.iteration(n)
    b.record(stream)
    torch.cuda.synchronize()
    ms = a.elapsed_time(b) / n
    out["porous_1024_back_to_back"] = {
        "workload": "porous 1024x1024 (the benchmark lattice), 400 iterations in one call",
        "l2": "state 75 MB stays L2-resident between iterations: not a DRAM roofline figure",
        "value": w.nodes / (ms * 1e-3) / 1e6, "unit": "MLUPS", "ms_per_step": ms}
    del lt
    # the same recipe at 4096^2 (1.2 GB of FP32 state, far beyond L2, so
    # back-to-back steps need no flush): where the memory system, not the
    # launch, sets the time
    peak = peaks()[0]
    w4 = synth.porous(4096, 4096, seed=1)
    big = {"workload": "porous 4096x4096 (same recipe, seed 1)", "l2": "state 1.2 GB > L2, steps back to back"}
    for st, kw in (("fp32", {}), ("fp16", {"h_max": 2e-3, "rounding": "stochastic"})):
        lt = lb2d.from_workload(w4, st, device=local, stream=stream.cuda_stream, **kw)
        lt.thermo(1 << 30)
        lt.iteration(5)
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        n = 50
        a.record(stream)
        lt.iteration(n)
        b.record(stream)
        torch.cuda.synchronize()
        ms = a.elapsed_time(b) / n
        big[st] = {"value": w4.nodes / (ms * 1e-3) / 1e6, "unit": "MLUPS", "ms_per_step": ms,
                   # a launch reads and writes the state once for two iterations
                   "bytes_all_nodes_frac": BYTES_PER_FLUID_NODE[st] / 2 * w4.nodes / (ms * 1e-3) / 1e9 / peak}
        del lt
    big["fp16_speedup_vs_fp32"] = big["fp16"]["value"] / big["fp32"]["value"]
    out["porous_4096"] = big
    # 256 periodic porous lattices, sides 64..512, in one launch per two
    # iterations against one launch per lattice and iteration, FP32 and FP16
    ws = synth.batch()
    nodes = sum(x.nodes for x in ws)
    fluid = sum(x.fluid_nodes for x in ws)
    peak = peaks()[0]
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    for st in ("fp32", "fp16"):
        # FP32 with the exact momentum pair, which keeps the slowest lattices
        # within 1e-5 of the oracle in u at 5000 iterations
        kw = {"h_max": 5e-3, "rounding": "stochastic"} if st != "fp32" else {"precise": True}
        lats = [lb2d.from_workload(x, st, device=local, stream=stream.cuda_stream, **kw) for x in ws]
        for lt in lats:
            lt.thermo(1 << 30)
        b = lb2d.Batch(lats)
        b.autotune(None)
        b.iteration(20, use_graph=True)
        torch.cuda.synchronize()
        n = 100
        e0.record(stream)
        b.iteration(n, use_graph=True)
        e1.record(stream)
        torch.cuda.synchronize()
        ms_b = e0.elapsed_time(e1) / n
        for lt in lats:
            lt.iteration(2)
        torch.cuda.synchronize()
        m = 10
        e0.record(stream)
        for _ in range(m):
            for lt in lats:
                lt.iteration(1)
        e1.record(stream)
        torch.cuda.synchronize()
        ms_s = e0.elapsed_time(e1) / m
        bpn = BYTES_PER_FLUID_NODE[st]
        out["batched" if st == "fp32" else "batched_fp16"] = {
            "workload": f"{len(ws)} periodic porous lattices, sides 64-512 step 32, "
                        f"porosity 0.4-0.9, tau 0.6-1.5 ({nodes} nodes, {fluid} fluid)",
            "storage": st + (" + precise momentum" if st == "fp32" else " stochastic"),
            "mlups_one_launch": nodes / (ms_b * 1e-3) / 1e6,
            "mlups_one_launch_per_lattice": nodes / (ms_s * 1e-3) / 1e6,
            "speedup": ms_s / ms_b, "ms_per_iteration_batched": ms_b,
            "ms_per_iteration_per_lattice": ms_s, "graph": True,
            # two iterations per launch: half the bytes per iteration
            "roofline_frac": bpn / 2 * fluid / (ms_b * 1e-3) / 1e9 / peak,
            "state_bytes": int(2 * bpn * nodes),
            "accuracy": ("rel. u <= 2.5e-6 on 8 sampled lattices after 5000 iterations (exact momentum pairs): meets 1e-5"
                         if st == "fp32" else
                         "rel. u up to 1.2e-2 on 8 sampled lattices after 5000 iterations: "
                         "misses 2e-3 on the slow ones")}
        del b, lats
    out["batched_fp16"]["speedup_vs_fp32_batched"] = (out["batched"]["ms_per_iteration_batched"]
                                                     / out["batched_fp16"]["ms_per_iteration_batched"])
    # config 3: two components with interforce and adhesion, 2048^2
    w3 = synth.shan_chen2(2048)
    lt = lb2d.from_workload(w3, "fp32", device=local, stream=stream.cuda_stream)
    lt.thermo(1 << 30)
    time_steps(lt, 5, flush, stream)
    t = time_steps(lt, min(args.steps, 40), flush, stream)
    ms = float(t.mean())
    out["shan_chen2_2048"] = {
        "workload": "2048^2 periodic, two components, interforce G = 0.9, adhesive ring +-0.3",
        "kernel": "k_fluid_sc2", "value": w3.nodes / (ms * 1e-3) / 1e6, "unit": "MLUPS",
        "ms_per_step": ms, "bytes_per_fluid_node": 144,
        "roofline_frac": 144 * w3.fluid_nodes / (ms * 1e-3) / 1e9 / peak}
    del lt
    # config 4: fluid + D2Q9 solute + reaction + growth, 1024 x 512
    w4 = synth.reactive()
    lt = lb2d.from_workload(w4, "fp32", device=local, stream=stream.cuda_stream)
    lt.thermo(1 << 30)
    time_steps(lt, 5, flush, stream)
    t = time_steps(lt, min(args.steps, 40), flush, stream)
    ms = float(t.mean())
    out["reactive_1024x512_q9"] = {
        "workload": "1024 x 512 channel, 40 discs, velocity inlet 0.02, D2Q9 solute, reaction and growth",
        "kernels": "k_fluid_solute<9> (fluid and solute fused) + k_grow_list (gather, decisions and flips over the surface list)",
        "value": w4.nodes / (ms * 1e-3) / 1e6, "unit": "MLUPS", "ms_per_step": ms,
        # 72 B fluid + 72 B D2Q9 solute; the fused kernel keeps the solvent
        # velocity (16 B of the unfused path) in registers
        "bytes_per_fluid_node": 144,
        "roofline_frac": 144 * w4.fluid_nodes / (ms * 1e-3) / 1e9 / peak}
    del lt
    return out


def run_gb300(args, world, rank, local, dist):
    import torch
    from paper_1202_0442_gb300 import build, lb2d, synth

    if not torch.cuda.is_available():
        raise SystemExit("bench.py needs a CUDA device (the library has no CPU path)")
    torch.cuda.set_device(local)
    if local == 0:
        build.build()
    if dist is not None:
        dist.barrier()
    dev = torch.device("cuda", local)
    stream = torch.cuda.current_stream(dev)

    w = synth.porous()
    storage = args.storage
    lt = lb2d.from_workload(w, storage, h_max=2e-3, device=local, stream=stream.cuda_stream)
    lt.thermo(THERMO_EVERY)
    # the thermo record of every THERMO_EVERY-th step is copied to the host inside
    # that step and read by the next thermo evaluation, so the host keeps
    # the stream fed
    lt.thermo_deferred(True)
    nodes, fluid = w.nodes, w.fluid_nodes

    l2 = torch.cuda.get_device_properties(dev).L2_cache_size
    flush_w = torch.empty(2 * l2 // 4, dtype=torch.float32, device=dev)
    flush_r = torch.ones(2 * l2 // 4, dtype=torch.float32, device=dev)
    sink = torch.zeros(1, dtype=torch.float32, device=dev)

    def flush():
        flush_w.fill_(1.0)
        sink.add_(flush_r.sum())

    for _ in range(args.warmup):
        flush()
        lt.iteration(1)
    torch.cuda.synchronize()

    ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(args.steps)]
    thermo_step = []
    sampler = clock_sampler(local) if local == 0 else None
    if dist is not None:
        dist.barrier()
    torch.cuda.synchronize()
    if sampler:
        sampler.start()
    launches0 = lt.launch_count()
    t_start = time.perf_counter()
    for k in range(args.steps):
        flush()
        ev[k][0].record(stream)
        lt.iteration(1)
        ev[k][1].record(stream)
    torch.cuda.synchronize()
    wall = time.perf_counter() - t_start
    launches = lt.launch_count() - launches0
    # reads the last deferred record (raises on a non-finite sum), if the run
    # has reached a thermo step
    last_thermo = lt.get_thermo() if args.warmup + args.steps >= THERMO_EVERY else None
    if dist is not None:
        dist.barrier()
    clocks = sampler.stop() if sampler else None
    for k in range(args.steps):
        step_no = args.warmup + k + 1
        thermo_step.append(step_no % THERMO_EVERY == 0)
    times = np.array([a.elapsed_time(b) for a, b in ev])
    ms_step = float(times.mean())
    plain = times[~np.array(thermo_step)] if (~np.array(thermo_step)).any() else times
    kernel_ms = float(np.median(plain))
    ms_step = max_over_ranks(ms_step, dist, world)
    value = world * nodes / (ms_step * 1e-3) / 1e6

    # e2e through the public API with pinned host buffers: every step uploads
    # a state snapshot, iterates once (output command: fresh node fields, no
    # thermo sums) and downloads density and velocity.  Two contexts on two
    # streams, each driven by its own host thread (the library releases the
    # GIL inside its calls), take alternate steps, so that one step's upload
    # overlaps the other's download and compute; the one-context figure is
    # reported beside it.
    import threading
    size = lt.state_size()
    stream2 = torch.cuda.Stream(dev)  # outlives the second context
    pair = [lt, lb2d.from_workload(w, storage, h_max=2e-3, device=local, stream=stream2.cuda_stream)]
    snaps, outs = [], []
    for x in pair:
        snaps.append(torch.empty(size, dtype=torch.uint8, pin_memory=True))
        x.save_state(snaps[-1])
        outs.append(tuple(torch.empty((w.ny, w.nx), dtype=torch.float32, pin_memory=True) for _ in range(3)))
        x.thermo(1 << 30)
        x.output(1)

    def e2e_steps(i, n):
        for _ in range(n):
            pair[i].load_state(snaps[i])
            pair[i].iteration(1)
            pair[i].velocity_f32(outs[i])

    for i in range(2):
        e2e_steps(i, 2)
    ke = 2 * max(2, min(args.steps, 20) // 2)
    e2e_vals = {}
    for label, nctx in (("one_context", 1), ("two_contexts", 2)):
        if dist is not None:
            dist.barrier()
        torch.cuda.synchronize()
        th = [threading.Thread(target=e2e_steps, args=(i, ke // nctx)) for i in range(nctx)]
        t0e = time.perf_counter()
        for t in th:
            t.start()
        for t in th:
            t.join()
        torch.cuda.synchronize()
        e2e_vals[label] = max_over_ranks((time.perf_counter() - t0e) / ke, dist, world)
    e2e_s = e2e_vals["two_contexts"]
    e2e = {"value": world * nodes / e2e_s / 1e6, "unit": "MLUPS", "h2d_bytes_per_step": int(size),
           "d2h_bytes_per_step": int(3 * 4 * nodes), "steps": ke,
           "how": "two contexts on two streams take alternate steps (one step's upload overlaps the other's "
                  "download); every step uploads its state and downloads its result inside the timed region",
           "one_context_value": world * nodes / e2e_vals["one_context"] / 1e6}
    pair[1].close()
    del pair[1]

    if rank != 0:
        return 0
    # context for the roofline at this size: a plain device copy of the
    # kernel's bytes (its populations in, its populations out) after the
    # same L2 flush.  Outside the timed region; not a kernel of this library.
    half = BYTES_PER_FLUID_NODE[storage] // 2 * nodes
    csrc = torch.ones(half // 4, dtype=torch.float32, device=dev)
    cdst = torch.empty_like(csrc)
    cev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(50)]
    for _ in range(3):
        flush()
        cdst.copy_(csrc)
    for a, b in cev:
        flush()
        a.record(stream)
        cdst.copy_(csrc)
        b.record(stream)
    torch.cuda.synchronize()
    copy_ms = float(np.median([a.elapsed_time(b) for a, b in cev]))
    copy_ctx = {"bytes": 2 * half, "gbs": 2 * half / (copy_ms * 1e-3) / 1e9, "ms": copy_ms,
                "kernel_vs_copy": copy_ms / kernel_ms,
                "what": "torch copy of the kernel's bytes (all node slots in and out) after the same flush"}
    del csrc, cdst
    peak, peak_kind = peaks()
    alg_bytes = BYTES_PER_FLUID_NODE[storage] * fluid
    achieved = alg_bytes / (kernel_ms * 1e-3) / 1e9
    traffic = recorded_traffic("k_fluid_local", storage, "porous1024")
    line = {
        "metric": METRIC, "value": value, "unit": "MLUPS", "n_gpus": world, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": ms_step, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "f32", "data": "synthetic",
        "config": {"workload": WORKLOAD, "nodes": nodes, "fluid_nodes": fluid,
                   "porosity": w.info["porosity"], "storage": storage,
                   "l2": "flushed before every timed step (write 2xL2, read 2xL2)",
                   "thermo_every": THERMO_EVERY,
                   "thermo_records": "deferred: copied to the host inside the thermo step, read by the next "
                                     f"thermo evaluation (the last, step {last_thermo['step']}, after the timed steps)"
                                     if last_thermo else "none: fewer iterations than the thermo interval",
                   "parallelism": f"replicas x{world}"},
        "mflups": world * fluid / (ms_step * 1e-3) / 1e6,
        "bytes_all_nodes_frac": BYTES_PER_FLUID_NODE[storage] * nodes / (kernel_ms * 1e-3) / 1e9 / peaks()[0],
        "roofline": {"bound": "hbm", "achieved": achieved, "peak": peak, "unit": "GB/s",
                     "frac": achieved / peak, "traffic": traffic, "peak_kind": peak_kind,
                     "kernel": "k_fluid_local", "kernel_ms": kernel_ms,
                     "frac_of_nominal_8000_gbs": achieved / 8000.0,
                     "algorithmic_bytes_per_launch": alg_bytes},
        "copy_same_bytes": copy_ctx,
        "e2e": e2e,
        "gpu_launches": int(launches),
        "wall_s_timed_region": wall,
    }
    if clocks:
        line["clocks"] = clocks
    if world == 1 and not args.no_variants:
        line["variants"] = variants(args, local, stream, flush, value)
    if world == 1 and not args.no_cpu_baseline:
        v, n, dt = oracle_rate(w, args.cpu_seconds, 2000)
        line["cpu_baseline"] = {"value": v, "unit": "MLUPS", "cores": 1, "kind": "oracle",
                                "sample": f"full 1024x1024 lattice, {n} iterations ({dt:.1f} s)"}
    print(json.dumps(line), flush=True)
    return 0


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=200)
    ap.add_argument("--warmup", type=int, default=10)
    ap.add_argument("--impl", default="gb300", choices=["gb300", "reference"])
    ap.add_argument("--storage", default="fp32", choices=["fp32", "fp16", "bf16"])
    ap.add_argument("--cpu-seconds", type=float, default=12.0)
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-variants", action="store_true")
    ap.add_argument("--mode", default="replicas", choices=["replicas", "split", "batch"])
    args = ap.parse_args()
    if args.warmup < 3:
        args.warmup = 3
    world, rank, local, dist = dist_setup(args)
    try:
        if args.impl == "reference":
            return run_reference(args, world, rank, dist)
        if args.mode == "split":
            return run_split(args, world, rank, local, dist)
        if args.mode == "batch":
            return run_batch_split(args, world, rank, local, dist)
        return run_gb300(args, world, rank, local, dist)
    finally:
        if dist is not None:
            dist.destroy_process_group()


if __name__ == "__main__":
    sys.exit(main())
