#!/usr/bin/env python
"""Benchmark of the event-driven e-prop hot path on one GB300 (or N replicas).

Workload: the million-neuron sparse network -- 1e6 LIF neurons, fixed
in-degree 1000 (1e9 plastic synapses stored as target|delay, FP32 weight,
BF16 trace), delays 1-5 steps, ~5 Hz, 100 readouts with random feedback,
continuous dynamics with an online weight update every 100 steps.  One
bench step = one simulate call of T = 1000 steps (1 s of biological time).

Prints one JSON line: synapse-events/s over K timed steps (device time,
CUDA events on the library's stream), the roofline of the synapse-trace
kernel, the FP64 oracle timed on a bounded sample on the host cores, the
end-to-end number through the public API with host buffers, and the SM
clocks sampled during the timed region.

    python bench.py [--gpus N] [--steps K] [--warmup W] [--impl reference]
"""
from __future__ import annotations

import argparse
import hashlib
import json
import os
import statistics
import subprocess
import sys
import threading
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "synapse-events/s and sim-time/wall-time vs HBM roofline at stated grad error"
UNIT = "synapse-events/s"
FALLBACK_HBM_GBS = 6800.0
TRACE_KERNEL_SRC = os.path.join(ROOT, "paper_2511_21674_gb300", "csrc", "kernels_window.cu")
TRAFFIC_FILE = os.path.join(ROOT, "profiles", "window_pass_million_sparse.md")


def parse():
    p = argparse.ArgumentParser()
    p.add_argument("--gpus", type=int, default=1)
    p.add_argument("--steps", type=int, default=5)
    p.add_argument("--warmup", type=int, default=3)
    p.add_argument("--impl", default="ours", choices=["ours", "reference"])
    p.add_argument("--workload", default="million", choices=["million", "scaling", "batched", "balanced"],
                   help="million: 1e6 LIF, in-degree 1000; scaling: the paper's scaling network "
                        "(128k ignore-and-fire neurons, in-degree 10,000, 20 s); batched: event "
                        "classification, 64 samples of uneven length per call; balanced: 1e5 LIF "
                        "E/I network, in-degree 1000, T = 2000, update window 100 (stored traces)")
    p.add_argument("--launch-mode", type=int, default=None,
                   help="0 eager launches, 1 graph of launches, 2 persistent step loop "
                        "(default: 1, and 2 for the batched workload)")
    p.add_argument("--scale", type=int, default=1,
                   help="scaling workload: input, recurrent and readout layers times this factor "
                        "(in-degrees and feedback out-degree fixed), as the paper's weak scaling grows it")
    p.add_argument("--n-rec", type=int, default=1_000_000)
    p.add_argument("--k-in", type=int, default=1000)
    p.add_argument("--T", type=int, default=1000)
    p.add_argument("--n-out", type=int, default=100)
    p.add_argument("--trace-dtype", default="bf16", choices=["bf16", "fp16", "fp32"])
    p.add_argument("--blocks-per-sm", type=int, default=0)
    p.add_argument("--trace-kernel", default="dense", choices=["dense", "band", "lazy"],
                   help="synapse-trace form: dense window pass (source-major records), the same "
                        "with band-major records (coefficients in shared memory), or lazy catch-up "
                        "at arrivals")
    p.add_argument("--no-cpu-baseline", action="store_true")
    p.add_argument("--no-forms", action="store_true",
                   help="skip the batched-form timing (event classification, batch 64)")
    p.add_argument("--cpu-sample-n", type=int, default=10_000)
    p.add_argument("--cpu-sample-T", type=int, default=300)
    return p.parse_args()


# ----------------------------------------------------------------- helpers


def measured_peaks():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    try:
        with open(path) as f:
            d = json.load(f)
        return float(d["hbm_gbs"]), "measured"
    except Exception:
        return FALLBACK_HBM_GBS, "fallback"


def recorded_traffic():
    """DRAM bytes of one window pass (its two launches) at full size,
    from the committed ncu summary, if it was taken on the current kernel
    source (sha256 recorded in the summary); else None."""
    try:
        text = open(TRAFFIC_FILE).read()
        src = hashlib.sha256(open(TRACE_KERNEL_SRC, "rb").read()).hexdigest()
        fields = dict(line.split(":", 1) for line in text.splitlines() if ":" in line and line[0] != " ")
        if fields.get("kernel_source_sha256", "").strip() != src:
            return None
        return float(fields["dram_bytes_per_window_at_full_size"].strip())
    except Exception:
        return None


class ClockSampler:
    """nvidia-smi clocks/throttle reasons every 200 ms during a region."""
    QUERY = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
             "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
             "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index):
        self.gpu = gpu_index
        self.proc = None
        self.lines = []

    def start(self):
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", f"--query-gpu={self.QUERY}", "--format=csv,noheader,nounits",
                 "-lms", "200", "-i", str(self.gpu)], stdout=subprocess.PIPE,
                stderr=subprocess.DEVNULL, text=True)
            self.t = threading.Thread(target=self._read, daemon=True)
            self.t.start()
        except Exception:
            self.proc = None

    def _read(self):
        for line in self.proc.stdout:
            self.lines.append(line.strip())

    def stop(self):
        if self.proc is None:
            return None
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except Exception:
            self.proc.kill()
        sm, smax, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for line in self.lines:
            parts = [x.strip() for x in line.split(",")]
            if len(parts) < 9:
                continue
            try:
                sm.append(float(parts[1]))
                smax.append(float(parts[2]))
            except ValueError:
                continue
            for name, val in zip(names, parts[5:9]):
                if val.lower().startswith("active"):
                    reasons.add(name)
        if not sm:
            return None
        return {"sm_mhz": statistics.median(sm), "sm_max_mhz": max(smax),
                "reasons": sorted(reasons), "samples": len(sm)}


def dist_setup(n_gpus):
    import torch
    rank = int(os.environ.get("RANK", "0"))
    world = int(os.environ.get("WORLD_SIZE", "1"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    if world > 1:
        import torch.distributed as dist
        torch.cuda.set_device(local)
        dist.init_process_group("nccl")
    else:
        torch.cuda.set_device(0)
    return rank, world, local


def barrier_max(value, world):
    import torch
    if world == 1:
        return value
    import torch.distributed as dist
    # NCCL reduces device tensors; the gloo backend (CPU tests) host tensors
    dev = "cuda" if dist.get_backend() == "nccl" else "cpu"
    t = torch.tensor([value], dtype=torch.float64, device=dev)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def replica_seed(rank):
    """Each replica builds its own network and drive (independent problems)."""
    return 1237 + rank


def barrier(world):
    if world > 1:
        import torch.distributed as dist
        dist.barrier()


# --------------------------------------------------------------- CPU oracle


def workload_config(args, nnz, world=1):
    """The workload one step runs (both arms report it)."""
    if args.workload == "batched":
        return {"workload": "event classification (N-MNIST-shaped, synthetic): batch 64, lengths 250-350, "
                            "2312 inputs, 200 ALIF (10% recurrent), 10 readouts, CE on each sample's last "
                            f"25 steps, one update window per call ({nnz} synapses)",
                "batch": 64, "T_per_step": 350, "synapses": nnz, "launch_mode": launch_mode(args),
                "trace_storage": "fp32", "parallelism": f"replicas{world}",
                "l2": "small working set (L2-resident): a latency-bound workload"}
    if args.workload == "scaling":
        sc = scaling_sizes(args)
        return {"workload": f"scaling: {sc['n_rec']} ignore-and-fire neurons at 5 Hz, recurrent "
                            f"in-degree {sc['k_rec']}, {sc['n_in']} Poisson inputs at 5 Hz "
                            f"(in-degree {sc['k_in']}), {sc['n_out']} readouts (in-degree "
                            f"{sc['k_out']}), feedback out-degree {sc['fb_outdeg']}, delays 1-5, "
                            f"update window {sc['update_interval']}, continuous, "
                            f"{sc['T']} steps per bench step ({nnz} synapses)",
                "n_rec": sc["n_rec"], "k_rec": sc["k_rec"], "synapses": nnz, "scale": args.scale,
                "T_per_step": sc["T"], "trace_storage": args.trace_dtype,
                "trace_form": args.trace_kernel, "parallelism": f"replicas{world}",
                "l2": "inputs larger than L2 (synapse records ~13 GB)"}
    if args.workload == "balanced":
        return {"workload": f"sparse balanced: 100000 LIF (80% excitatory), fixed in-degree 1000 ({nnz} "
                            "synapses), delays 1-5, Poisson drive (~5-10 Hz), 500 readout-coupled "
                            "neurons, 1 readout (sum of sinusoids), T = 2000, update window 100, "
                            "continuous (traces stored between windows), lr 1e-8",
                "n_rec": 100_000, "k_in": 1000, "synapses": nnz, "T_per_step": 2000,
                "trace_storage": args.trace_dtype, "trace_form": args.trace_kernel,
                "parallelism": f"replicas{world}",
                "l2": "inputs larger than L2 (synapse records ~1 GB per step)"}
    return {"workload": f"million_sparse: {args.n_rec} LIF, in-degree {args.k_in} ({nnz} synapses), "
                        f"delays 1-5, ~5 Hz, {args.n_out} readouts, update window 100, continuous",
            "n_rec": args.n_rec, "k_in": args.k_in, "synapses": nnz, "T_per_step": args.T,
            "trace_storage": args.trace_dtype, "trace_form": args.trace_kernel,
            "parallelism": f"replicas{world}",
            "l2": "inputs larger than L2 (synapse records ~10 GB per step)"}


# the scaling experiment's network (Methods, "Scaling"): base size, 20 s
SCALING = dict(n_rec=128_000, k_rec=10_000, n_in=1000, k_in=100, n_out=10, k_out=1000, fb_outdeg=100,
               T=20_000, update_interval=1000)


def scaling_sizes(args):
    """The scaling network grown by --scale: the paper's weak scaling enlarges
    the input, recurrent and readout layers together at fixed in-degrees."""
    f = max(1, int(getattr(args, "scale", 1)))
    return dict(SCALING, n_rec=SCALING["n_rec"] * f, n_in=SCALING["n_in"] * f, n_out=SCALING["n_out"] * f)


# the bounded sample of it the CPU oracle runs
SCALING_SAMPLE = dict(n_rec=2000, k_rec=1000, n_in=100, k_in=10, n_out=10, k_out=100, fb_outdeg=20,
                      T=100, update_interval=100)


def launch_mode(args):
    if args.launch_mode is not None:
        return args.launch_mode
    return 2 if args.workload == "batched" else 1


def cpu_model():
    """The host CPU's model string (lscpu / /proc/cpuinfo), for the record."""
    try:
        out = subprocess.run(["lscpu"], capture_output=True, text=True, timeout=10).stdout
        for key in ("Model name", "Vendor ID"):
            for line in out.splitlines():
                if line.startswith(key):
                    return line.split(":", 1)[1].strip()
    except Exception:
        pass
    return "unknown"


def cpu_baseline(args, steps=1):
    """The FP64 oracle (test infrastructure, untuned) on a bounded sample of
    the same workload: cpu_sample_n neurons with the same in-degree, delays,
    drive and rates, cpu_sample_T steps (one update window)."""
    import oracle
    from workloads import configs as C
    oracle.build()
    threads = oracle.set_threads(os.cpu_count() or 1)
    if args.workload == "batched":
        W = C.event_classification(batch=4)
        sample = (f"event classification, 4 samples of 250-350 steps x {steps}, FP64 time-driven "
                  f"oracle, {threads} threads")
    elif args.workload == "scaling":
        W = C.scaling_network(**SCALING_SAMPLE)
        sample = ("scaling network sample: 2000 ignore-and-fire neurons, recurrent in-degree 1000, "
                  "100 Poisson inputs (in-degree 10), 10 readouts (in-degree 100), feedback out-degree 20, "
                  f"100 steps x {steps}, FP64 time-driven oracle, {threads} threads")
    elif args.workload == "balanced":
        W = C.sparse_balanced(n_rec=args.cpu_sample_n, T=args.cpu_sample_T, n_coupled=500,
                              update_interval=100, continuous=1, lr=1e-8)
        sample = (f"sparse balanced sample: {args.cpu_sample_n} LIF, in-degree 1000, delays 1-5, "
                  f"500 readout-coupled, {args.cpu_sample_T} steps x {steps}, FP64 time-driven oracle, "
                  f"{threads} threads")
    else:
        W = C.million_sparse(n_rec=args.cpu_sample_n, k_in=args.k_in, T=args.cpu_sample_T,
                             n_out=args.n_out)
        sample = (f"{args.cpu_sample_n} LIF neurons, in-degree {args.k_in}, delays 1-5, "
                  f"~5 Hz, {args.n_out} readouts, {args.cpu_sample_T} steps x {steps}, "
                  f"FP64 time-driven oracle, {threads} threads")
    s = W["spec"]
    if args.workload != "batched":
        s.update_interval = s.T
    o = oracle.Oracle(s, W["ptr"], W["col"], W["w"], W["delay"], W["w_out"], W["out_mask"],
                      W["feedback"])
    outdeg = np.diff(W["ptr"])
    tot_events, tot_time = 0, 0.0
    for _ in range(steps):
        t0 = time.perf_counter()
        r = o.simulate(s.T, W["x_ptr"], W["x_ids"], W["targets"], W["window"], W["lengths"])
        tot_time += time.perf_counter() - t0
        tot_events += int((r["raster"].sum(axis=(0, 1)) * outdeg[s.n_in:]).sum())
        if s.n_in:
            src = np.asarray(W["x_ids"], np.int64)
            tot_events += int(outdeg[src].sum())
    return {"value": tot_events / tot_time, "unit": UNIT, "cores": threads, "kind": "oracle",
            "sample": sample, "events": tot_events, "seconds": tot_time, "cpu_model": cpu_model()}


def batched_form_timing(calls=10, warmup=3):
    """Form (2) on the event-classification workload (batch 64, lengths
    250-350, 200 ALIF, 2312 inputs): ms per simulate call launched eagerly
    (launch_mode 0), as a captured graph (1) and with every step of the call in
    one launch (2; a network of this size runs so in every mode); CUDA events on
    the network's stream, inputs resident."""
    import torch
    import paper_2511_21674_gb300 as ep
    from workloads import configs as C
    W = C.event_classification(batch=64)
    s = W["spec"]
    out = {"workload": "event classification: batch 64, lengths 250-350, 2312 inputs, 200 ALIF, "
                       "10 readouts, CE on each sample's last 25 steps, one window per call"}
    for mode in (0, 1, 2):
        net = ep.Network(s, W["ptr"], W["col"], W["w"], W["delay"], W["w_out"], W["out_mask"],
                         W["feedback"], launch_mode=mode, record_grad=0)
        net.set_inputs(W["x_ptr"], W["x_ids"], W["targets"], W["window"], W["lengths"], s.T)
        for _ in range(warmup):
            net.simulate(s.T)
        net.sync()
        st = torch.cuda.current_stream()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(st)
        for _ in range(calls):
            net.simulate(s.T)
        e1.record(st)
        torch.cuda.synchronize()
        ms = e0.elapsed_time(e1) / calls
        stats = net.stats()
        out[f"ms_per_call_mode{mode}"] = ms
        out[f"kernel_launches_mode{mode}"] = stats["kernel_launches"]
        if mode == 2:
            out["samples_per_s"] = s.batch / (ms / 1000.0)
            out["events_per_s"] = stats["events"] / (ms / 1000.0)
        net.close()
    return out


def run_reference(args):
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return
    W = max(args.warmup, 0)
    base = cpu_baseline(args, steps=1 + 0 * W)  # warm: builds the oracle
    K = max(args.steps, 1)
    res = cpu_baseline(args, steps=K)
    sec_per_step = res["seconds"] / K
    line = {"impl": "reference", "metric": METRIC, "value": res["value"], "unit": UNIT,
            "n_gpus": args.gpus, "steps": K, "warmup": args.warmup,
            "ms_per_step": 1000.0 * sec_per_step, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": workload_config(args, args.n_rec * args.k_in, args.gpus),
            "cpu_baseline": {"kind": "oracle", "cores": res["cores"], "sample": res["sample"],
                             "cpu_model": res["cpu_model"],
                             "value": res["value"], "unit": UNIT},
            "e2e": {"value": res["value"], "unit": UNIT, "h2d_bytes_per_step": 0,
                    "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)
    del base


# ------------------------------------------------------------------ GPU arm


def run_ours(args):
    import torch
    rank, world, local = dist_setup(args.gpus)
    side = torch.cuda.Stream()          # graphs are captured on a non-default stream
    with torch.cuda.stream(side):
        _run_ours(args, rank, world, local)


def _run_ours(args, rank, world, local):
    import torch
    import paper_2511_21674_gb300 as ep
    from workloads import configs as C
    from workloads import gpu_build as G
    torch.manual_seed(0)
    if args.workload == "batched":
        W = C.event_classification(batch=64, seed=1235 + rank)
    elif args.workload == "scaling":
        W = G.scaling_torch(seed=replica_seed(rank) + 4, **scaling_sizes(args))
    elif args.workload == "balanced":
        # lr 1e-8 keeps the rate in the 5-10 Hz band over the timed calls
        # (the regression signal through unit-variance feedback to every
        # neuron raises it after ~50 updates at 1e-7)
        W = C.sparse_balanced(seed=replica_seed(rank) + 2, update_interval=100, continuous=1, lr=1e-8)
    else:
        W = G.million_sparse_torch(n_rec=args.n_rec, k_in=args.k_in, T=args.T, n_out=args.n_out,
                                   seed=replica_seed(rank))
    spec = W["spec"]
    torch.cuda.empty_cache()        # the build's freed temporaries back to the device
    trace_dtype = {"fp32": 0, "bf16": 1, "fp16": 2}[args.trace_dtype]
    if args.workload == "batched":
        trace_dtype = 0                  # single-window form: no traces are stored
    net = ep.Network(spec, W["ptr"], W["col"], W["w"], W["delay"], W["w_out"], W["out_mask"], W["feedback"],
                     launch_mode=launch_mode(args), trace_dtype=trace_dtype, record_grad=0, record_raster=0,
                     profile=1, blocks_per_sm=args.blocks_per_sm,
                     trace_kernel=(0 if args.workload == "batched" else
                                   {"dense": 3, "band": 4, "lazy": 1}[args.trace_kernel]))
    nnz = int(W["col"].shape[0])
    del W["ptr"], W["col"], W["w"], W["delay"], W["w_out"], W["feedback"], W["out_mask"]
    torch.cuda.empty_cache()
    T = spec.T
    # inputs: pinned host buffers (the same arrays serve every step)
    x_ptr = torch.from_numpy(W["x_ptr"]).pin_memory()
    x_ids = torch.from_numpy(np.concatenate([W["x_ids"], np.zeros(1, np.int32)])).pin_memory()[:len(W["x_ids"])]
    targets = torch.from_numpy(np.ascontiguousarray(W["targets"], np.float32)).pin_memory()
    window = torch.from_numpy(W["window"]).pin_memory()
    lengths = torch.from_numpy(W["lengths"]).pin_memory()
    net.set_inputs(x_ptr, x_ids, targets, window, lengths, T)
    stream = torch.cuda.current_stream()
    for _ in range(max(args.warmup, 3)):
        net.simulate(T)
    net.sync()

    # ---- device-timed region: K simulate calls, inputs resident in HBM
    K = args.steps
    clocks = ClockSampler(local)
    barrier(world)
    torch.cuda.synchronize()
    clocks.start()
    ev0 = torch.cuda.Event(enable_timing=True)
    ev1 = torch.cuda.Event(enable_timing=True)
    ev0.record(stream)
    events = launches = trace_launches = windows = 0
    trace_ms = 0.0
    for _ in range(K):
        net.simulate(T)
        st = net.stats()
        events += st["events"]
        launches += st["kernel_launches"]
        trace_launches += st["trace_launches"]
        windows += st["windows"]
        trace_ms += st["trace_ms"]
    ev1.record(stream)
    torch.cuda.synchronize()
    barrier(world)
    clk = clocks.stop()
    ms = ev0.elapsed_time(ev1)
    ms_max = barrier_max(ms, world)
    ev_total = barrier_max(events, world) * world if world > 1 else events
    value = ev_total / (ms_max / 1000.0)

    # ---- end to end through the public API with host buffers
    h2d = (x_ptr.numel() * 8 + x_ids.numel() * 4 + targets.numel() * 4 + window.numel() +
           lengths.numel() * 4)
    # results land in pinned host buffers
    loss_t = torch.zeros(spec.batch, dtype=torch.float32).pin_memory()
    y_t = torch.zeros((spec.batch, T, spec.n_out), dtype=torch.float32).pin_memory()
    loss_host, y_host = loss_t.numpy(), y_t.numpy()
    barrier(world)
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    e2e_events = 0
    for _ in range(K):
        net.set_inputs(x_ptr, x_ids, targets, window, lengths, T)
        net.simulate(T)
        # the step's results back on the host: readout trace y and loss
        st_r = net.lib.eprop_readout(net.h, y_host.ctypes.data, loss_host.ctypes.data, None, 0)
        if st_r != 0:
            raise RuntimeError(f"eprop_readout failed: {st_r}")
        e2e_events += net.stats()["events"]
    torch.cuda.synchronize()
    e2e_s = barrier_max(time.perf_counter() - t0, world)
    e2e_value = (e2e_events * world) / e2e_s

    # ---- roofline of the synapse-trace kernel
    bytes_per_event = 16.0 if trace_dtype else 20.0          # j|d 4 r, w 4 r/w, trace 2|4 r/w
    peak, peak_src = measured_peaks()
    achieved = events * bytes_per_event / (trace_ms / 1000.0) / 1e9 if trace_ms > 0 else None
    # per window pass (the unit `achieved` averages over): DRAM bytes from
    # the committed ncu capture, scaled to full size (see profiles/)
    traffic = recorded_traffic() if (args.trace_kernel == "dense" and args.workload == "million") else None
    net.close()
    if rank != 0:
        return
    line = {
        "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": K,
        "warmup": max(args.warmup, 3), "ms_per_step": ms_max / K, "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "f32", "data": "synthetic",
        "config": workload_config(args, nnz, world),
        "sim_time_per_wall_time": (T * spec.dt / 1000.0) / (ms_max / K / 1000.0),
        "real_time_factor": (ms_max / K / 1000.0) / (T * spec.dt / 1000.0),
        "events_per_step": events / K,
        "mean_rate_hz": events / K / nnz / (T * spec.dt / 1000.0),
        "grad_error": "FP32 traces: within 1e-5 of each gradient's magnitude sum vs the FP64 oracle "
                      "(scaled replicas on every synapse, this workload on 256 sampled synapses); "
                      "BF16 traces: ~5e-4 relative L2 vs the oracle (gated at 1e-2)",
        "roofline": {"bound": "hbm", "achieved": achieved, "peak": peak, "unit": "GB/s",
                     "frac": (achieved / peak) if achieved else None, "traffic": traffic,
                     "kernel": {"dense": "window_pass_kernel (spiking-row and idle-row launches per update window)",
                                "band": "window_band_kernel (band-major records, the band's coefficients in "
                                        "shared memory) after band_rows_kernel (row records of the window)",
                                "lazy": "trace_window_kernel (lazy: rows with an arrival in the window)"
                                }[args.trace_kernel],
                     "bytes_per_event": bytes_per_event,
                     "stream_bytes_per_window": nnz * bytes_per_event,
                     "algorithmic_bytes_per_window": (events * bytes_per_event / windows) if windows else None,
                     "traffic_unit": "DRAM bytes per window pass (both launches)",
                     "peak_source": f"{peak_src} (hbm_gbs)",
                     "trace_ms_per_step": trace_ms / K, "trace_launches_per_step": trace_launches / K},
        "samples_per_s": spec.batch * K / (ms_max / 1000.0),
        "e2e": {"value": e2e_value, "unit": UNIT, "h2d_bytes_per_step": int(h2d),
                "d2h_bytes_per_step": int(loss_host.nbytes + y_host.nbytes)},
        "gpu_launches": int(launches),
        "clocks": clk,
    }
    if args.workload == "batched":
        # a latency-bound workload (a few MB, L2-resident): no HBM roofline
        line["roofline"] = {"bound": "latency", "achieved": None, "peak": None, "unit": None, "frac": None,
                            "traffic": None, "note": "64 samples x 200 neurons: launch and barrier latency "
                                                     "bound; the HBM fraction is not meaningful"}
    if not args.no_forms and args.workload == "million":
        try:
            line["form2_batched"] = batched_form_timing()
        except Exception as exc:  # the main line stands on its own
            line["form2_batched"] = {"error": str(exc)}
    if not args.no_cpu_baseline:
        try:
            cb = cpu_baseline(args, steps=1)
            line["cpu_baseline"] = {k: cb[k] for k in ("value", "unit", "cores", "kind", "sample", "cpu_model")}
        except Exception as exc:  # the GPU line stands on its own
            line["cpu_baseline"] = {"error": str(exc)}
    print(json.dumps(line), flush=True)


def main():
    args = parse()
    if args.impl == "reference":
        run_reference(args)
        return
    run_ours(args)


if __name__ == "__main__":
    main()
