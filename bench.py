"""Benchmark of the skipped-step extrapolation (Sec. 3.3, Eq. for f_t) on GB300.

One step = one skipped diffusion step over every block of the workload: the
host computes the fp64 weights for the target timestep from the live history
and one grouped persistent kernel streams the K cached slots of every branch
tensor and writes the predictions (HBM-bound K-term reduction).

Default workload: FLUX.1-dev 1024^2 shapes (19 double-stream blocks with image
and text streams, 38 single-stream blocks: 114 bf16 tensors, 1.08 G elements
per slot, K = 5). The history is filled by walking the 50-step schedule
(r = 6) to a mid-schedule window of K equispaced nodes; the timed steps cycle
over that window's skipped targets. Inputs (12.9 GB per step) exceed L2
(~129 MB), so no flush is needed between steps.

Usage: python bench.py [--gpus N] [--steps K] [--warmup W] [--config NAME]
                       [--impl ours|reference]
Under torchrun each rank runs its own replica (independent samples, no data
exchange); timing is the max over ranks.

Besides the contract's keys, the JSON line carries: `roofline` (achieved GB/s
of the timed kernel against the measured copy peak, DRAM traffic per launch
from the committed ncu record when it matches the kernel sources),
`schedule_loop` (Alg. 1's whole online stage over the schedule), `parity` (the
timed step's predictions against the oracle on a sample), `workloads` (the
other configurations and the gated, cache-write and full-step-epilogue paths,
each with its own clock sample), `cpu_baseline` (the oracle on the host
cores), `e2e` (the step through the public API from and to pinned host
buffers) and `clocks`.
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
sys.path.insert(0, ROOT)

METRIC = "extrapolation GB/s & % of HBM peak; µs per skipped step (all blocks), 1 GB300"
# configurations timed after the headline (FLUX.1-dev 1024^2), each on its own
# filled history: (preset, [(variant, step, hidden states fused, gated)]).
# step "skip" is a skipped step (cb_extrapolate / cb_extrapolate_gated);
# "full" a full step's cache write (cb_cache_push) and "full-fused" the cache
# write with the hidden-state update (cb_cache_push_residual); full steps run
# after the skipped ones, from an emptied history.
OTHER_WORKLOADS = [
    ("pixart", [("prediction-only", "skip", False, False), ("fused", "skip", True, False),
                ("gated", "skip", True, True), ("full-step epilogue", "full-fused", True, False)]),
    ("dit512", [("prediction-only", "skip", False, False)]),
    ("dit256", [("fused", "skip", True, False), ("prediction-only", "skip", False, False),
                ("gated", "skip", True, True), ("full-step epilogue, gated", "full-fused", True, True)]),
    ("dit256-k3", [("fused", "skip", True, False), ("prediction-only", "skip", False, False)]),
    ("flux", [("fused", "skip", True, False), ("cache write", "full", False, False),
              ("full-step epilogue", "full-fused", True, False)]),
]
NOMINAL_HBM_GBS = 7900.0
KERNEL_SOURCES = ["paper_2608_23429_gb300/csrc/extrapolate_bulk.cu", "paper_2608_23429_gb300/csrc/bulk_kernel.cuh",
                  "paper_2608_23429_gb300/csrc/extrapolate.cu", "paper_2608_23429_gb300/csrc/direct_kernel.cuh",
                  "paper_2608_23429_gb300/csrc/cb_math.cuh", "paper_2608_23429_gb300/csrc/cb_device.h",
                  "paper_2608_23429_gb300/csrc/cb_async.cuh", "paper_2608_23429_gb300/csrc/extrapolate_bulk_precise.cuh"]


def kernel_hash() -> str:
    h = hashlib.sha256()
    for p in KERNEL_SOURCES:
        with open(os.path.join(ROOT, p), "rb") as fh:
            h.update(fh.read())
    return h.hexdigest()[:16]


def measured_peaks() -> tuple[float, str]:
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as fh:
            return float(json.load(fh)["hbm_gbs"]), "measured"
    except (OSError, KeyError, ValueError):
        return 6800.0, "fallback"


def recorded_traffic(config: str) -> float | None:
    """DRAM bytes per launch from the committed ncu summary, if it was taken on
    the current kernel source (else None)."""
    path = os.path.join(ROOT, "profiles", f"extrapolate_bulk_{config}_traffic.txt")
    try:
        fields = dict(line.split("=", 1) for line in open(path).read().split() if "=" in line)
    except OSError:
        return None
    if fields.get("kernel_sha") != kernel_hash():
        return None
    try:
        return float(fields["dram_bytes_per_launch"])
    except (KeyError, ValueError):
        return None


class Clocks:
    """nvidia-smi sampling during the timed region."""

    Q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
         "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
         "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, index: int):
        self.index = index
        self.f = tempfile.NamedTemporaryFile("w+", suffix=".csv", delete=False)
        self.p = None

    def __enter__(self):
        try:
            self.p = subprocess.Popen(["nvidia-smi", f"--id={self.index}", f"--query-gpu={self.Q}",
                                       "--format=csv,noheader,nounits", "-lms", "50"],
                                      stdout=self.f, stderr=subprocess.DEVNULL)
        except OSError:
            self.p = None
        time.sleep(0.3)
        return self

    def __exit__(self, *exc):
        if self.p is not None:
            self.p.terminate()
            try:
                self.p.wait(timeout=5)
            except subprocess.TimeoutExpired:
                self.p.kill()

    def summary(self) -> dict:
        self.f.flush()
        rows = []
        for line in open(self.f.name).read().splitlines():
            parts = [x.strip() for x in line.split(",")]
            if len(parts) < 9:
                continue
            try:
                rows.append(dict(sm=float(parts[1]), max=float(parts[2]), power=float(parts[3]),
                                 hw=parts[5], hwt=parts[6], swt=parts[7], swp=parts[8]))
            except ValueError:
                continue
        os.unlink(self.f.name)
        if not rows:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["unavailable"], "samples": 0}
        top = max(r["power"] for r in rows)
        load = [r for r in rows if r["power"] >= 0.5 * top] or rows
        reasons = []
        for key, name in (("hw", "hw_slowdown"), ("hwt", "hw_thermal_slowdown"),
                          ("swt", "sw_thermal_slowdown"), ("swp", "sw_power_cap")):
            if any(r[key].lower().startswith("active") for r in load):
                reasons.append(name)
        return {"sm_mhz": statistics.median(r["sm"] for r in load), "sm_max_mhz": max(r["max"] for r in rows),
                "reasons": reasons, "samples": len(load), "power_w_max": top}


def dist_env():
    ws = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return ws, rank, local


def max_over_ranks(x: float, device) -> float:
    """Max of a per-rank timing over all ranks (measurement only; no data moves)."""
    import torch
    import torch.distributed as dist
    if not (dist.is_available() and dist.is_initialized()) or dist.get_world_size() == 1:
        return x
    t = torch.tensor([float(x)], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def workload_description(w) -> dict:
    slot = sum(t.numel for t in w.tensors) * w.esize()
    return {"workload": w.name, "tensors": len(w.tensors), "K": w.K, "storage": w.cache_dtype,
            "slot_bytes": slot,
            "schedule": (f"explicit nodes {list(w.explicit_nodes)}, targets {list(w.explicit_targets)}"
                         if w.explicit_nodes else f"T={w.T}, full every r={w.r}")}


def full_mask(w, cb):
    """The schedule's full steps (Sec. 3.3 set F plus warm-up), from the library."""
    mask, _ = cb.cb_schedule_full(w.T, w.r, w.s0, w.s1, w.K)
    return mask


def pick_window(w, cb):
    """The product's timed window: see window_of."""
    return window_of(w, full_mask(w, cb))


def window_of(w, mask):
    """Walk a schedule mask to the first window of K equispaced nodes past the
    warm-up; return (full steps pushed in order, skipped steps that follow)."""
    full = [s for s in range(w.T) if mask[s]]
    for k in range(w.K - 1, len(full) - 1):
        win = full[k - w.K + 1:k + 1]
        if len({b - a for a, b in zip(win, win[1:])}) == 1 and win[-1] - win[0] == w.r * (w.K - 1):
            targets = [s for s in range(win[-1] + 1, full[k + 1])]
            if targets:
                return full[:k + 1], targets
    raise RuntimeError("no equispaced window in the schedule")


def cpu_oracle_run(w, feats_host, wts, seconds: float, nthreads: int):
    """Time the oracle on a bounded sample; returns (GB/s, elements, reps, seconds)."""
    import oracle as orc
    reps, t0 = 0, time.perf_counter()
    n = feats_host[0].size
    while True:
        orc.extrapolate([feats_host], wts, orc.BF16, orc.BF16, nthreads=nthreads)
        reps += 1
        el = time.perf_counter() - t0
        if el >= seconds:
            break
    gbs = reps * n * (w.K + 1) * 2 / el / 1e9
    return gbs, n, reps, el


def oracle_parity(orc, host, wts, gpu_bits) -> dict:
    """The oracle's fp64 prediction for the sampled elements (the first
    gpu_bits.size of the CPU baseline's sample), rounded once to bf16, against
    the GPU's bits."""
    import numpy as np
    n = gpu_bits.size
    F = [h[:n] for h in host]
    o64, _ = orc.extrapolate([F], wts, orc.BF16, orc.FP64, nthreads=os.cpu_count() or 1)
    ref = orc.convert(o64[0], orc.FP64, orc.BF16)
    Fd = np.array([(f.astype(np.uint32) << 16).view(np.float32).astype(np.float64) for f in F])
    bound = (np.abs(np.asarray(wts, dtype=np.float64))[:, None] * np.abs(Fd)).sum(0)
    return parity_stats(gpu_bits, ref, o64[0], bound)


def cpu_model() -> str:
    """The host CPU's model name (lscpu, else /proc/cpuinfo)."""
    try:
        out = subprocess.run(["lscpu"], capture_output=True, text=True, timeout=10).stdout
        for line in out.splitlines():
            if line.strip().lower().startswith("model name"):
                return line.split(":", 1)[1].strip()
    except (OSError, subprocess.SubprocessError):
        pass
    try:
        for line in open("/proc/cpuinfo"):
            if line.lower().startswith(("model name", "cpu part")):
                return line.split(":", 1)[1].strip()
    except OSError:
        pass
    return "unknown"


def sample_host_features(w, torch, wl, orc, n_elems: int, device):
    """A bounded contiguous sample of the largest tensor at K nodes (generator bytes)."""
    i = max(range(len(w.tensors)), key=lambda k: w.tensors[k].numel)
    full, targets = window_of(w, orc.full_schedule(w.T, w.r, w.s0, w.s1, w.K))  # the oracle's own schedule
    nodes = full[-w.K:]
    host = []
    for s in nodes:
        f = wl.trajectory(w, i, w.timesteps[s], s, device).reshape(-1)[:n_elems]
        host.append(f.contiguous().cpu().view(torch.int16).numpy().view("uint16").copy())
    t_nodes = [w.timesteps[s] for s in nodes]
    wts = orc.weights(t_nodes, w.timesteps[targets[0]], w.t_min, w.t_max)
    return host, wts, i


def parity_stats(gpu_bits, ref_bits, ref64, bound64) -> dict:
    """bf16 results against the oracle: ulp distance of the bit patterns, with
    exact cancellations (|gpu - exact| <= 2^-40 sum_j |w_j F_j|) counted apart."""
    import numpy as np

    def ordered(b):
        b = b.astype(np.int64)
        return np.where(b & 0x8000, -(b & 0x7FFF), b)

    d = np.abs(ordered(gpu_bits) - ordered(ref_bits))
    g64 = (gpu_bits.astype(np.uint32) << 16).view(np.float32).astype(np.float64)
    floor = np.abs(g64 - ref64) <= 2.0 ** -40 * bound64
    return {"n": int(d.size), "exact": int((d == 0).sum()), "one_ulp": int((d == 1).sum()),
            "floor": int(((d > 1) & floor).sum()), "bad": int(((d > 1) & ~floor).sum()),
            "max_ulp": int(d.max()) if d.size else 0}


def fill_window(torch, cb, wl, w, plan, cdt, pushed, dev, stream):
    """The schedule's full steps up to the timed window, pushed in order."""
    for s in pushed:
        feats = [wl.trajectory(w, i, w.timesteps[s], s, dev) for i in range(len(w.tensors))]
        torch.cuda.synchronize()
        cb.cb_cache_push(plan, feats, cdt, w.timesteps[s], stream=stream)
        stream.synchronize()
        del feats


def time_workload(torch, cb, wl, dev, name: str, variants, steps: int, warmup: int, peak: float) -> list:
    """More steps of one more workload in the launch configuration of the
    headline: the same window walk, one launch per step, per-launch events on
    the launching stream. variants: (label, step, fused, gated) on one filled
    history (see OTHER_WORKLOADS)."""
    w = wl.PRESETS[name]()
    K = w.K
    pushed, targets = pick_window(w, cb)
    node_t = [w.timesteps[s] for s in full_mask(w, cb).nonzero()[0]]
    cdt = cb.CB_BF16 if w.cache_dtype == "bf16" else cb.CB_FP32
    tdt = torch.bfloat16 if w.cache_dtype == "bf16" else torch.float32
    plan = cb.cb_plan_create(node_t, K, [(t.layer, t.branch, t.numel, t.group) for t in w.tensors], cdt,
                             w.t_min, w.t_max)
    cb.cb_plan_set_shapes(plan, [t.shape for t in w.tensors])
    cache = torch.empty(cb.cb_plan_cache_bytes(plan), dtype=torch.uint8, device=dev)
    cb.cb_plan_bind_cache(plan, cache, cache.numel())
    stream = torch.cuda.Stream(device=dev)
    fill_window(torch, cb, wl, w, plan, cdt, pushed, dev, stream)
    outs = [torch.empty(t.shape, dtype=tdt, device=dev) for t in w.tensors]
    n_groups = cb.cb_plan_num_groups(plan)
    slot_elems = sum(t.numel for t in w.tensors)
    esz = 2 if w.cache_dtype == "bf16" else 4
    t_targets = [w.timesteps[s] for s in targets]
    gg = torch.Generator(device=dev).manual_seed(7)
    gates = [(0.5 * torch.randn(t.shape[0], t.shape[-1], generator=gg, device=dev)).to(torch.bfloat16)
             for t in w.tensors]
    gate_bytes = sum(t.shape[0] * t.shape[-1] * 2 for t in w.tensors)
    src = None
    # fresh, strictly monotone times for the full steps (pushed from an emptied history)
    span = (w.timesteps[-1] - w.timesteps[0]) / 1e6
    push_t = iter([w.timesteps[0] + span * i for i in range(1000000)])
    rows = []
    for label, step, fused, gated in variants:
        resid = [wl.hidden_state(w, g, dev) for g in range(n_groups)] if fused else None
        resid_elems = sum(w.group_numel(g) for g in range(n_groups)) if fused else 0
        outs_p = cb.ptr_array(outs)
        resid_p = cb.ptr_array(resid) if resid is not None else None
        gates_p = cb.ptr_array(gates) if gated else None
        if step == "skip":
            # K slot reads + one output write (+ hidden state read and write, + gates)
            bytes_step = slot_elems * esz * (K + 1) + resid_elems * 2 * 2 + (gate_bytes if gated else 0)

            def launch(k):
                t = t_targets[k % len(t_targets)]
                if gated:
                    cb.cb_extrapolate_gated(plan, t, outs_p, cdt, resid_p, cb.CB_BF16, gates_p, cb.CB_BF16,
                                            stream=stream)
                else:
                    cb.cb_extrapolate(plan, t, outs_p, cdt, resid_p, cb.CB_BF16, stream=stream)
        else:
            if src is None:  # the features of one generated full step, re-pushed with fresh times
                src = [wl.trajectory(w, i, w.timesteps[pushed[-1]], pushed[-1], dev) for i in range(len(w.tensors))]
                torch.cuda.synchronize()
                cb.cb_plan_reset(plan)
            src_p = cb.ptr_array(src)
            # features read + slot written (+ hidden state read and write, + gates)
            bytes_step = slot_elems * (src[0].element_size() + esz)
            if step == "full-fused":
                bytes_step += resid_elems * 2 * 2 + (gate_bytes if gated else 0)

            def launch(k):
                t = next(push_t)
                if step == "full":
                    cb.cb_cache_push(plan, src_p, cdt, t, stream=stream)
                else:
                    cb.cb_cache_push_residual(plan, src_p, cdt, t, resid_p, cb.CB_BF16, gates_p, cb.CB_BF16,
                                              stream=stream)
        w0, w1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        w0.record(stream)
        for k in range(warmup):
            launch(k)
        w1.record(stream)
        stream.synchronize()
        # at least ~0.3 s of timed steps, so that the clock sampler sees the load
        n = max(steps, int(0.3e3 / max(w0.elapsed_time(w1) / warmup, 1e-3)))
        ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(n)]
        with Clocks(torch.cuda.current_device()) as clk:
            for k in range(n):
                ev[k][0].record(stream)
                launch(k)
                ev[k][1].record(stream)
            stream.synchronize()
        clocks = clk.summary()
        if cb.cb_plan_device_status(plan, stream=stream) != 0:
            raise RuntimeError(f"device status set while timing {name}")
        us = sorted(a.elapsed_time(b) * 1e3 for a, b in ev)
        mean_us = sum(us) / len(us)
        rows.append({"workload": w.name, "variant": label, "step": step, "K": K, "fused_residual": bool(fused),
                     "gated": bool(gated), "bytes_per_step": bytes_step, "us_per_step": round(mean_us, 2),
                     "us_per_step_median": round(us[len(us) // 2], 2),
                     "gbs": round(bytes_step / (mean_us * 1e-6) / 1e9, 2),
                     "frac": round(bytes_step / (mean_us * 1e-6) / 1e9 / peak, 4), "steps": n,
                     "clocks": {"sm_mhz": clocks["sm_mhz"], "reasons": clocks["reasons"]}})
        del resid
    cb.cb_plan_destroy(plan)
    del cache, outs, src
    torch.cuda.empty_cache()
    return rows


def run_reference(args):
    """The oracle on the host cores: each step is a bounded sample of the workload."""
    ws, rank, _ = dist_env()
    if rank != 0:
        return 0
    import numpy as np
    import torch

    import oracle as orc
    from paper_2608_23429_gb300 import workloads as wl
    orc.build()
    w = wl.PRESETS[args.config]()
    n = args.cpu_elems
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    host, wts, ti = sample_host_features(w, torch, wl, orc, n, dev)
    threads = os.cpu_count() or 1
    for _ in range(args.warmup):
        orc.extrapolate([host], wts, orc.BF16, orc.BF16, nthreads=threads)
    times = []
    for _ in range(args.steps):
        t0 = time.perf_counter()
        orc.extrapolate([host], wts, orc.BF16, orc.BF16, nthreads=threads)
        times.append(time.perf_counter() - t0)
    total = sum(times)
    bytes_step = n * (w.K + 1) * 2
    value = bytes_step * args.steps / total / 1e9
    desc = workload_description(w)
    sample = f"{n} contiguous elements of tensor {ti} (K={w.K} bf16 slots + bf16 output) per step"
    line = {
        "impl": "reference", "metric": METRIC, "value": round(value, 3), "unit": "GB/s", "n_gpus": ws,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": round(total / args.steps * 1e3, 3),
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
        "data": "synthetic", "config": dict(desc, sample=sample),
        "cpu_baseline": {"value": round(value, 3), "unit": "GB/s", "cores": threads, "kind": "oracle",
                         "sample": sample},
        "e2e": {"value": round(value, 3), "unit": "GB/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }
    print(json.dumps(line))
    del np
    return 0


def run_ours(args):
    import torch
    import torch.distributed as dist

    ws, rank, local = dist_env()
    if ws > 1:
        torch.cuda.set_device(local)
        dist.init_process_group("nccl", init_method="env://")
    else:
        torch.cuda.set_device(0)
    dev = torch.device("cuda", torch.cuda.current_device())

    import oracle as orc
    from paper_2608_23429_gb300 import build as cbuild
    cbuild.build()
    orc.build()
    from paper_2608_23429_gb300 import chebboost as cb
    from paper_2608_23429_gb300 import workloads as wl

    w = wl.PRESETS[args.config]()
    if args.scale > 1:
        w = wl.scaled(w, args.scale)
    if args.history:
        w.K = args.history
    K = w.K
    tiny = bool(w.explicit_nodes)
    if tiny:  # explicit nodes and targets instead of a schedule; L2-resident, a latency case
        w.timesteps = list(w.explicit_nodes) + list(w.explicit_targets)
        pushed = list(range(len(w.explicit_nodes)))
        targets = list(range(len(pushed), len(w.timesteps)))
        node_t = list(w.explicit_nodes)
    else:
        pushed, targets = pick_window(w, cb)
        node_t = [w.timesteps[s] for s in full_mask(w, cb).nonzero()[0]]
    tensors = [(t.layer, t.branch, t.numel, t.group) for t in w.tensors]
    cdt = cb.CB_BF16 if w.cache_dtype == "bf16" else cb.CB_FP32
    tdt = torch.bfloat16 if w.cache_dtype == "bf16" else torch.float32
    plan = cb.cb_plan_create(node_t, K, tensors, cdt, w.t_min, w.t_max)
    cache = torch.empty(cb.cb_plan_cache_bytes(plan), dtype=torch.uint8, device=dev)
    cb.cb_plan_bind_cache(plan, cache, cache.numel())
    cb.cb_plan_set_option(plan, cb.CB_OPT_KERNEL, {"auto": cb.CB_KERNEL_AUTO, "direct": cb.CB_KERNEL_DIRECT,
                                                   "bulk": cb.CB_KERNEL_BULK}[args.kernel])
    stream = torch.cuda.Stream(device=dev)
    fill_window(torch, cb, wl, w, plan, cdt, pushed, dev, stream)  # full steps up to the timed window
    outs = [torch.empty(t.shape, dtype=tdt, device=dev) for t in w.tensors]
    slot_elems = sum(t.numel for t in w.tensors)
    esz = 2 if w.cache_dtype == "bf16" else 4
    fused = w.fused if args.fused == "auto" else args.fused == "on"
    fused = fused or args.gated  # gates act on the hidden-state update only
    n_groups = cb.cb_plan_num_groups(plan)
    resid = [wl.hidden_state(w, g, dev) for g in range(n_groups)] if fused else None
    resid_elems = sum(w.group_numel(g) for g in range(n_groups)) if fused else 0
    # K slot reads + one output write (+ hidden state read and write)
    bytes_step = slot_elems * esz * (K + 1) + resid_elems * 2 * 2
    t_targets = [w.timesteps[s] for s in targets]
    gates = None
    if args.gated or args.step == "full-fused":
        cb.cb_plan_set_shapes(plan, [t.shape for t in w.tensors])
    if args.gated:  # per-(batch, channel) gates of each branch, bf16
        gg = torch.Generator(device=dev).manual_seed(7)
        gates = [(0.5 * torch.randn(t.shape[0], t.shape[-1], generator=gg, device=dev)).to(torch.bfloat16)
                 for t in w.tensors]
        bytes_step += sum(t.shape[0] * t.shape[-1] * 2 for t in w.tensors) if fused else 0
    kernel_name = "extrapolate_kernel" if args.kernel == "direct" else "extrapolate_bulk_kernel"
    # persistent buffers: their pointer arrays are built once, as a serving loop would
    outs_p = cb.ptr_array(outs)
    resid_p = cb.ptr_array(resid) if resid is not None else None
    gates_p = cb.ptr_array(gates) if gates is not None else None

    def extrapolate_at(t):
        if gates is not None:
            cb.cb_extrapolate_gated(plan, t, outs_p, cdt, resid_p, cb.CB_BF16, gates_p, cb.CB_BF16, stream=stream)
        else:
            cb.cb_extrapolate(plan, t, outs_p, cdt, resid_p, cb.CB_BF16, stream=stream)

    launches_per_step = 1
    if args.step == "skip" and args.launch == "per-block":
        # the same step as one launch per block: each call covers only that
        # block's tensors (and its residual groups)
        blocks = sorted({t.layer for t in w.tensors})
        per_block = []
        for layer in blocks:
            mine = [i for i, t in enumerate(w.tensors) if t.layer == layer]
            groups = {w.tensors[i].group for i in mine if w.tensors[i].group >= 0}
            o = cb.ptr_array([outs[i] if i in mine else None for i in range(len(w.tensors))])
            r = (cb.ptr_array([resid[g] if g in groups else None for g in range(n_groups)])
                 if resid is not None else None)
            g_ = (cb.ptr_array([gates[i] if i in mine else None for i in range(len(w.tensors))])
                  if gates is not None else None)
            per_block.append((o, r, g_))
        launches_per_step = len(per_block)

        def step(k):
            t = t_targets[k % len(t_targets)]
            for o, r, g_ in per_block:
                if g_ is not None:
                    cb.cb_extrapolate_gated(plan, t, o, cdt, r, cb.CB_BF16, g_, cb.CB_BF16, stream=stream)
                else:
                    cb.cb_extrapolate(plan, t, o, cdt, r, cb.CB_BF16, stream=stream)
    elif args.step == "skip":
        def step(k):
            extrapolate_at(t_targets[k % len(t_targets)])
    else:
        # a full step's cache write (row a4), optionally with the fused epilogue:
        # the features come from one generated full step, re-pushed with fresh times
        fdt = torch.float32 if args.feat_dtype == "fp32" else tdt
        src = [wl.trajectory(w, i, w.timesteps[pushed[-1]], pushed[-1], dev, out_dtype=fdt)
               for i in range(len(w.tensors))]
        sdt = cb.CB_FP32 if fdt == torch.float32 else cb.CB_BF16
        bytes_step = slot_elems * (fdt.itemsize + esz)
        if args.step == "full-fused":
            if resid is None:
                resid = [wl.hidden_state(w, g, dev) for g in range(n_groups)]
                resid_elems = sum(w.group_numel(g) for g in range(n_groups))
            bytes_step += resid_elems * 2 * 2 + (sum(t.shape[0] * t.shape[-1] * 2 for t in w.tensors)
                                                 if gates is not None else 0)
        cb.cb_plan_reset(plan)
        t0 = w.timesteps[0]
        span = (w.timesteps[-1] - w.timesteps[0]) / (args.warmup + args.steps + 1)
        times = iter([t0 + span * i for i in range(args.warmup + args.steps + 1)])
        # the fused epilogue runs the skipped-step kernel on a one-entry history
        kernel_name = "push_kernel" if args.step == "full" else kernel_name
        src_p = cb.ptr_array(src)
        resid_p = cb.ptr_array(resid) if resid is not None else None

        def step(k):
            t = next(times)
            if args.step == "full":
                cb.cb_cache_push(plan, src_p, sdt, t, stream=stream)
            else:
                cb.cb_cache_push_residual(plan, src_p, sdt, t, resid_p, cb.CB_BF16, gates_p, cb.CB_BF16,
                                          stream=stream)

    for k in range(args.warmup):
        step(k)
    stream.synchronize()
    if ws > 1:
        dist.barrier()
    torch.cuda.synchronize()
    ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(args.steps)]
    with Clocks(torch.cuda.current_device()) as clk:
        t_all0 = torch.cuda.Event(enable_timing=True)
        t_all1 = torch.cuda.Event(enable_timing=True)
        t_all0.record(stream)
        h0 = time.perf_counter()
        for k in range(args.steps):
            ev[k][0].record(stream)
            step(k)
            ev[k][1].record(stream)
        t_all1.record(stream)
        host_ms = (time.perf_counter() - h0) * 1e3 / args.steps  # submission time per step
        stream.synchronize()
        torch.cuda.synchronize()
        if ws > 1:
            dist.barrier()
    clocks = clk.summary()
    dev_status = cb.cb_plan_device_status(plan, stream=stream)
    if dev_status != 0:
        raise RuntimeError(f"device status {dev_status}: a bounded wait ran out during the timed steps")
    total_ms = t_all0.elapsed_time(t_all1)
    kern_ms = [a.elapsed_time(b) for a, b in ev]
    total_ms = max_over_ranks(total_ms, dev)
    ms_step = total_ms / args.steps
    value = bytes_step * args.steps * ws / (total_ms / 1e3) / 1e9
    avg_kern = sum(kern_ms) / len(kern_ms)
    peak, peak_src = measured_peaks()
    achieved = bytes_step / (avg_kern / 1e3) / 1e9

    # ---- the timed step once more at the first target: its predictions for the
    # largest tensor (the CPU baseline's sample) are checked against the oracle
    check = None
    if rank == 0 and ws == 1 and not args.no_cpu and args.step == "skip" and not tiny:
        ti = max(range(len(w.tensors)), key=lambda k: w.tensors[k].numel)
        extrapolate_at(t_targets[0])
        stream.synchronize()
        n_chk = min(args.cpu_elems, w.tensors[ti].numel)
        check = (ti, outs[ti].reshape(-1)[:n_chk].cpu().view(torch.int16).numpy().view("uint16").copy())

    # ---- the whole online loop of Alg. 1 over the schedule, ring evolving
    sched = None
    if args.step == "skip" and args.schedule_reps > 0 and not tiny:
        sched = run_schedule_loop(args, torch, cb, wl, w, plan, cdt, dev, stream, extrapolate_at, bytes_step)

    # ---- end to end through the public API with host buffers: upload the K
    # cached feature sets from pinned host memory (push), extrapolate, read the
    # predictions back; every copy is inside the timed region.
    e2e = None
    if not args.no_e2e and args.step == "skip" and not args.gated:
        e2e = run_e2e(args, torch, cb, wl, w, plan, cdt, tdt, dev, pushed, t_targets, bytes_step, ws, fused)

    cpu = None
    parity = None
    if check is not None:
        host, wts, ti = sample_host_features(w, torch, wl, orc, args.cpu_elems, dev)
        assert ti == check[0]
        parity = oracle_parity(orc, host, wts, check[1])
        parity["sample"] = (f"{check[1].size} elements of tensor {ti} ({w.tensors[ti].shape}) at the first timed "
                            f"target, predicted by one more launch after the timed steps")
        threads = os.cpu_count() or 1
        gbs, n, reps, el = cpu_oracle_run(w, host, wts, args.cpu_seconds, threads)
        gbs1, _, reps1, el1 = cpu_oracle_run(w, host, wts, args.cpu_seconds / 2, 1)
        cpu = {"value": round(gbs, 3), "unit": "GB/s", "cores": threads, "kind": "oracle",
               "value_1_thread": round(gbs1, 3), "cpu_model": cpu_model(),
               "sample": f"{n} contiguous elements of tensor {ti} at the first timed target, "
                         f"{reps} passes in {el:.1f} s on {threads} threads, {reps1} passes in {el1:.1f} s "
                         f"on 1 thread (fp64 oracle, bf16 in/out)"}

    cb.cb_plan_destroy(plan)
    del outs, resid, cache
    torch.cuda.empty_cache()

    # ---- the other configurations' skipped steps (same launch configuration)
    others = None
    if (rank == 0 and ws == 1 and args.step == "skip" and args.config == "flux" and args.scale == 1
            and not args.history and not args.gated and args.launch == "per-step" and args.kernel == "auto"
            and args.workload_steps > 0):
        peak_now, _ = measured_peaks()
        others = []
        for name, variants in OTHER_WORKLOADS:
            others += time_workload(torch, cb, wl, dev, name, variants, args.workload_steps, 3, peak_now)

    if rank == 0:
        desc = workload_description(w)
        desc.update({"bytes_per_step": bytes_step, "fused_residual": fused, "step": args.step,
                     "gated": bool(args.gated), "targets": targets,
                     "history_steps": pushed[-K:],
                     "l2": ("L2-resident inputs: a latency case (us_per_step), not a bandwidth one" if tiny
                            else "inputs larger than L2 (no flush)"),
                     "launch": ("1 grouped persistent kernel per step" if launches_per_step == 1
                                else f"{launches_per_step} launches per step (one per block)"),
                     "parallelism": f"replicas x{ws}" if ws > 1 else "1 GPU"})
        line = {
            "metric": METRIC, "value": round(value, 2), "unit": "GB/s", "n_gpus": ws, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": round(ms_step, 4),
            "us_per_step": round(ms_step * 1e3, 2), "host_us_per_step": round(host_ms * 1e3, 2),
            "pct_hbm_peak": round(100 * value / ws / peak, 2),
            "pct_nominal_hbm_peak": round(100 * value / ws / NOMINAL_HBM_GBS, 2),
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f32",
            "data": "synthetic", "config": desc,
            "roofline": {"bound": "hbm", "achieved": round(achieved, 2), "peak": peak, "unit": "GB/s",
                         "frac": round(achieved / peak, 4), "peak_source": peak_src,
                         "nominal_peak": NOMINAL_HBM_GBS, "nominal_source": "GB300 HBM3e datasheet, 7.9 TB/s",
                         "traffic": (recorded_traffic(args.config) if args.scale == 1 and args.step == "skip"
                                     and not args.gated else None),
                         "kernel": kernel_name,
                         "avg_launch_us": round(avg_kern * 1e3, 2)},
            "schedule_loop": sched, "parity": parity, "workloads": others,
            "cpu_baseline": cpu, "e2e": e2e, "clocks": clocks, "gpu_launches": args.steps * launches_per_step,
        }
        print(json.dumps(line))
    if ws > 1:
        dist.destroy_process_group()
    return 0


def host_memory_is_device_mapped(ptr: int) -> bool:
    """True when a pinned host pointer is directly usable by kernels (UVA mapping)."""
    import ctypes
    try:
        rt = ctypes.CDLL("libcudart.so.13")
    except OSError:
        return False
    dptr = ctypes.c_void_p()
    rc = rt.cudaHostGetDevicePointer(ctypes.byref(dptr), ctypes.c_void_p(ptr), 0)
    return rc == 0 and dptr.value == ptr


def run_schedule_loop(args, torch, cb, wl, w, plan, cdt, dev, stream, extrapolate_at, bytes_step):
    """Alg. 1's online stage over the whole schedule, `schedule_reps` times from an
    empty history: warm-up and full steps push that step's features (generated
    once, before the timed loops), skipped steps extrapolate with the ring as it
    evolves. Each launch is bracketed by events on the launching stream; only
    the skipped steps count toward the metric, the pushes are timed apart."""
    mask = full_mask(w, cb)
    full = [s for s in range(w.T) if mask[s]]
    skipped = [s for s in range(w.T) if not mask[s]]
    feats = {}
    for s in full:
        ts = [wl.trajectory(w, i, w.timesteps[s], s, dev) for i in range(len(w.tensors))]
        feats[s] = (ts, cb.ptr_array(ts))
    torch.cuda.synchronize()
    per_rep, push_us = [], []
    for _ in range(args.schedule_reps):
        cb.cb_plan_reset(plan)
        evs = []
        for s in range(w.T):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record(stream)
            if mask[s]:
                cb.cb_cache_push(plan, feats[s][1], cdt, w.timesteps[s], stream=stream)
            else:
                extrapolate_at(w.timesteps[s])
            b.record(stream)
            evs.append((s, a, b))
        stream.synchronize()
        if cb.cb_plan_device_status(plan, stream=stream) != 0:
            raise RuntimeError("device status set during the schedule loop")
        ms_skip = sum(a.elapsed_time(b) for s, a, b in evs if not mask[s])
        ms_push = sum(a.elapsed_time(b) for s, a, b in evs if mask[s])
        per_rep.append(ms_skip * 1e3 / len(skipped))
        push_us.append(ms_push * 1e3 / len(full))
    del feats
    torch.cuda.empty_cache()
    best, med = min(per_rep), statistics.median(per_rep)
    return {"reps": args.schedule_reps, "full_steps": len(full), "skipped_steps": len(skipped),
            "us_per_skipped_best": round(best, 2), "us_per_skipped_median": round(med, 2),
            "gbs_best": round(bytes_step / (best * 1e-6) / 1e9, 2),
            "gbs_median": round(bytes_step / (med * 1e-6) / 1e9, 2),
            "us_per_push_mean": round(statistics.mean(push_us), 2),
            "note": "whole schedule per repetition from an empty history; pushes run in the loop, excluded"}


def run_e2e(args, torch, cb, wl, w, plan, cdt, tdt, dev, pushed, t_targets, bytes_step, ws, fused):
    """One skipped step through the public API with every input and output in
    pinned host memory: the K cached feature sets are pushed from the host, the
    step is extrapolated, and the predictions (and hidden states) land in host
    memory. zerocopy: the kernels read and write the pinned buffers over the
    CPU-GPU link (they are device-mapped); copy: explicit staging copies."""
    K = w.K
    nodes = pushed[-K:]
    host_feats = []  # K sets of pinned host features (the full steps' outputs)
    for s in nodes:
        host_feats.append([wl.trajectory(w, i, w.timesteps[s], s, dev).cpu().pin_memory()
                           for i in range(len(w.tensors))])
    host_outs = [torch.empty(t.shape, dtype=tdt).pin_memory() for t in w.tensors]
    n_groups = cb.cb_plan_num_groups(plan)
    host_resid = [wl.hidden_state(w, g, dev).cpu().pin_memory() for g in range(n_groups)] if fused else None
    mode = args.e2e_mode
    if mode == "zerocopy" and not host_memory_is_device_mapped(host_outs[0].data_ptr()):
        mode = "copy"
    # hidden states are read by the bulk kernel's bulk copies, which this
    # bench only drives from device memory: fused steps stage them instead
    if fused:
        mode = "copy"
    stream = torch.cuda.Stream(device=dev)
    slot = sum(t.numel for t in w.tensors) * (2 if w.cache_dtype == "bf16" else 4)
    resid_bytes = sum(w.group_numel(g) for g in range(n_groups)) * 2 if fused else 0
    if mode == "copy":
        dev_feats = [torch.empty(t.shape, dtype=tdt, device=dev) for t in w.tensors]
        outs = [torch.empty(t.shape, dtype=tdt, device=dev) for t in w.tensors]
        resid = [torch.empty_like(r, device=dev) for r in host_resid] if fused else None

    split = []  # per step: (start, pushes done, end) events

    def step(k):
        cb.cb_plan_reset(plan)
        t = t_targets[k % len(t_targets)]
        ev = [torch.cuda.Event(enable_timing=True) for _ in range(3)]
        split.append(ev)
        with torch.cuda.stream(stream):
            ev[0].record(stream)
            if mode == "zerocopy":
                for j, s in enumerate(nodes):
                    cb.cb_cache_push(plan, host_feats[j], cdt, w.timesteps[s], stream=stream)
                ev[1].record(stream)
                cb.cb_extrapolate(plan, t, host_outs, cdt, host_resid, cb.CB_BF16, stream=stream)
                ev[2].record(stream)
                return
            for j, s in enumerate(nodes):
                for d, h in zip(dev_feats, host_feats[j]):
                    d.copy_(h, non_blocking=True)
                cb.cb_cache_push(plan, dev_feats, cdt, w.timesteps[s], stream=stream)
            ev[1].record(stream)
            if fused:
                for d, h in zip(resid, host_resid):
                    d.copy_(h, non_blocking=True)
            cb.cb_extrapolate(plan, t, outs, cdt, resid, cb.CB_BF16, stream=stream)
            for h, o in zip(host_outs, outs):
                h.copy_(o, non_blocking=True)
            if fused:
                for h, d in zip(host_resid, resid):
                    h.copy_(d, non_blocking=True)
            ev[2].record(stream)

    steps = max(1, args.e2e_steps)
    for k in range(2):
        step(k)
    stream.synchronize()
    split.clear()
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    a.record(stream)
    for k in range(steps):
        step(k)
    b.record(stream)
    stream.synchronize()
    ms = max_over_ranks(a.elapsed_time(b) / steps, dev)
    push_ms = sum(e[0].elapsed_time(e[1]) for e in split) / steps
    extrap_ms = sum(e[1].elapsed_time(e[2]) for e in split) / steps
    # the host link's own bound: one large pinned host -> device copy
    link = torch.empty(1 << 30, dtype=torch.uint8).pin_memory()
    link_dev = torch.empty(link.numel(), dtype=torch.uint8, device=dev)
    with torch.cuda.stream(stream):
        link_dev.copy_(link, non_blocking=True)
        a.record(stream)
        for _ in range(3):
            link_dev.copy_(link, non_blocking=True)
        b.record(stream)
    stream.synchronize()
    link_gbs = 3 * link.numel() / (a.elapsed_time(b) / 1e3) / 1e9
    del link, link_dev
    h2d, d2h = K * slot + resid_bytes, slot + resid_bytes
    return {"value": round(bytes_step * ws / (ms / 1e3) / 1e9, 2), "unit": "GB/s",
            "h2d_bytes_per_step": h2d, "d2h_bytes_per_step": d2h,
            "ms_per_step": round(ms, 3), "steps": steps, "mode": mode,
            "push_ms": round(push_ms, 3), "extrapolate_ms": round(extrap_ms, 3),
            "host_link_gbs": round(link_gbs, 1),
            "frac_of_host_link": round((h2d + d2h) / (ms / 1e3) / 1e9 / link_gbs, 4),
            "path": "cb_cache_push x K from host buffers + cb_extrapolate into host buffers"}


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=50)
    ap.add_argument("--warmup", type=int, default=5)
    ap.add_argument("--config", default="flux", choices=["tiny", "dit256", "dit256-k3", "dit512", "pixart", "flux"])
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--fused", default="auto", choices=["auto", "on", "off"],
                    help="add the predictions into the blocks' hidden states (auto: as the workload states)")
    ap.add_argument("--e2e-mode", default="zerocopy", choices=["zerocopy", "copy"],
                    help="e2e host buffers: read/written by the kernels over C2C, or staged by copies")
    ap.add_argument("--step", default="skip", choices=["skip", "full", "full-fused"],
                    help="skip: a skipped step (the metric); full: a full step's cache write; "
                         "full-fused: the cache write with the hidden-state update")
    ap.add_argument("--gated", action="store_true", help="per-(batch, channel) gates on the hidden-state update")
    ap.add_argument("--feat-dtype", default="bf16", choices=["bf16", "fp32"],
                    help="type of the full step's features (--step full / full-fused)")
    ap.add_argument("--kernel", default="auto", choices=["auto", "direct", "bulk"],
                    help="skipped-step kernel variant")
    ap.add_argument("--history", type=int, default=0,
                    help="history size K instead of the workload's own (1..8; changes the schedule's warm-up)")
    ap.add_argument("--scale", type=int, default=1,
                    help="divide every tensor's token count (small cases for profiling only)")
    ap.add_argument("--cpu-seconds", type=float, default=10.0)
    ap.add_argument("--cpu-elems", type=int, default=1 << 24)
    ap.add_argument("--launch", default="per-step", choices=["per-step", "per-block"],
                    help="skipped step as one grouped launch (the design) or one launch per block")
    ap.add_argument("--schedule-reps", type=int, default=5,
                    help="repetitions of the whole schedule loop (0: skip it)")
    ap.add_argument("--e2e-steps", type=int, default=5)
    ap.add_argument("--workload-steps", type=int, default=20,
                    help="timed steps of each other configuration after the headline (0: skip them)")
    ap.add_argument("--no-e2e", action="store_true")
    ap.add_argument("--no-cpu", action="store_true")
    args = ap.parse_args()
    if args.warmup < 3:
        args.warmup = 3
    if args.impl == "reference":
        return run_reference(args)
    return run_ours(args)


if __name__ == "__main__":
    sys.exit(main())
