#!/usr/bin/env python
"""Benchmark of the MoTE FFN-layer forward pass on B200.

  python bench.py [--gpus N] [--steps K] [--warmup W] [--workload c4|c2|c1|c3-T|c5-T|p3-T ...]
                  [--impl ours|reference] [--shared-bits 16|8|4] [--no-sweep]

One "step" is one pass of the whole layer (route, dispatch, Q_a(x), gate/up ternary GEMM, Q_a(h),
down ternary GEMM, shared bf16 FFN, combine) over one batch of synthetic tokens; for the stacked
workloads (c5, p*) one pass of all their layers.  Weights are ternarized once, before the timed
region (offline step).  Prints ONE JSON line.

The headline record is the workload named by --workload (default c4, the largest single layer);
K steps are timed exactly.  At one GPU the line also carries "workloads": a compact record of every
workload of the five configurations (c1, c2, c3 at 1/8/32/64 tokens, c4, c5 at 1/32/2048 tokens),
each timed for about a second.

Multi-GPU: the layer is token-parallel with no exchange step, so every rank holds a full replica
and its own batch (weak scaling, no collective on the data path); the job value is the sum of the
ranks' tokens over the slowest rank's time.  `--gpus N` without a launcher (no WORLD_SIZE in the
environment) starts the N replica processes itself.
"""
from __future__ import annotations

import argparse
import json
import os
import socket
import statistics
import subprocess
import sys
import threading
import time

import numpy as np
import torch

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

from workloads import synth  # noqa: E402

L2_FLUSH_BYTES = 512 << 20
NOMINAL = {"int8_tops": 4500.0, "bf16_tflops": 2250.0, "hbm_gbs": 8000.0}     # datasheet, dense
SWEEP = ["c1", "c2", "c3-1", "c3-8", "c3-32", "c3-64", "c4", "c5-1", "c5-32", "c5-2048"]
SUSTAINED_MIN_MS = 300.0          # a timed region at least this long is compared with sustained peaks


def parse_workload(name: str) -> synth.Workload:
    if "-" in name:                                     # c3-8, c5-32, p3-1, p05-2048 ...
        base, T = name.split("-", 1)
        return synth.WORKLOADS[base].with_T(int(T))
    return synth.WORKLOADS[name]


def workload_label(wl: synth.Workload) -> str:
    return wl.name if wl.T == synth.WORKLOADS[wl.name].T and wl.name not in ("c3", "c5") else f"{wl.name}-{wl.T}"


def measured_peaks():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(path):
        p = json.load(open(path))
        return dict(hbm_gbs=p["hbm_gbs"], bf16_tflops=p["bf16_tflops"],
                    bf16_tflops_sustained=p.get("bf16_tflops_sustained", p["bf16_tflops"]), source="measured")
    return dict(hbm_gbs=6650.0, bf16_tflops=1590.0, bf16_tflops_sustained=1400.0, source="fallback")


class ClockSampler:
    """Samples SM clocks and throttle reasons with nvidia-smi (every 20 ms) and reports the samples
    that fall between begin() and end(): start it early enough (wait_first) that the tool is already
    printing when the timed region begins."""
    FIELDS = ("clocks.sm,clocks.max.sm,clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, index: int):
        self.index, self.proc, self.lines = index, None, []
        self.t_begin = self.t_end = None

    def start(self):
        try:
            self.proc = subprocess.Popen(["nvidia-smi", "-i", str(self.index), "--query-gpu=" + self.FIELDS,
                                          "--format=csv,noheader,nounits", "-lms", "20"],
                                         stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.thread = threading.Thread(target=self._read, daemon=True)
            self.thread.start()
        except OSError:
            self.proc = None
        return self

    def _read(self):
        for line in self.proc.stdout:
            self.lines.append((time.monotonic(), line.strip()))

    def wait_first(self, timeout: float = 1.0):
        """Returns once the first sample has arrived (or after `timeout` seconds)."""
        t0 = time.monotonic()
        while self.proc is not None and not self.lines and time.monotonic() - t0 < timeout:
            time.sleep(0.005)
        return self

    def begin(self):
        self.t_begin = time.monotonic()

    def end(self):
        self.t_end = time.monotonic()

    def stop(self) -> dict:
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        if self.t_end is None:
            self.end()
        time.sleep(0.045)                               # the sample that was being taken when the region ended
        self.proc.terminate()
        self.thread.join(timeout=2)
        parsed = []
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for t, ln in self.lines:
            p = [s.strip() for s in ln.split(",")]
            if len(p) < 6:
                continue
            try:
                parsed.append((t, float(p[0]), float(p[1]),
                               [n for n, v in zip(names, p[2:6]) if v.lower().startswith("active")]))
            except ValueError:
                continue
        # a line is read within a few ms of its sample; samples of the region, else the one nearest to it
        lo = (self.t_begin if self.t_begin is not None else 0.0) + 0.002
        hi = self.t_end + 0.022
        inside = [q for q in parsed if lo <= q[0] <= hi]
        if not inside and parsed:
            mid = 0.5 * (lo + hi)
            inside = [min(parsed, key=lambda q: abs(q[0] - mid))]
        sm = [q[1] for q in inside]
        reasons = sorted({r for q in inside for r in q[3]})
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": inside[-1][2] if inside else None,
                "reasons": reasons, "samples": len(sm)}


def gemms_in_pairs(launches: int, T: int, shared_bits: int) -> bool:
    """Whether a tensor-path layer call of so many launches ran the routed and the shared GEMM of a step as one (most short
    prefills do): router, Q_a(x), gate/up, Q_a(h), down and combine, beside the dispatch scan of more than 512 tokens and
    the code expansion of an RTN-coded shared expert from 768 tokens on.  Apart they are at least one launch more."""
    return launches - (T > 512) - (shared_bits != 16 and T >= 768) == 6


def gemm_ops(wl: synth.Workload, stage: str) -> float:
    """Multiply and add counted as two; int8 in the routed stages, bf16 in the shared ones."""
    rows = wl.T if stage.startswith("shared") else wl.T * wl.k
    return (4.0 if "gateup" in stage else 2.0) * rows * wl.d * wl.f


SHARED_STAGE = {"gateup_ternary": "shared_gateup", "down_ternary": "shared_down"}


def mixed_peak(wl: synth.Workload, stage: str, int8_tops: float, bf16_tflops: float) -> float:
    """The rate of a pair of GEMMs whose routed part runs at the int8 peak and whose shared part at the bf16 one."""
    r, sh = gemm_ops(wl, stage), gemm_ops(wl, SHARED_STAGE[stage])
    return (r + sh) / (r / int8_tops + sh / bf16_tflops)


def stage_work(wl: synth.Workload, stage: str, stream_path: bool, experts_touched: float, shared_bits: int = 16,
               peaks: dict | None = None, paired: bool = False):
    """Algorithmic work of one launch of a stage: (amount, kind), kind 'int8' | 'bf16' | 'mixed' | 'bytes'.
    On the decode path the gate/up and down stages each cover the routed AND the shared expert and
    are bound by the weight bytes they stream: 2-bit codes of the experts that received tokens plus
    the shared matrices (bf16, or RTN codes of shared_bits bits).  In a short prefill whose GEMMs run in pairs they
    cover both too, and are bound by those bytes or by the tensor work of both ('mixed')."""
    P, T, d, f = wl.T * wl.k, wl.T, wl.d, wl.f
    sh_bytes = shared_bits / 8.0
    if stream_path:
        if stage == "gateup_ternary":
            return experts_touched * 2 * f * d / 4 + 2.0 * f * d * sh_bytes, "bytes"
        if stage == "down_ternary":
            return experts_touched * f * d / 4 + f * d * sh_bytes, "bytes"
    # the four GEMMs: tensor work, or -- with few tokens -- the bytes they must move, whichever takes
    # longer at the peaks (a short prefill streams the weights once and is bound by that)
    gemm_bytes = {"gateup_ternary": experts_touched * 2 * f * d / 4 + P * d + P * f * 2.0,
                  "down_ternary": experts_touched * f * d / 4 + P * f + P * d * 4.0,
                  "shared_gateup": 2.0 * f * d * sh_bytes + T * d * 2.0 + T * f * 2.0,
                  "shared_down": f * d * sh_bytes + T * f * 2.0 + T * d * 2.0}
    if stage in gemm_bytes:
        ops, nbytes = gemm_ops(wl, stage), gemm_bytes[stage]
        kind = "bf16" if stage.startswith("shared") else "int8"
        if paired and stage in SHARED_STAGE:
            ops += gemm_ops(wl, SHARED_STAGE[stage])
            nbytes += gemm_bytes[SHARED_STAGE[stage]]
            kind = "mixed"
        if peaks is not None:
            rate = {"int8": peaks["int8_tops"], "bf16": peaks["bf16_tflops"]}
            t_ops = ops / ((mixed_peak(wl, stage, *rate.values()) if kind == "mixed" else rate[kind]) * 1e12)
            if nbytes / (peaks["hbm_gbs"] * 1e9) > t_ops:
                return nbytes, "bytes"
        return ops, kind
    if stage == "quant_x":
        return T * d * 2.0 + P * d * 1.0, "bytes"
    if stage == "quant_h":
        return P * f * 3.0, "bytes"
    if stage == "combine":
        return T * d * (4.0 + 4.0 * wl.k + 2.0), "bytes"
    if stage == "route":
        return T * d * 2.0, "bytes"
    return P * 12.0, "bytes"


def max_over_ranks(values, device, world: int):
    """Every rank passes its own times; all get the slowest rank's (the job is as slow as that)."""
    if world <= 1:
        return list(values)
    import torch.distributed as dist
    t = torch.tensor(list(values), dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return t.tolist()


def job_tokens_per_s(world: int, tokens_per_rank: int, steps: int, total_ms: float) -> float:
    """Whole-job throughput of `world` replicas, each processing its own batch (weak scaling, no
    collective on the data path): all ranks' tokens over the slowest rank's time."""
    return world * tokens_per_rank * steps / (total_ms * 1e-3)


def replica_command(n: int, argv: list[str], port: int) -> list[str]:
    """The launch of n replica processes of this script on one node (what `--gpus n` runs when no
    launcher has set WORLD_SIZE): one rank per GPU, rendezvous on the loopback address."""
    return [sys.executable, "-m", "torch.distributed.run", "--nnodes=1", f"--nproc-per-node={n}",
            "--master-addr", "127.0.0.1", "--master-port", str(port), os.path.abspath(__file__), *argv]


def free_port() -> int:
    with socket.socket() as s:
        s.bind(("127.0.0.1", 0))
        return s.getsockname()[1]


def int8_peak(mote_binding, rank: int, local_rank: int) -> dict:
    """The int8 tensor pipe's speed of light, measured with the library's MMA-only kernel
    (tcgen05.mma.kind::i8 M128 N256 K32 on shared-memory-resident operands): a burst figure (best of
    a few 5 ms launches from idle clocks) and a sustained one (median launch of the second half of
    about a second of back-to-back launches, clocks sampled meanwhile)."""
    burst = mote_binding.mote_int8_mma_peak(800, repeats=5)
    sampler = ClockSampler(local_rank).start().wait_first() if rank == 0 else None
    if sampler:
        sampler.begin()
    long = mote_binding.mote_int8_mma_peak(1600, repeats=80)
    clocks = sampler.stop() if sampler else None
    ms = long["ms_in_order"][len(long["ms_in_order"]) // 2:]
    sustained = long["ops"] / (statistics.median(ms) * 1e-3) / 1e12
    return {"burst_tops": burst["tops_best"], "sustained_tops": sustained, "sustained_clocks": clocks,
            "how": "libmote mote_int8_mma_peak: tcgen05.mma.kind::i8 M128xN256xK32, smem-resident operands, all SMs"}


class LayerSet:
    """The device-resident layers of one base workload (c3, c5 ... share them across batch sizes)."""

    def __init__(self, base: synth.Workload, mote, dev, n_layers: int | None, shared_bits: int, path: str):
        self.base, self.mote, self.dev = base, mote, dev
        self.is_stack = base.n_layers > 1
        n = base.n_layers if n_layers is None else n_layers
        self.master = None
        if self.is_stack:
            # 36 layers of 0.8 G weights each: drawn on the device (minutes on the host); every layer distinct
            self.layers = [mote.MoteLayer.from_device_draws(base.d, base.f, base.E, base.k, base.norm_topk,
                                                            synth.device_draw(base, l, dev), device=dev) for l in range(n)]
        else:
            self.master = synth.master_layer(base)
            self.layers = [mote.MoteLayer.from_master(self.master, device=dev)]
        if shared_bits != 16:                               # offline step: RTN codes of the shared expert
            self.layers = [l.quantize_shared(shared_bits) for l in self.layers]
            torch.cuda.empty_cache()
        if path != "auto":                                  # force one implementation (default: the library picks)
            for l in self.layers:
                l.path = {"simt": mote.PATH_SIMT, "tensor": mote.PATH_TENSOR, "stream": mote.PATH_STREAM}[path]
        self.stack = mote.MoteStack(self.layers) if self.is_stack else None


def measure(ls: LayerSet, wl: synth.Workload, args, steps: int | None, rank: int, local_rank: int, world: int,
            peaks: dict, flush: torch.Tensor) -> dict:
    """Times one workload: `steps` steps exactly (or, steps=None, as many as fill about a second)
    device-resident, then the per-stage times of the same launch configuration over a loop of
    similar length, then the end-to-end loop with host buffers."""
    mote, dev, layers, is_stack = ls.mote, ls.dev, ls.layers, ls.is_stack
    from paper_2506_14435_b200.binding import mote_moe_forward_host, mote_moe_forward_profile
    if is_stack:
        x = synth.device_tokens(wl, dev, stream=rank)
        x_host = x.cpu().pin_memory()
    else:
        x_bits = synth.tokens(wl, stream=rank)
        x_host = torch.from_numpy(x_bits.view(np.int16).copy()).view(torch.bfloat16).pin_memory()
        x = x_host.to(dev)
    out_host = torch.empty_like(x_host).pin_memory()
    out = torch.empty_like(x)
    stream = torch.cuda.current_stream()
    tensor_ok = wl.d % 128 == 0 and wl.f % 128 == 0     # the library's own choice, restated for the work model
    stream_path = (wl.T <= (32 if tensor_ok else 64) and wl.d % 64 == 0 and wl.f % 64 == 0) \
        if args.path == "auto" else args.path == "stream"

    def step_device():
        if is_stack:
            mote.mote_stack_forward(ls.stack, x, out=out)
        else:
            mote.mote_moe_forward(layers[0], x, out=out)

    def step_host():
        if is_stack:                                    # host buffers in and out around the C-ABI call
            x.copy_(x_host, non_blocking=True)
            mote.mote_stack_forward(ls.stack, x, out=out)
            out_host.copy_(out, non_blocking=True)
            torch.cuda.synchronize()
        else:
            mote_moe_forward_host(layers[0], x_host, out_host)      # synchronises the stream itself

    def barrier():
        if world > 1:
            import torch.distributed as dist
            dist.barrier()
        torch.cuda.synchronize()

    def timed_loop(step_fn, n):
        starts = [torch.cuda.Event(enable_timing=True) for _ in range(n)]
        ends = [torch.cuda.Event(enable_timing=True) for _ in range(n)]
        for i in range(n):
            flush.fill_(i & 0xFF)                       # evict L2 between iterations
            starts[i].record(stream)
            step_fn()
            ends[i].record(stream)
        torch.cuda.synchronize()
        return [s.elapsed_time(e) for s, e in zip(starts, ends)]

    # experts that receive tokens (decides the decode path's algorithmic bytes), layer by layer
    touched = []
    cur = x
    for layer in layers:
        taps = layer.alloc_taps(wl.T, names=["offsets"])
        nxt = mote.mote_moe_forward(layer, mote.mote_rms_norm(cur) if is_stack else cur,
                                    residual=cur if is_stack else None, taps=taps)
        layer_launches = mote.lib.mote_last_launch_count()
        touched.append(int((taps["offsets"][1:] - taps["offsets"][:-1] > 0).sum().item()))
        cur = nxt
    experts_touched = sum(touched) / len(touched)

    # ---- device-resident timing
    for _ in range(args.warmup):
        step_device()
    launches_per_step = mote.lib.mote_last_launch_count()
    if steps is None:                                   # fill about a second
        est = statistics.median(timed_loop(step_device, 3))
        steps = int(min(2000, max(10, 1000.0 / max(est + 0.25, 1e-3))))
    step_timed = step_device
    if args.graph:
        # the whole step (every launch of the C-ABI call) captured once in a CUDA graph and replayed:
        # the library only enqueues on the caller's stream, so a caller may capture it
        graph = torch.cuda.CUDAGraph()
        side = torch.cuda.Stream()
        side.wait_stream(stream)
        with torch.cuda.stream(side):
            step_device()
        stream.wait_stream(side)
        torch.cuda.synchronize()
        with torch.cuda.graph(graph, stream=side):
            step_device()
        step_timed = graph.replay
        for _ in range(3):
            step_timed()
    sampler = ClockSampler(local_rank).start().wait_first() if rank == 0 else None
    barrier()
    if sampler:
        sampler.begin()
    per_step = timed_loop(step_timed, steps)
    barrier()
    clocks = sampler.stop() if sampler else None
    total_ms = sum(per_step)

    # ---- per-stage device times of the same launch configuration (events on the launch stream), over a
    # loop about as long as the timed one, so that both run at the same clocks
    stage_acc = {}
    n_prof = max(3, min(steps, int(500.0 / max(total_ms / steps, 1e-3)) + 1))
    sampler = ClockSampler(local_rank).start().wait_first() if rank == 0 else None
    if sampler:
        sampler.begin()
    for i in range(n_prof):
        flush.fill_(i & 0xFF)
        cur = x
        tot = {}
        for layer in layers:
            nxt = torch.empty_like(cur)
            ms = mote_moe_forward_profile(layer, mote.mote_rms_norm(cur) if is_stack else cur, out=nxt,
                                          residual=cur if is_stack else None)
            for k_, v in ms.items():
                tot[k_] = tot.get(k_, 0.0) + v
            cur = nxt
        for k_, v in tot.items():
            stage_acc.setdefault(k_, []).append(v)
    stage_clocks = sampler.stop() if sampler else None
    stage_raw = {k_: statistics.mean(v) for k_, v in stage_acc.items()}    # summed over the layers
    # Every stage time carries the cost of the event pair around it (an event record serialises the
    # chain of programmatic dependent launches): the stages this path folds into a neighbour launch
    # nothing, so what they show is that cost alone.  It is taken off the stages that do launch.
    n_l0 = len(layers)
    paired = not stream_path and gemms_in_pairs(layer_launches, wl.T, args.shared_bits)    # the shared stages launch nothing
    folded = (("dispatch", "quant_x", "shared_gateup", "shared_down", "combine") if stream_path
              else ("shared_gateup", "shared_down") if paired else ("combine",))
    event_ms = min(stage_raw[k_] for k_ in folded) / n_l0
    if event_ms * 1e3 > 4.0:                             # a "folded" stage that did launch: no estimate
        event_ms = 0.0
    stage_ms = {k_: (0.0 if k_ in folded and v / n_l0 - event_ms < 1.5e-3 else max(v - event_ms * n_l0, 0.0))
                for k_, v in stage_raw.items()}

    # ---- end to end: host buffers in and out
    for _ in range(min(args.warmup, 3)):
        step_host()
    barrier()
    e2e_ms = []
    for i in range(steps):
        flush.fill_(i & 0xFF)
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        step_host()
        e2e_ms.append((time.perf_counter() - t0) * 1e3)
    barrier()
    e2e_total = sum(e2e_ms)
    if not bool(torch.isfinite(out.float()).all()):
        raise SystemExit("non-finite layer output: the timing would not be valid")

    total_ms, e2e_total = max_over_ranks([total_ms, e2e_total], dev, world)
    ms_per_step = total_ms / steps
    sustained = total_ms >= SUSTAINED_MIN_MS
    n_l = len(layers)
    dom = max(stage_ms, key=stage_ms.get)
    work, kind = stage_work(wl, dom, stream_path, experts_touched, args.shared_bits, peaks, paired)
    dur_s = stage_ms[dom] * 1e-3 / n_l                  # average duration of one launch of that kernel
    from paper_2506_14435_b200 import traffic
    label = workload_label(wl)
    if kind == "bytes":
        roof = dict(bound="hbm", achieved=work / dur_s / 1e9, peak=peaks["hbm_gbs"], unit="GB/s",
                    peak_source=f"of {peaks['source']} (copy bandwidth)", frac_of_nominal=work / dur_s / 1e9 / NOMINAL["hbm_gbs"])
    elif kind == "int8":
        peak = peaks["int8_tops_sustained"] if sustained else peaks["int8_tops"]
        roof = dict(bound="tensor", achieved=work / dur_s / 1e12, peak=peak, unit="TOP/s",
                    peak_source=("of measured: the library's tcgen05 kind::i8 MMA-only loop, " +
                                 ("sustained figure (timed region of %.0f ms)" % total_ms if sustained else "burst figure")),
                    peak_burst=peaks["int8_tops"], peak_sustained=peaks["int8_tops_sustained"],
                    peak_2x_bf16_burst=2.0 * peaks["bf16_tflops"], frac_of_nominal=work / dur_s / 1e12 / NOMINAL["int8_tops"])
    elif kind == "mixed":
        mix = [peaks["int8_tops_sustained"], peaks["bf16_tflops_sustained"]] if sustained else [peaks["int8_tops"], peaks["bf16_tflops"]]
        roof = dict(bound="tensor", achieved=work / dur_s / 1e12, peak=mixed_peak(wl, dom, *mix), unit="TOP/s",
                    peak_source=f"of measured, routed work at the int8 MMA-only loop's rate and shared work at cuBLAS bf16's "
                                f"({peaks['source']}), " + ("sustained" if sustained else "burst"),
                    frac_of_nominal=work / dur_s / 1e12 / mixed_peak(wl, dom, NOMINAL["int8_tops"], NOMINAL["bf16_tflops"]))
    else:
        peak = peaks["bf16_tflops_sustained"] if sustained else peaks["bf16_tflops"]
        roof = dict(bound="tensor", achieved=work / dur_s / 1e12, peak=peak, unit="TFLOP/s",
                    peak_source=f"of {peaks['source']} (cuBLAS bf16, " + ("sustained)" if sustained else "burst)"),
                    frac_of_nominal=work / dur_s / 1e12 / NOMINAL["bf16_tflops"])
    roof["frac"] = roof["achieved"] / roof["peak"]
    roof["traffic"] = traffic.lookup(label, dom, "stream" if stream_path else "tensor")
    roof["kernel"] = dom
    roof["kernel_ms"] = dur_s * 1e3
    roof["algorithmic_work_per_launch"] = work
    roof["sm_mhz"] = stage_clocks["sm_mhz"] if stage_clocks else None
    weight_bytes = n_l * (experts_touched * 3 * wl.d * wl.f / 4 + 3.0 * wl.d * wl.f * args.shared_bits / 8)
    sm_mhz = clocks["sm_mhz"] if clocks else None
    rec = {
        "workload": label, "wl": wl, "steps": steps, "ms_per_step": ms_per_step, "total_ms": total_ms,
        "us_per_layer": ms_per_step * 1e3 / n_l, "us_per_token": ms_per_step * 1e3 / wl.T,
        "tokens_per_s": job_tokens_per_s(world, wl.T, steps, total_ms),
        "ms_x_sm_mhz": ms_per_step * sm_mhz if sm_mhz else None,
        "layers": n_l, "experts_touched": experts_touched, "stream_path": stream_path,
        "stage_ms": stage_ms, "stage_event_overhead_us": event_ms * 1e3, "roofline": roof,
        "weights_touched_gbs": weight_bytes / (ms_per_step * 1e-3) / 1e9,
        "e2e": {"value": job_tokens_per_s(world, wl.T, steps, e2e_total), "unit": "tokens/s",
                "h2d_bytes_per_step": int(x_host.numel() * 2), "d2h_bytes_per_step": int(out_host.numel() * 2)},
        "gpu_launches": launches_per_step * steps, "launches_per_step": launches_per_step, "clocks": clocks,
    }
    # the two quantities the targets are stated on
    P = wl.T * wl.k
    if stream_path:
        rec["decode_hbm"] = {"weight_bytes_per_step": weight_bytes, "gbs": rec["weights_touched_gbs"],
                             "frac_of_measured": rec["weights_touched_gbs"] / peaks["hbm_gbs"],
                             "frac_of_nominal": rec["weights_touched_gbs"] / NOMINAL["hbm_gbs"],
                             "note": "all weight bytes touched (2-bit codes of the experts that received tokens + the "
                                     "shared expert) over the whole step; the stream kernels cover both"}
    elif not paired:
        t_routed = (stage_ms["gateup_ternary"] + stage_ms["down_ternary"]) * 1e-3 / n_l
        t_with_q = t_routed + stage_ms["quant_h"] * 1e-3 / n_l
        ops = 6.0 * wl.d * wl.f * P
        pk = peaks["int8_tops_sustained"] if sustained else peaks["int8_tops"]
        rec["routed_gemms"] = {"int8_ops": ops, "ms": t_routed * 1e3, "tops": ops / t_routed / 1e12,
                               "frac_of_measured": ops / t_routed / 1e12 / pk,
                               "frac_of_nominal": ops / t_routed / 1e12 / NOMINAL["int8_tops"],
                               "frac_of_measured_with_quant_h": ops / t_with_q / 1e12 / pk}
    return rec


def compact(rec: dict) -> dict:
    r = rec["roofline"]
    out = {"workload": rec["workload"], "T": rec["wl"].T, "layers": rec["layers"], "steps": rec["steps"],
           "path": "stream" if rec["stream_path"] else "tensor",
           "ms_per_step": round(rec["ms_per_step"], 5), "us_per_layer": round(rec["us_per_layer"], 2),
           "tokens_per_s": round(rec["tokens_per_s"], 1), "ms_x_sm_mhz": rec["ms_x_sm_mhz"],
           "sm_mhz": rec["clocks"]["sm_mhz"] if rec["clocks"] else None,
           "dominant": r["kernel"],
           "roofline": {k: r[k] for k in ("bound", "achieved", "peak", "unit", "frac", "frac_of_nominal", "kernel_ms",
                                          "algorithmic_work_per_launch", "traffic")},
           "weights_touched_gbs": round(rec["weights_touched_gbs"], 1),
           "e2e_tokens_per_s": round(rec["e2e"]["value"], 1), "launches_per_step": rec["launches_per_step"]}
    for k in ("decode_hbm", "routed_gemms"):
        if k in rec:
            out[k] = {a: b for a, b in rec[k].items() if a != "note"}
    return out


def run_ours(args):
    rank = int(os.environ.get("RANK", 0))
    local_rank = int(os.environ.get("LOCAL_RANK", 0))
    world = int(os.environ.get("WORLD_SIZE", 1))
    if not torch.cuda.is_available():
        raise SystemExit("bench.py needs a CUDA device: there is no CPU fallback for the product path")
    torch.cuda.set_device(local_rank)
    dev = torch.device("cuda", local_rank)
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl", device_id=dev)
    import paper_2506_14435_b200 as mote
    from paper_2506_14435_b200 import binding

    peaks = measured_peaks()
    i8 = int8_peak(binding, rank, local_rank)
    peaks["int8_tops"], peaks["int8_tops_sustained"] = i8["burst_tops"], i8["sustained_tops"]
    flush = torch.empty(L2_FLUSH_BYTES, dtype=torch.uint8, device=dev)

    wl = parse_workload(args.workload)
    base = synth.WORKLOADS[wl.name]
    ls = LayerSet(base, mote, dev, args.layers, args.shared_bits, args.path)
    head = measure(ls, wl, args, args.steps, rank, local_rank, world, peaks, flush)

    # the headline's own record also serves the sweep when its timed region was long enough to count as
    # sustained; a short one (the driver's 20 steps of c4 are 40 ms) is measured again for about a second
    records = {head["workload"]: head} if head["total_ms"] >= SUSTAINED_MIN_MS else {}
    sweep = world == 1 and not args.no_sweep and args.shared_bits == 16 and args.path == "auto" and not args.graph \
        and args.layers is None
    cb = None
    if world == 1 and rank == 0:
        master, x_bits = ls.master, None
        if ls.is_stack:                                     # the oracle needs host-drawn weights: layer 0, scaled by the depth
            master = synth.master_layer(wl)
        x_bits = synth.tokens(wl)
        cb = cpu_baseline(wl, master, x_bits, budget_s=12.0, shared_bits=args.shared_bits)
        if ls.is_stack:
            cb["value"] /= head["layers"]
            cb["sample"] += f"; one layer timed, value divided by the {head['layers']} layers of the stack"
        del master
    if sweep:
        for name in sorted(SWEEP, key=lambda n: parse_workload(n).name != wl.name):     # the resident layers first
            w = parse_workload(name)
            if workload_label(w) in records:
                continue
            if w.name != ls.base.name:
                del ls
                torch.cuda.empty_cache()
                ls = LayerSet(synth.WORKLOADS[w.name], mote, dev, None, 16, "auto")
            records[workload_label(w)] = measure(ls, w, args, None, rank, local_rank, world, peaks, flush)
    if rank != 0:
        if world > 1:
            import torch.distributed as dist
            dist.destroy_process_group()
        return

    decode = wl.T <= 64
    line = {
        "metric": "MoTE layer tokens/sec (prefill)" if not decode else "MoTE layer tokens/sec (decode batch)",
        "value": head["tokens_per_s"], "unit": "tokens/s", "n_gpus": world, "steps": args.steps, "warmup": args.warmup,
        "ms_per_step": head["ms_per_step"], "us_per_layer": head["us_per_layer"],
        "us_per_token": head["us_per_token"], "ms_x_sm_mhz": head["ms_x_sm_mhz"], "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "int8xint2->int32 routed, bf16 shared" + (
            "" if args.shared_bits == 16 else f" (weights RTN int{args.shared_bits}, weight-only)"), "data": "synthetic",
        "config": {"workload": head["workload"], "d": wl.d, "f": wl.f, "E": wl.E, "k": wl.k, "T_per_gpu": wl.T,
                   "layers": head["layers"], "experts_touched_per_layer": head["experts_touched"],
                   "shared_bits": args.shared_bits, "path": args.path,
                   "launch": "CUDA graph replay of the step" if args.graph else "direct launches",
                   "pre_norm": "rms, eps 1e-6, unit gain" if ls.is_stack or wl.n_layers > 1 else "none (the caller's)",
                   "l2": "flushed between timed iterations (512 MiB write)", "parallelism": f"replicas x{world}"},
        "stage_ms": head["stage_ms"], "stage_event_overhead_us": head["stage_event_overhead_us"],
        "roofline": head["roofline"],
        "weights_touched_gbs": head["weights_touched_gbs"],
        "e2e": head["e2e"], "gpu_launches": head["gpu_launches"], "clocks": head["clocks"],
        "int8_peak": i8,
    }
    for k in ("decode_hbm", "routed_gemms"):
        if k in head:
            line[k] = head[k]
    if cb is not None:
        line["cpu_baseline"] = cb
    if sweep:
        line["workloads"] = [compact(records[workload_label(parse_workload(n))]) for n in SWEEP]
    print(json.dumps(line))
    if world > 1:
        import torch.distributed as dist
        dist.destroy_process_group()


def cpu_baseline(wl, master, x_bits, budget_s: float, n_tokens: int | None = None, shared_bits: int = 16):
    """The oracle as it stands, on the host cores, on a bounded sample of the same workload: a
    short probe fixes the sample size so that the timed run takes about `budget_s` seconds."""
    from oracle import mote_oracle as O
    layer_or = O.build_layer(master)                     # offline step, not timed (as on the GPU)
    if shared_bits != 16:
        layer_or = O.quantize_shared(layer_or, shared_bits)
    n0 = min(wl.T, 32)
    t0 = time.perf_counter()
    O.moe_forward(layer_or, x_bits, token_subset=np.arange(n0))
    rate = n0 / max(time.perf_counter() - t0, 1e-6)
    n = n_tokens or int(min(wl.T, max(n0, rate * budget_s)))
    sub = np.arange(n)
    passes, dt = 0, 0.0
    while True:                                          # whole passes over the sample until the budget is used
        t0 = time.perf_counter()
        O.moe_forward(layer_or, x_bits, token_subset=sub)
        dt += time.perf_counter() - t0
        passes += 1
        if dt >= 0.8 * budget_s or dt + dt / passes > 2.5 * budget_s:
            break
    return {"value": n * passes / dt, "unit": "tokens/s", "cores": torch.get_num_threads(), "kind": "oracle",
            "sample": f"first {n} of {wl.T} tokens of {wl.name} (routing for all tokens), {passes} pass(es), {dt:.2f} s",
            "seconds": dt}


def run_reference(args):
    rank = int(os.environ.get("RANK", 0))
    if rank != 0:
        return
    wl = parse_workload(args.workload)
    master = synth.master_layer(wl)
    from oracle import mote_oracle as O
    layer_or = O.build_layer(master)
    del master
    if args.shared_bits != 16:
        layer_or = O.quantize_shared(layer_or, args.shared_bits)
    x_bits = synth.tokens(wl)
    n = min(wl.T, 128 if wl.d * wl.f < 8e6 else 32)
    sub = np.arange(n)
    for _ in range(args.warmup):
        O.moe_forward(layer_or, x_bits, token_subset=sub)
    t0 = time.perf_counter()
    for _ in range(args.steps):
        O.moe_forward(layer_or, x_bits, token_subset=sub)
    dt = time.perf_counter() - t0
    val = n * args.steps / dt
    if wl.n_layers > 1:
        val /= wl.n_layers                                  # one layer timed; a step of the stack is n_layers of them
    decode = wl.T <= 64
    print(json.dumps({
        "impl": "reference",
        "metric": "MoTE layer tokens/sec (prefill)" if not decode else "MoTE layer tokens/sec (decode batch)",
        "value": val, "unit": "tokens/s", "n_gpus": int(os.environ.get("WORLD_SIZE", 1)), "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": dt / args.steps * 1e3, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "fp64 / exact integers", "data": "synthetic",
        "config": {"workload": workload_label(wl), "d": wl.d, "f": wl.f, "E": wl.E, "k": wl.k, "T_per_gpu": wl.T,
                   "layers": wl.n_layers, "shared_bits": args.shared_bits},
        "cpu_baseline": {"value": val, "unit": "tokens/s", "cores": torch.get_num_threads(), "kind": "oracle",
                         "sample": f"each step = first {n} of {wl.T} tokens of {wl.name}" +
                                   (f", one layer (value divided by the {wl.n_layers} layers)" if wl.n_layers > 1 else "")},
        "e2e": {"value": val, "unit": "tokens/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }))


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=None,
                    help="timed steps of the headline workload (default: 400 for ours, about a second at c4; 3 for the reference)")
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--workload", default="c4")
    ap.add_argument("--layers", type=int, default=None, help="layers of a stacked workload (c5-T: default 36)")
    ap.add_argument("--shared-bits", type=int, default=16, choices=[16, 8, 4],
                    help="storage of the shared expert: bf16, or RTN INT8 / INT4 codes (Section 4.3)")
    ap.add_argument("--path", default="auto", choices=["auto", "simt", "tensor", "stream"],
                    help="implementation of the layer (auto: the library's own choice per shape)")
    ap.add_argument("--graph", action="store_true",
                    help="time the step as a CUDA graph replay (captured once from the same C-ABI call)")
    ap.add_argument("--no-sweep", action="store_true", help="leave out the records of the other workloads")
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    args = ap.parse_args()
    if args.steps is None:
        args.steps = 400 if args.impl == "ours" else 3
    args.warmup = max(args.warmup, 3) if args.impl == "ours" else args.warmup
    if args.gpus > 1 and "WORLD_SIZE" not in os.environ:
        # no launcher: start the replicas ourselves, one process per GPU (the reference arm has one rank's work)
        if args.impl == "ours" and torch.cuda.device_count() < args.gpus:
            raise SystemExit(f"--gpus {args.gpus}: only {torch.cuda.device_count()} CUDA device(s) visible")
        raise SystemExit(subprocess.call(replica_command(args.gpus, sys.argv[1:], free_port())))
    if args.impl == "reference":
        run_reference(args)
    else:
        run_ours(args)


if __name__ == "__main__":
    main()
