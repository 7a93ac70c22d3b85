#!/usr/bin/env python
"""Benchmark of the int8 convolution hot path on B200.

One "step" is one pass of the whole path (activation layout rewrite, MMA kernel with fused
shift/clip epilogue, split-reduction finish when the embedding has one) over a batch of G
independent instances of the headline convolution shape, each instance with its own input,
weight, output and scratch buffers, so that every launch reads cold data (G x working set is
larger than the 126 MB L2).  The G launches of a step are captured once in a CUDA graph; since
the instances share nothing, they are dealt onto `--streams` branches of that graph so that kernels
of different instances overlap on the GPU (throughput of the batch is what `value` reports), and the
embedding is chosen by the planner's concurrent timed selection.  `--streams 1` runs one call after
the other; `per_config` reports both series for every shape.

Prints ONE JSON line (rank 0).  `--impl reference` times the CPU oracle instead.
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

from paper_2104_04731_b200.synth import CONFIGS, REPORT_EXTRA, ConvShape, int8_uniform  # noqa: E402

METRIC = "int8 conv TOPS (2*N*K*P*Q*C*R*S / device time)"
UNIT = "TOPS"
HEADLINE = 4  # index into CONFIGS: the large-batch, compute-bound 3x3 stride-2 shape
L2_BYTES = 126 * 1024 * 1024
INT8_TO_BF16_RATIO = 2.0  # nominal dense int8 : bf16 tensor throughput on B200 (4.5 : 2.25 PFLOP/s)

# DRAM traffic of the dominant kernel from an ncu capture (dram__bytes_read.sum + dram__bytes_write.sum
# per launch), valid only for the sources it was taken on (the kernel and the host code that picks its
# tile, stage count and launch shape); see profiles/.
KERNEL_SOURCES = ("conv_mma.cu", "conv_mma_pair.cu", "conv_mma_common.cuh", "conv_mma_cluster.cuh", "api.cpp", "planner.cpp", "tma.cpp", "b2c_internal.h")


def kernel_sources_sha1():
    return hashlib.sha1(b"".join(open(os.path.join(ROOT, "paper_2104_04731_b200", "csrc", f), "rb").read()
                                 for f in KERNEL_SOURCES)).hexdigest()
# (per tile shape "tile_m x tile_n" of the channel-pack map on the headline shape)
NCU_TRAFFIC = {"conv_mma_sha1": "b71f4b0e53f919cb076ee4a40d053814ff74a945",
               "bytes_per_launch": {"256x256": 2839680, "256x128": 2839552, "128x256": 2860800}}


def load_peaks():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(path):
        p = json.load(open(path))
        return {"hbm_gbs": float(p["hbm_gbs"]), "bf16_tflops": float(p["bf16_tflops"]),
                "bf16_tflops_sustained": float(p.get("bf16_tflops_sustained", p["bf16_tflops"])), "source": "measured"}
    return {"hbm_gbs": 6650.0, "bf16_tflops": 1590.0, "bf16_tflops_sustained": 1400.0, "source": "fallback"}


def roofline_time_us(cfg: ConvShape, peaks) -> tuple:
    """(t_roof_us, bound) with t = max(useful ops / int8 peak, algorithmic bytes / HBM bandwidth)."""
    t_c = 2.0 * cfg.macs / (peaks["bf16_tflops"] * INT8_TO_BF16_RATIO * 1e12) * 1e6
    t_m = cfg.algorithmic_bytes / (peaks["hbm_gbs"] * 1e9) * 1e6
    return (t_c, "tensor") if t_c >= t_m else (t_m, "hbm")


class ClockSampler:
    """Samples SM clocks and throttle reasons with nvidia-smi while the timed region runs."""

    Q = ("clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
         "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, index: int):
        self.index = index
        self.proc = None
        self.lines = []

    def start(self):
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", "-i", str(self.index), "--query-gpu=" + self.Q, "--format=csv,noheader,nounits", "-lms", "100"],
                stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.t = threading.Thread(target=self._read, daemon=True)
            self.t.start()
        except Exception:
            self.proc = None

    def _read(self):
        for line in self.proc.stdout:
            self.lines.append(line.strip())

    def stop(self):
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
            f = [t.strip() for t in ln.split(",")]
            if len(f) < 7:
                continue
            try:
                sm.append(float(f[0]))
                mx.append(float(f[1]))
            except ValueError:
                continue
            for name, v in zip(names, f[3:7]):
                if v.lower().startswith("active"):
                    reasons.add(name)
        return {"sm_mhz": float(np.median(sm)) if sm else None, "sm_max_mhz": max(mx) if mx else None,
                "samples": len(sm), "reasons": sorted(reasons)}


# ----------------------------------------------------------------------------------------------------
# GPU arm
# ----------------------------------------------------------------------------------------------------
class Instances:
    """G independent instances of one shape, each with its own plan (own packed weights) and buffers."""

    def __init__(self, b2c, torch, cfg: ConvShape, G: int, policy_or_id: int, in_layout=0, prepacked=None):
        self.cfg, self.G, self.in_layout = cfg, G, in_layout
        d = b2c.make_desc(cfg.N, cfg.C, cfg.H, cfg.W, cfg.K, cfg.R, cfg.S, cfg.stride, cfg.pad, cfg.dilation, cfg.shift,
                          in_layout, b2c.LAYOUT_NCHW, cfg.out_mode)
        first = b2c.Plan(d, policy_or_id)
        self.emb = first.info()
        self.plans = [first] + [b2c.Plan(d, self.emb.id) for _ in range(G - 1)]
        oshape = (cfg.N, cfg.K, cfg.P, cfg.Q)
        xh, wh = cfg.tensors()
        if in_layout == 1:
            xh = np.ascontiguousarray(xh.transpose(0, 2, 3, 1))
        self.x, self.y32, self.y8, self.ws = [], [], [], []
        for i, p in enumerate(self.plans):
            # distinct memory per instance; the values repeat (timing does not depend on them)
            self.x.append(torch.from_numpy(xh).cuda())
            p.set_weights(torch.from_numpy(wh).cuda())
            self.y32.append(torch.empty(oshape, dtype=torch.int32, device="cuda") if cfg.out_mode & 1 else None)
            self.y8.append(torch.empty(oshape, dtype=torch.int8, device="cuda") if cfg.out_mode & 2 else None)
            self.ws.append(torch.empty(max(16, p.workspace_bytes()), dtype=torch.uint8, device="cuda"))
        torch.cuda.synchronize()
        self.launches_per_instance = self._count_launches()
        self.graph = None
        self.side = None
        self.streams = 1

    def _count_launches(self):
        """Kernels of this library per call: layout rewrite (if any) + MMA kernel + split finish (if any)."""
        e, c = self.emb, self.cfg
        n = 1
        if e.variant in (1, 4, 5, 6, 8, 9) or (e.variant in (0, 7) and not (self.in_layout == 1 and c.C % 32 == 0)):
            n += 1
        cluster = (e.map_m != 2 and e.variant not in (6, 7, 8, 9) and e.split_k in (2, 4, 8) and e.tile_n >= 32 * e.split_k
                   and (e.variant in (0, 1, 4, 5) or e.tile_n <= 128))  # the swapped map (map_m = k) and the phase pack never cluster
        if e.split_k > 1 and not cluster and (c.out_mode & 2):
            n += 1  # a split reduction that is not a cluster goes through memory and needs the finish kernel
        return n

    def run_all(self, torch=None, streams=1):
        """Enqueues every instance once.  With streams > 1 the instances (which share no buffer and no
        plan) are dealt round-robin onto that many side streams forked from, and joined back into, the
        current stream, so that kernels of different instances may run side by side on the GPU."""
        if streams <= 1:
            for i, p in enumerate(self.plans):
                p.run(self.x[i], self.y32[i], self.y8[i], self.ws[i])
            return
        if self.side is None or len(self.side) != streams:
            self.side = [torch.cuda.Stream() for _ in range(streams)]
        cur = torch.cuda.current_stream()
        fork = torch.cuda.Event()
        fork.record(cur)
        for s in self.side:
            s.wait_event(fork)
        for i, p in enumerate(self.plans):
            p.run(self.x[i], self.y32[i], self.y8[i], self.ws[i], stream=self.side[i % streams])
        for s in self.side:
            join = torch.cuda.Event()
            join.record(s)
            cur.wait_event(join)

    def capture(self, torch, repeat=1, streams=1):
        self.run_all(torch, streams)
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            for _ in range(repeat):
                self.run_all(torch, streams)
        self.graph = g
        self.streams = streams

    def step(self):
        if self.graph is not None:
            self.graph.replay()
        else:
            self.run_all()

    def verify(self, which=(0, -1)):
        """Compares the outputs the last step left in the given instances with the CPU oracle, element by
        element (every instance has the same seeded input and weights)."""
        import oracle
        import torch

        c = self.cfg
        x, w = c.tensors()
        ref32, ref8 = oracle.conv2d_int8(x, w, c.stride, c.pad, c.dilation, c.shift)
        torch.cuda.synchronize()
        for i in which:
            if self.y32[i] is not None and not np.array_equal(self.y32[i].cpu().numpy(), ref32):
                return False
            if self.y8[i] is not None and not np.array_equal(self.y8[i].cpu().numpy(), ref8):
                return False
        return True

    def check_status(self, b2c):
        for p in self.plans:
            s = p.device_status()
            if s != 0:
                raise RuntimeError("device status " + b2c.status_string(s))

    def destroy(self):
        self.graph = None
        for p in self.plans:
            p.destroy()


def max_over_ranks(torch, dist, value: float, device) -> float:
    """MAX of a per-rank scalar over the process group (the job is as slow as its slowest rank)."""
    if dist is None:
        return float(value)
    t = torch.tensor([value], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


LAST_STEP_MS = []  # per-step device times of the most recent time_steps call (this rank)


def time_steps(torch, fn, steps, warmup, dist=None, min_warm_s=0.2):
    for _ in range(warmup):
        fn()
    # a step is a fraction of a millisecond: keep warming until the clocks have had time to ramp
    t_end = time.perf_counter() + min_warm_s
    while time.perf_counter() < t_end:
        fn()
        torch.cuda.synchronize()
    torch.cuda.synchronize()
    if dist is not None:
        dist.barrier()
    torch.cuda.synchronize()
    ev = [torch.cuda.Event(enable_timing=True) for _ in range(steps + 1)]
    ev[0].record()
    for i in range(steps):
        fn()
        ev[i + 1].record()
    torch.cuda.synchronize()
    LAST_STEP_MS[:] = [ev[i].elapsed_time(ev[i + 1]) for i in range(steps)]
    ms = max_over_ranks(torch, dist, ev[0].elapsed_time(ev[steps]), "cuda")
    if dist is not None:
        dist.barrier()
    return ms


def instances_for(cfg, min_bytes=8 * L2_BYTES, lo=8, hi=256):
    per = cfg.algorithmic_bytes + cfg.N * cfg.C * cfg.H * cfg.W  # plus a packed copy of the input
    return int(max(lo, min(hi, -(-min_bytes // per))))


def measure_shape(b2c, torch, cfg, steps, warmup, peaks, policy, dist=None, graph=True, streams=1):
    """Combined (whole path, NCHW in), Op (MMA kernel alone on a resident packed operand) and Transf.,
    one call after the other on one stream (latency series); and the same batch of instances dealt
    onto `streams` graph branches with the embedding chosen for throughput (concurrent series)."""
    G = instances_for(cfg)
    inst = Instances(b2c, torch, cfg, G, policy)
    if graph:
        inst.capture(torch)
    ms = time_steps(torch, inst.step, steps, warmup, dist)
    inst.check_status(b2c)
    verified = inst.verify()
    per_call_us = ms * 1e3 / (steps * G)
    st_sorted = sorted(LAST_STEP_MS)
    emb = inst.emb.as_dict()
    launches = inst.launches_per_instance
    inst.destroy()
    # Warm series: the same instance relaunched on the same buffers (L2-resident), and the paper's
    # Table-3 split: Op. = MMA kernel alone on an already rewritten operand, Transf. = the rest.
    warm = Instances(b2c, torch, cfg, 1, emb["id"])
    warm.capture(torch, repeat=20)
    ms_w = time_steps(torch, warm.step, 10, 3, None, 0.0)
    warm.destroy()
    op = op_only(b2c, torch, cfg, emb["variant"], emb["tile_n"], emb["split_k"], steps, warmup, graph, 1, emb["map_m"],
                 emb["tile_m"])
    t_roof, bound = roofline_time_us(cfg, peaks)
    keys = ("id", "variant_name", "map_m", "tile_m", "tile_n", "split_k", "workspace_bytes", "o_mac", "o_data", "device_us")
    res = {
        "shape": cfg.name, "instances": G, "warm_us": ms_w * 1e3 / (10 * 20),
        "combined_us_median": st_sorted[len(st_sorted) // 2] * 1e3 / G, "combined_us_min": st_sorted[0] * 1e3 / G,
        "op_us": op["us"] if op else None, "transf_us": max(0.0, per_call_us - op["us"]) if op else None, "cold": bool(G * cfg.algorithmic_bytes >= L2_BYTES), "combined_us": per_call_us, "tops": 2.0 * cfg.macs / (per_call_us * 1e-6) / 1e12,
        "roofline_us": t_roof, "bound": bound, "roofline_frac": t_roof / per_call_us,
        "embedding": {k: emb[k] for k in keys},
        "launches_per_call": launches, "verified": verified,
    }
    if graph and streams > 1:
        conc = Instances(b2c, torch, cfg, G, b2c.POLICY_AUTO_TIMED_CONCURRENT)
        conc.capture(torch, streams=streams)
        ms_c = time_steps(torch, conc.step, steps, warmup, dist)
        conc.check_status(b2c)
        res["concurrent_verified"] = conc.verify()
        us_c = ms_c * 1e3 / (steps * G)
        emb_c = conc.emb.as_dict()
        conc.destroy()
        res["concurrent"] = {"streams": streams, "us_per_call": us_c, "tops": 2.0 * cfg.macs / (us_c * 1e-6) / 1e12,
                             "roofline_frac": t_roof / us_c, "embedding": {k: emb_c[k] for k in keys}}
    return res


def scaled_shape(cfg: ConvShape, peaks, target_us=50.0) -> ConvShape:
    """Same per-image shape with the batch scaled until the roofline time reaches `target_us`."""
    t, _ = roofline_time_us(cfg, peaks)
    mult = max(1, int(np.ceil(target_us / t)))
    return ConvShape(cfg.name + "_xN%d" % (cfg.N * mult), cfg.N * mult, cfg.C, cfg.H, cfg.W, cfg.K, cfg.R, cfg.S,
                     cfg.stride, cfg.pad, cfg.dilation, cfg.shift, cfg.out_mode)


def measure_scaled(b2c, torch, cfg, peaks, steps=10):
    """Secondary series: one large-batch problem per launch (working set beyond L2), whole path; and,
    where the channel count allows it, the same problem with NHWC input (the layout a previous int8
    layer of this library leaves behind), for which the channel-pack map needs no rewrite."""
    big = scaled_shape(cfg, peaks)
    t_roof, bound = roofline_time_us(big, peaks)

    def one(in_layout):
        d = b2c.make_desc(big.N, big.C, big.H, big.W, big.K, big.R, big.S, big.stride, big.pad, big.dilation, big.shift,
                          in_layout, 0, big.out_mode)
        plan = b2c.Plan(d, b2c.POLICY_AUTO_TIMED)
        emb = plan.info()
        shape = (big.N, big.C, big.H, big.W) if in_layout == 0 else (big.N, big.H, big.W, big.C)
        x = torch.randint(-128, 128, shape, dtype=torch.int8, device="cuda")
        w = torch.randint(-128, 128, (big.K, big.C, big.R, big.S), dtype=torch.int8, device="cuda")
        oshape = (big.N, big.K, big.P, big.Q)
        y32 = torch.empty(oshape, dtype=torch.int32, device="cuda") if big.out_mode & 1 else None
        y8 = torch.empty(oshape, dtype=torch.int8, device="cuda") if big.out_mode & 2 else None
        ws = torch.empty(max(16, plan.workspace_bytes()), dtype=torch.uint8, device="cuda")
        plan.set_weights(w)
        ms = time_steps(torch, lambda: plan.run(x, y32, y8, ws), steps, 3, None, 0.05)
        per = sorted(LAST_STEP_MS)
        # the two halves on their own (the paper's Transf. and Op. columns), and the layout kernel's achieved
        # bandwidth on the bytes it reads and writes
        data_b, _ = plan.footprint()
        halves = {}
        if data_b:
            ms_t = time_steps(torch, lambda: plan.rewrite_activations(x, ws), steps, 3, None, 0.0)
            ms_o = time_steps(torch, lambda: plan.run_rewritten(x, y32, y8, ws), steps, 3, None, 0.0)
            moved = x.numel() + data_b
            halves = {"transf_us": ms_t * 1e3 / steps, "op_us": ms_o * 1e3 / steps, "transf_bytes": moved,
                      "transf_gbs": moved / (ms_t * 1e-3 / steps) / 1e9,
                      "transf_frac_of_copy_bandwidth": moved / (ms_t * 1e-3 / steps) / 1e9 / peaks["hbm_gbs"]}
        st = plan.device_status()
        plan.destroy()
        if st != 0:
            raise RuntimeError("device status " + b2c.status_string(st))
        us = ms * 1e3 / steps
        return {"us": us, "us_median": per[len(per) // 2] * 1e3, "us_min": per[0] * 1e3, **halves,
                "tops": 2.0 * big.macs / (us * 1e-6) / 1e12, "roofline_frac": t_roof / us,
                "embedding": {"variant": b2c.VARIANT_NAMES[emb.variant], "tile_m": emb.tile_m, "tile_n": emb.tile_n,
                              "split_k": emb.split_k, "swapped": emb.map_m == b2c.AXIS_K}}

    res = {"shape": big.name, "roofline_us": t_roof, "bound": bound, "bytes": big.algorithmic_bytes}
    res.update(one(0))
    if big.C % 32 == 0:
        res["nhwc_input"] = one(1)
    return res


def op_only(b2c, torch, cfg, emb_variant, tile_n, split_k, steps, warmup, graph=True, streams=1, map_m=1, tile_m=128):
    """Device time of the MMA kernel alone: same embedding but with the layout rewrite already done
    (channel-pack map: NHWC input with padded channels; stencil-unroll in-kernel: unchanged)."""
    if emb_variant in (0, 7) and cfg.C % 32 == 0:
        d = b2c.make_desc(cfg.N, cfg.C, cfg.H, cfg.W, cfg.K, cfg.R, cfg.S, cfg.stride, cfg.pad, cfg.dilation, cfg.shift, 1, 0, cfg.out_mode)
        ids = [e.id for e in b2c.enumerate_embeddings(d)
               if e.variant == emb_variant and e.tile_n == tile_n and e.split_k == split_k and e.map_m == map_m
               and e.tile_m == tile_m]
        if not ids:
            return None
        G = instances_for(cfg)
        inst = Instances(b2c, torch, cfg, G, ids[0], in_layout=1)
    elif emb_variant in (2, 3):
        # stencil unroll inside the kernel: there is no separate rewrite, the kernel is the whole path
        d = b2c.make_desc(cfg.N, cfg.C, cfg.H, cfg.W, cfg.K, cfg.R, cfg.S, cfg.stride, cfg.pad, cfg.dilation, cfg.shift, 0, 0, cfg.out_mode)
        ids = [e.id for e in b2c.enumerate_embeddings(d)
               if e.variant == emb_variant and e.tile_n == tile_n and e.split_k == split_k and e.map_m == map_m
               and e.tile_m == tile_m]
        G = instances_for(cfg)
        inst = Instances(b2c, torch, cfg, G, ids[0])
    else:
        return None
    if graph:
        inst.capture(torch, streams=streams)
    ms = time_steps(torch, inst.step, steps, warmup)
    inst.check_status(b2c)
    us = ms * 1e3 / (steps * G)
    n = inst.launches_per_instance
    inst.destroy()
    return {"us": us, "launches_per_call": n}


def e2e_measure(b2c, torch, cfg, steps, warmup, dist=None):
    """Same metric through the host-buffer C-ABI calls, host memory to host memory.

    Main figure: the streaming call (b2c_plan_run_host_async): the plan holds the weights (uploaded once, outside
    the timed region, as a layer's parameters are), and EVERY call copies its own input batch from pinned host
    memory and reads its outputs back, copy in / path / copy out of successive calls overlapping.  Also timed:
    the one-shot call (b2c_conv2d_int8_host), which uploads x and w, runs and reads back, one call after the other."""
    xh, wh = cfg.tensors()
    ring = 4
    xs = [torch.from_numpy(np.roll(xh, i, axis=0).copy()).pin_memory().numpy() for i in range(ring)]
    w = torch.from_numpy(wh).pin_memory().numpy()
    oshape = (cfg.N, cfg.K, cfg.P, cfg.Q)
    y32s = [torch.empty(oshape, dtype=torch.int32).pin_memory().numpy() if cfg.out_mode & 1 else None for _ in range(ring)]
    y8s = [torch.empty(oshape, dtype=torch.int8).pin_memory().numpy() if cfg.out_mode & 2 else None for _ in range(ring)]
    ybytes = sum(a[0].nbytes for a in (y32s, y8s) if a[0] is not None)

    def timed(fn, nsteps):
        for _ in range(max(1, warmup)):
            fn()
        torch.cuda.synchronize()
        if dist is not None:
            dist.barrier()
        t0 = time.perf_counter()
        for _ in range(nsteps):
            fn()
        torch.cuda.synchronize()
        return max_over_ranks(torch, dist, time.perf_counter() - t0, "cuda")

    # streaming: one plan, weights resident
    desc = b2c.make_desc(cfg.N, cfg.C, cfg.H, cfg.W, cfg.K, cfg.R, cfg.S, cfg.stride, cfg.pad, cfg.dilation, cfg.shift,
                         out_mode=cfg.out_mode)
    plan = b2c.Plan(desc, b2c.POLICY_AUTO_TIMED)
    wd = torch.from_numpy(wh).cuda()
    plan.set_weights(wd)
    torch.cuda.synchronize()
    reps = 64

    def stream_fn():
        for i in range(reps):
            k = i % ring
            plan.run_host_async(xs[k], y32s[k], y8s[k])
        plan.host_sync()

    sec = timed(stream_fn, steps)
    plan.destroy()
    out = {"sec": sec, "calls": steps * reps, "h2d": xs[0].nbytes * reps, "d2h": ybytes * reps}

    # one-shot: x and w up, run, outputs down, synchronised, every call
    reps1 = 8

    def oneshot_fn():
        for _ in range(reps1):
            b2c.conv2d_int8_host(xs[0], w, cfg.stride, cfg.pad, cfg.dilation, cfg.shift, y32s[0], y8s[0])

    sec1 = timed(oneshot_fn, steps)
    out["one_shot"] = {"sec": sec1, "calls": steps * reps1, "h2d": (xs[0].nbytes + w.nbytes) * reps1, "d2h": ybytes * reps1}
    return out


def launch_floor_us(torch, launches=200):
    """Device time per launch of a graph of back-to-back one-element kernels: the floor any
    sequence of dependent kernel launches pays, measured the same way as the convolutions."""
    t = torch.zeros(1, device="cuda")
    for _ in range(3):
        t.add_(1.0)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        for _ in range(launches):
            t.add_(1.0)
    ms = time_steps(torch, g.replay, 10, 3, None, 0.0)
    return ms * 1e3 / (10 * launches)


def cpu_baseline(cfg, budget_s=12.0):
    """The oracle as it stands on the host cores, on a bounded sample of the workload."""
    import oracle

    x, w = cfg.tensors()
    cores = os.cpu_count() or 1
    n_probe = 1
    t0 = time.perf_counter()
    oracle.conv2d_int8(x[:n_probe], w, cfg.stride, cfg.pad, cfg.dilation, cfg.shift, True, True)
    t_probe = time.perf_counter() - t0
    n = int(max(1, min(cfg.N, budget_s / 3.0 / max(t_probe, 1e-6))))
    best = None
    for _ in range(3):
        t0 = time.perf_counter()
        oracle.conv2d_int8(x[:n], w, cfg.stride, cfg.pad, cfg.dilation, cfg.shift, True, True)
        dt = time.perf_counter() - t0
        best = dt if best is None else min(best, dt)
    macs = cfg.macs // cfg.N * n
    # one thread, and the separate stencil-unroll + GEMM path (single-threaded), on one image
    t0 = time.perf_counter()
    oracle.conv2d_int8(x[:1], w, cfg.stride, cfg.pad, cfg.dilation, cfg.shift, True, True, threads=1)
    t_one = time.perf_counter() - t0
    t0 = time.perf_counter()
    oracle.conv2d_via_im2col_gemm(x[:1], w, cfg.stride, cfg.pad, cfg.dilation)
    t_gemm = time.perf_counter() - t0
    macs1 = cfg.macs // cfg.N
    return {"value": 2.0 * macs / best / 1e12, "unit": UNIT, "cores": cores, "kind": "oracle",
            "sample": "%d of %d images of %s, best of 3, OpenMP over (n, k)" % (n, cfg.N, cfg.name), "seconds": best,
            "single_thread": 2.0 * macs1 / t_one / 1e12, "im2col_gemm_single_thread": 2.0 * macs1 / t_gemm / 1e12}


def _graph_us(torch, fn, repeat=20, replays=5):
    """Device time of one call of fn, from a CUDA graph of `repeat` calls replayed `replays` times."""
    fn()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        for _ in range(repeat):
            fn()
    ms = time_steps(torch, g.replay, replays, 3, None, 0.0)
    return ms * 1e3 / (replays * repeat)


def candidates_report(b2c, torch, shapes):
    """The paper's Table 3/4/5 layout on this machine: for every shape, every layout variant (and
    the swapped axis map) at its fastest schedule, with the device time split into Transf. (layout
    rewrite), Op. (MMA kernel + epilogue) and Combined, and the memory of the rewritten activations
    and packed weights; all relative to the channel-pack map with zero-padded channels, which is
    the paper's reference strategy.  Buffers are relaunched in place (L2 resident)."""
    out = []
    for cfg in shapes:
        d = b2c.make_desc(cfg.N, cfg.C, cfg.H, cfg.W, cfg.K, cfg.R, cfg.S, cfg.stride, cfg.pad, cfg.dilation, cfg.shift,
                          0, 0, cfg.out_mode)
        xh, wh = cfg.tensors()
        x, w = torch.from_numpy(xh).cuda(), torch.from_numpy(wh).cuda()
        oshape = (cfg.N, cfg.K, cfg.P, cfg.Q)
        y32 = torch.empty(oshape, dtype=torch.int32, device="cuda") if cfg.out_mode & 1 else None
        y8 = torch.empty(oshape, dtype=torch.int8, device="cuda") if cfg.out_mode & 2 else None
        best = {}
        for e in b2c.enumerate_embeddings(d):
            plan = b2c.Plan(d, e.id)
            ws = torch.empty(max(16, plan.workspace_bytes()), dtype=torch.uint8, device="cuda")
            plan.set_weights(w)
            us = _graph_us(torch, lambda: plan.run(x, y32, y8, ws), repeat=10, replays=3)
            key = (e.variant, e.map_m == b2c.AXIS_K)
            if key not in best or us < best[key][0]:
                best[key] = (us, e.id)
            plan.destroy()
        rows = []
        for (variant, swapped), (_, eid) in sorted(best.items()):
            plan = b2c.Plan(d, eid)
            e = plan.info()
            ws = torch.empty(max(16, plan.workspace_bytes()), dtype=torch.uint8, device="cuda")
            plan.set_weights(w)
            combined = _graph_us(torch, lambda: plan.run(x, y32, y8, ws))
            data_b, weight_b = plan.footprint()
            transf = _graph_us(torch, lambda: plan.rewrite_activations(x, ws)) if data_b else 0.0
            op = _graph_us(torch, lambda: plan.run_rewritten(x, y32, y8, ws))
            if plan.device_status() != 0:
                raise RuntimeError("device status")
            plan.destroy()
            rows.append({"variant": b2c.VARIANT_NAMES[variant] + ("+swap" if swapped else ""), "tile_n": e.tile_n,
                         "split_k": e.split_k, "op_us": op, "transf_us": transf, "combined_us": combined,
                         "data_bytes": data_b if data_b else cfg.N * cfg.C * cfg.H * cfg.W, "weight_bytes": weight_b,
                         "o_mac": e.o_mac, "o_data": e.o_data, "reference": variant == 0 and not swapped})
        out.append({"shape": cfg.name, "rows": rows})
    return out


def grouped_report(b2c, torch, N=8, C=256, H=28, W=28, R=3, stride=1, pad=1, shift=6):
    """Depth-wise layer (Section 6.1 names it as the same low-channel problem): all groups in one launch
    against the same layer written as a dense convolution with block-diagonal weights (zeros elsewhere)."""
    rng = np.random.default_rng(2104)
    xh = rng.integers(-128, 128, (N, C, H, W), dtype=np.int8)
    wg = rng.integers(-128, 128, (C, 1, R, R), dtype=np.int8)
    wd = np.zeros((C, C, R, R), dtype=np.int8)
    wd[np.arange(C), np.arange(C)] = wg[:, 0]
    d = b2c.make_desc(N, C, H, W, C, R, R, stride, pad, 1, shift, 0, 0, 2)
    P = (H + 2 * pad - R) // stride + 1
    x = torch.from_numpy(xh).cuda()
    y8 = torch.empty((N, C, P, P), dtype=torch.int8, device="cuda")
    rows, outs = [], []
    for name, groups, wh, policy in (("grouped, in place, one launch", C, wg, 0),
                                     ("grouped, form chosen by timing", C, wg, b2c.POLICY_AUTO_TIMED),
                                     ("dense plan given block-diagonal weights", 1, wd, b2c.POLICY_AUTO_TIMED)):
        plan = b2c.Plan(d, policy, groups=groups) if groups > 1 else b2c.Plan(d, policy)
        ws = torch.empty(max(16, plan.workspace_bytes()), dtype=torch.uint8, device="cuda")
        plan.set_weights(torch.from_numpy(wh).cuda())
        us = _graph_us(torch, lambda: plan.run(x, None, y8, ws))
        if plan.device_status() != 0:
            raise RuntimeError("device status")
        e = plan.info()
        rows.append({"form": name, "us": us, "embedding": b2c.VARIANT_NAMES[e.variant], "tile_n": e.tile_n,
                     "weight_elements": int(wh.size)})
        outs.append(y8.clone())
        plan.destroy()
    return {"shape": "depthwise_n%d_c%d_%dx%d_%dx%d" % (N, C, H, W, R, R), "rows": rows,
            "same_result": bool(torch.equal(outs[0], outs[1]) and torch.equal(outs[0], outs[2]))}


def print_candidates_markdown(report):
    for sh in report:
        ref = next((r for r in sh["rows"] if r["reference"]), None)
        print("\n### %s" % sh["shape"])
        print("| embedding | tile_n | split | Op. us | Transf. us | Combined us | Op. x | Combined x | data x | weights x | total mem x |")
        print("|---|---|---|---|---|---|---|---|---|---|---|")
        for r in sorted(sh["rows"], key=lambda r: r["combined_us"]):
            if ref:
                rel = (ref["op_us"] / r["op_us"], ref["combined_us"] / r["combined_us"], r["data_bytes"] / ref["data_bytes"],
                       r["weight_bytes"] / ref["weight_bytes"],
                       (r["data_bytes"] + r["weight_bytes"]) / (ref["data_bytes"] + ref["weight_bytes"]))
            else:
                rel = (float("nan"),) * 5
            print("| %s | %d | %d | %.2f | %.2f | %.2f | x%.2f | x%.2f | x%.3f | x%.3f | x%.3f |" % (
                r["variant"] + (" (reference)" if r["reference"] else ""), r["tile_n"], r["split_k"], r["op_us"],
                r["transf_us"], r["combined_us"], *rel))


def run_reference(args):
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return 0
    cfg = CONFIGS[args.config]
    import oracle

    x, w = cfg.tensors()
    cores = os.cpu_count() or 1
    t0 = time.perf_counter()
    oracle.conv2d_int8(x[:1], w, cfg.stride, cfg.pad, cfg.dilation, cfg.shift, True, True)
    t_probe = time.perf_counter() - t0
    total = max(1, args.steps + args.warmup)
    n = int(max(1, min(cfg.N, 60.0 / total / max(t_probe, 1e-6))))
    for _ in range(args.warmup):
        oracle.conv2d_int8(x[:n], w, cfg.stride, cfg.pad, cfg.dilation, cfg.shift, True, True)
    t0 = time.perf_counter()
    for _ in range(args.steps):
        oracle.conv2d_int8(x[:n], w, cfg.stride, cfg.pad, cfg.dilation, cfg.shift, True, True)
    sec = time.perf_counter() - t0
    macs = cfg.macs // cfg.N * n
    value = 2.0 * macs * args.steps / sec / 1e12
    sample = "%d of %d images of %s per step" % (n, cfg.N, cfg.name)
    line = {
        "impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": args.gpus, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": sec * 1e3 / args.steps, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "int8 x int8 -> int64 (range-checked to int32)", "data": "synthetic",
        "config": {"workload": cfg.name, "sample": sample},
        "cpu_baseline": {"value": value, "unit": UNIT, "cores": cores, "kind": "oracle", "sample": sample},
        "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
        "gpu_launches": 0,
    }
    print(json.dumps(line))
    return 0


def shard_report(world: int, instances_per_rank: int, ops_per_instance: float, steps: int, ms_max: float) -> float:
    """Whole-job TOPS: every rank runs its own `instances_per_rank` instances per step (weak scaling,
    no data-path collective); the job time is the slowest rank's."""
    return world * instances_per_rank * ops_per_instance * steps / (ms_max * 1e-3) / 1e12


def run_ours(args):
    import torch

    import paper_2104_04731_b200 as b2c

    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    if not torch.cuda.is_available():
        raise SystemExit("bench.py needs a CUDA device (there is no CPU fallback)")
    torch.cuda.set_device(local)
    dist = None
    if world > 1:
        import torch.distributed as dist_mod

        dist_mod.init_process_group("nccl", device_id=torch.device("cuda", local))
        dist = dist_mod
    b2c.load()
    peaks = load_peaks()
    cfg = CONFIGS[args.config]
    if args.scaled:
        cfg = scaled_shape(cfg, peaks)
    auto = b2c.POLICY_AUTO_TIMED_CONCURRENT if args.streams > 1 else b2c.POLICY_AUTO_TIMED
    policy = auto if args.embedding is None else args.embedding
    if args.pick:
        v, tn, sk, tm = (tuple(int(t) for t in args.pick.split(",")) + (128,))[:4]
        d0 = b2c.make_desc(cfg.N, cfg.C, cfg.H, cfg.W, cfg.K, cfg.R, cfg.S, cfg.stride, cfg.pad, cfg.dilation, cfg.shift,
                           0, 0, cfg.out_mode)
        policy = next(e.id for e in b2c.enumerate_embeddings(d0)
                      if (e.variant, e.tile_n, e.split_k, e.tile_m) == (v, tn, sk, tm) and e.map_m == b2c.AXIS_NPQ)
    graph = not args.no_graph
    if args.report == "candidates":
        rep = candidates_report(b2c, torch, CONFIGS + REPORT_EXTRA)
        grps = [grouped_report(b2c, torch, N=n) for n in (8, 128)]
        print(json.dumps({"report": "candidates", "shapes": rep, "grouped": grps}))
        print_candidates_markdown(rep)
        for grp in grps:
            print("\n### %s (grouped / depth-wise, Section 6.1)" % grp["shape"])
            print("| form | us | embedding | tile_n | weight elements |")
            print("|---|---|---|---|---|")
            for r in grp["rows"]:
                print("| %s | %.2f | %s | %d | %d |" % (r["form"], r["us"], r["embedding"], r["tile_n"], r["weight_elements"]))
            print("(same int8 output from all forms: %s)" % grp["same_result"])
        return 0

    sampler = ClockSampler(local)
    if rank == 0:
        sampler.start()
    # ---- headline: whole path, device-resident inputs ------------------------------------------
    G = args.instances if args.instances else instances_for(cfg)
    inst = Instances(b2c, torch, cfg, G, policy)
    if graph:
        inst.capture(torch, streams=args.streams)
    ms = time_steps(torch, inst.step, args.steps, args.warmup, dist, args.min_warm_s)
    inst.check_status(b2c)
    step_ms = sorted(LAST_STEP_MS)
    clocks = sampler.stop() if rank == 0 else None
    # the timed graph did the work: first and last instance of the last step against the oracle
    verified = inst.verify() if rank == 0 else None
    if verified is False:
        raise SystemExit("bench: the timed graph's output differs from the oracle")
    emb = inst.emb
    inst_launches = inst.launches_per_instance
    launches = inst.launches_per_instance * G * args.steps
    ops = 2.0 * cfg.macs
    value = shard_report(world, G, ops, args.steps, ms)
    per_call_us = ms * 1e3 / (args.steps * G)
    inst.destroy()

    # ---- the dominant kernel alone (the paper's "Op." column) for the roofline -------------------
    op = None
    if not args.no_op_pass:
        op = op_only(b2c, torch, cfg, emb.variant, emb.tile_n, emb.split_k, args.steps, args.warmup, graph, args.streams,
                     emb.map_m, emb.tile_m)
    t_roof, bound = roofline_time_us(cfg, peaks)
    op_us = op["us"] if op else per_call_us
    op_steps = sorted(LAST_STEP_MS) if op else step_ms
    # the same kernel with one launch in flight (one call after the other on one stream)
    alone = None
    if op and graph and args.streams > 1 and rank == 0:
        alone = op_only(b2c, torch, cfg, emb.variant, emb.tile_n, emb.split_k, max(2, args.steps // 2), 3, graph, 1, emb.map_m,
                        emb.tile_m)
    # second denominator: this library's own issue-rate measurement of the intrinsic (no loads, all SMs)
    issue = None
    if rank == 0:
        r_us, r_cyc = b2c.measure_mma_rate(256, 20000)
        mma_ops = 2.0 * 128 * 256 * 32
        issue = {"tile": "128x256x32", "mmas_per_sm": 20000, "device_us": r_us, "cycles_per_mma": r_cyc,
                 "tops": 148 * 20000 * mma_ops / (r_us * 1e-6) / 1e12, "ops_per_clock_all_sms": 148 * mma_ops / r_cyc}
        # the two-SM form the headline kernel issues (each block's tensor core reads half of B from its peer)
        p_us, p_cyc = b2c.measure_mma_rate_pair(256, 20000)
        issue["two_sm"] = {"tile": "256x256x32", "mmas_per_pair": 20000, "device_us": p_us, "cycles_per_mma": p_cyc,
                           "tops": 74 * 20000 * 2.0 * 256 * 256 * 32 / (p_us * 1e-6) / 1e12}
    if bound == "tensor":
        achieved, peak, runit = ops / (op_us * 1e-6) / 1e12, peaks["bf16_tflops"] * INT8_TO_BF16_RATIO, "TFLOP/s"
    else:
        achieved, peak, runit = cfg.algorithmic_bytes / (op_us * 1e-6) / 1e9, peaks["hbm_gbs"], "GB/s"
    sha = kernel_sources_sha1()
    traffic = None
    if NCU_TRAFFIC["conv_mma_sha1"] == sha and args.config == HEADLINE and not args.scaled and emb.variant == 0:
        traffic = NCU_TRAFFIC["bytes_per_launch"].get("%dx%d" % (emb.tile_m, emb.tile_n))
    kname = "conv_mma_pair_kernel" if emb.tile_m == 256 else "conv_mma_kernel"
    launches_per_step = (op["launches_per_call"] if op else inst_launches) * G
    roofline = {"bound": bound, "achieved": achieved, "peak": peak, "unit": runit, "frac": achieved / peak,
                "traffic": traffic, "kernel": kname, "kernel_us": op_us,
                "kernel_us_median": op_steps[len(op_steps) // 2] * 1e3 / G, "kernel_us_min": op_steps[0] * 1e3 / G,
                "kernel_us_note": "timed region / launches, %d launches in flight" % (args.streams if graph else 1),
                "kernel_us_alone": alone["us"] if alone else None,
                "frac_alone": (ops / (alone["us"] * 1e-6) / 1e12 / peak) if (alone and bound == "tensor") else None,
                "peak_source": "%s bf16 burst x %.0f (nominal int8:bf16)" % (peaks["source"], INT8_TO_BF16_RATIO)
                if bound == "tensor" else peaks["source"] + " copy bandwidth"}
    if issue is not None and bound == "tensor":
        # both denominators, and the fraction that does not depend on the clock the peaks were taken at:
        # ops per SM clock of the timed kernel (time x median SM clock sampled during the run) against the
        # ops per clock the intrinsic issues at
        roofline["peak_i8_issue_rate"] = issue
        roofline["frac_vs_issue_rate"] = achieved / issue["tops"]
        roofline["frac_vs_larger_peak"] = achieved / max(peak, issue["tops"])
        if emb.tile_m == 256 and "two_sm" in issue:
            roofline["frac_vs_two_sm_issue_rate"] = achieved / issue["two_sm"]["tops"]
        if clocks and clocks.get("sm_mhz"):
            roofline["frac_clock_normalised"] = (ops / (op_us * 1e-6) / (clocks["sm_mhz"] * 1e6)) / issue["ops_per_clock_all_sms"]

    # ---- end to end through the host-buffer call ----------------------------------------------------
    e2e = None
    if not args.no_e2e:
        e = e2e_measure(b2c, torch, cfg, max(1, min(args.steps, 5)), 1, dist)
        steps_e = max(1, min(args.steps, 5))
        o = e["one_shot"]
        e2e = {"value": world * e["calls"] * ops / e["sec"] / 1e12, "unit": UNIT,
               "h2d_bytes_per_step": e["h2d"], "d2h_bytes_per_step": e["d2h"],
               "call": "b2c_plan_run_host_async + b2c_plan_host_sync (weights resident in the plan; 64 calls per step, "
                       "each copying its input from pinned host memory and its outputs back, three in flight)",
               "us_per_call": e["sec"] / e["calls"] * 1e6,
               "host_link_gbs": (e["h2d"] + e["d2h"]) * steps_e / e["sec"] / 1e9,
               "one_shot": {"call": "b2c_conv2d_int8_host (x and w up, run, outputs down, synchronised, per call)",
                            "value": world * o["calls"] * ops / o["sec"] / 1e12, "unit": UNIT,
                            "us_per_call": o["sec"] / o["calls"] * 1e6,
                            "h2d_bytes_per_step": o["h2d"], "d2h_bytes_per_step": o["d2h"]}}

    per_config = None
    if rank == 0 and not args.headline_only:
        per_config = []
        for c in CONFIGS:
            r = measure_shape(b2c, torch, c, max(2, args.steps // 2), 3, peaks, b2c.POLICY_AUTO_TIMED, None, graph,
                              args.streams)
            per_config.append(r)
    scaled = None
    if rank == 0 and not args.headline_only:
        scaled = [measure_scaled(b2c, torch, c, peaks) for c in CONFIGS]
    cpu = cpu_baseline(cfg) if (rank == 0 and world == 1 and not args.no_cpu) else None

    if dist is not None:
        dist.barrier()
        dist.destroy_process_group()
    if rank != 0:
        return 0
    line = {
        "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps, "warmup": args.warmup,
        "ms_per_step": ms / args.steps, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
        "dtype": "s8 x s8 -> s32", "data": "synthetic",
        "config": {"workload": cfg.name, "instances_per_step": G, "per_call_us": per_call_us,
                   "per_call_us_median": step_ms[len(step_ms) // 2] * 1e3 / G, "per_call_us_min": step_ms[0] * 1e3 / G,
                   "l2": "inputs larger than L2: %d distinct buffer sets per step (%.0f MB)" % (G, G * (cfg.algorithmic_bytes) / 1e6),
                   "cuda_graph": graph, "streams": args.streams if graph else 1,
                   "parallelism": "independent instances sharded over ranks, no collective",
                   "embedding": {"variant": b2c.VARIANT_NAMES[emb.variant], "tile_m": emb.tile_m, "tile_n": emb.tile_n,
                                 "split_k": emb.split_k, "swapped": emb.map_m == b2c.AXIS_K, "planner_us": emb.device_us}},
        "roofline": roofline, "roofline_time_us": t_roof, "whole_path_roofline_frac": t_roof / per_call_us,
        "e2e": e2e, "gpu_launches": launches, "clocks": clocks, "verified": verified,
    }
    if cpu is not None:
        line["cpu_baseline"] = cpu
    if per_config is not None:
        line["per_config"] = per_config
    if scaled is not None:
        line["scaled"] = scaled
        line["launch_floor_us"] = launch_floor_us(torch)
    print(json.dumps(line))
    return 0


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=20)
    ap.add_argument("--warmup", type=int, default=5)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--config", type=int, default=HEADLINE, help="index into the five benchmark shapes")
    ap.add_argument("--embedding", type=int, default=None, help="embedding id; default: timed selection")
    ap.add_argument("--no-graph", action="store_true")
    ap.add_argument("--no-cpu", action="store_true")
    ap.add_argument("--headline-only", action="store_true", help="skip the per-shape and scaled-batch series")
    ap.add_argument("--pick", default=None, help="first embedding with variant,tile_n,split_k[,tile_m] (instead of an id; schedules of the window unroll "
                         "can agree in all of them: --embedding tells them apart)")
    ap.add_argument("--scaled", action="store_true", help="use the batch-scaled version of the shape as the workload")
    ap.add_argument("--instances", type=int, default=0, help="instances per step (default: enough to exceed L2)")
    ap.add_argument("--min-warm-s", type=float, default=0.2, help="extra time-based warm-up before the timed steps")
    ap.add_argument("--streams", type=int, default=16,
                    help="graph branches the independent instances of a step are dealt onto (1 = one call after the other)")
    ap.add_argument("--report", default=None, choices=["candidates"],
                    help="candidates: per-shape table of every layout variant (Op./Transf./Combined/memory), no bench line")
    ap.add_argument("--no-op-pass", action="store_true", help="skip the separate pass that times the MMA kernel alone")
    ap.add_argument("--no-e2e", action="store_true", help="skip the host-buffer end-to-end pass")
    args = ap.parse_args()
    args.warmup = max(args.warmup, 3) if args.impl == "ours" else args.warmup
    if args.impl == "reference":
        return run_reference(args)
    if args.gpus > 1 and "WORLD_SIZE" not in os.environ:
        # started as a plain script: start one rank per GPU (the same command a launcher would give)
        import socket

        with socket.socket() as sk:
            sk.bind(("127.0.0.1", 0))
            port = sk.getsockname()[1]
        cmd = [sys.executable, "-m", "torch.distributed.run", "--nnodes=1", "--nproc-per-node", str(args.gpus),
               "--master-addr", "127.0.0.1", "--master-port", str(port), os.path.abspath(__file__)] + sys.argv[1:]
        return subprocess.call(cmd)
    return run_ours(args)


if __name__ == "__main__":
    sys.exit(main())
