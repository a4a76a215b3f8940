"""Benchmark of the masked secure linear layer on GB300.

One step = one pass of the whole per-call path of Pi_Sec-Linear over one batch
of tokens: Init X (PRG masks R, T_i, E_x and U_x, K), rotation + encode +
mask-add of X, the server's ring product Z = X' [W'; P]^T over Z_{2^32}, and the
unmask + decode.  Init W (public chains and the masked weights) is one-time and
is timed apart (``init_w_s``).

Workloads (``--workload``; seeded synthetic inputs, activations ~ N(0,1),
weights ~ N(0,0.02), Example 3.1 parameters):
  decoder_70b_prefill_2048     (default) one 70B decoder layer: 4 masked linears
                               (QKV 8192->10240, O 8192->8192, gate+up 8192->57344,
                               down 28672->8192) + fp32 RMSNorm / causal GQA
                               attention / SwiGLU / residuals, 2048 tokens
  attn_proj_7b_512x4096x4096   X 512 x 4096, W 4096 x 4096
  ffn_7b_2048x4096x14336       up 4096 -> 14336 then down 14336 -> 4096, 2048 tokens
  decode_70b_sweep             every linear of a 70B layer at 1..256 tokens
L2 is flushed (256 MiB write) between timed steps.

  python bench.py [--gpus N] [--steps K] [--warmup W] [--impl mine|reference]

Prints one JSON line (rank 0).  With N > 1 (torchrun) every rank runs an
independent replica on its own GPU (weak scaling, no data-path collective).
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

from paper_2607_29221_gb300 import workloads as wl  # noqa: E402

METRIC = "masked ring-GEMM effective TOPS (Z_2^32) and masked-layer tokens/s; % of roofline"
L2_FLUSH_BYTES = 256 << 20
DEFAULT_WORKLOAD = "decoder_70b_prefill_2048"
DECODER_SEED = 11          # weights of the decoder layer: seeds 11..14 (QKV, O, gate+up, down)


def _peaks():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    try:
        with open(path) as f:
            d = json.load(f)
        return float(d["hbm_gbs"]), float(d["bf16_tflops"]), float(d["bf16_tflops_sustained"]), "measured"
    except Exception:
        return 6800.0, 1900.0, 1700.0, "fallback"


def _traffic(kernel: str, workload: str):
    """DRAM bytes of `kernel` per step of `workload` from the committed ncu
    capture (profiles/traffic.json), or None if there is none or the kernel's
    source changed since the capture."""
    import hashlib
    try:
        with open(os.path.join(ROOT, "profiles", "traffic.json")) as f:
            rec = json.load(f)[f"{kernel}@{workload}"]
        with open(os.path.join(ROOT, rec["source"]), "rb") as f:
            if hashlib.sha256(f.read()).hexdigest() != rec["source_sha256"]:
                return None
        return float(rec["dram_bytes_per_step"])
    except Exception:
        return None


def _config(wk, world):
    """The workload as both arms report it (the JSON line's `config`)."""
    cfg = {"workload": wk.name, "l": wk.l,
           "linears": [{"name": x.name, "m": x.m, "n": x.n} for x in wk.linears],
           "params": "Example 3.1: d=3, r=1536/1024/652, t=80/80, sigma=0.5, b=16",
           "l2": "flushed between timed steps (256 MiB write)",
           "parallelism": f"replicas x{world}"}
    if wk.name == "decoder_70b_prefill_2048":
        cfg["glue"] = "fp32 RMSNorm, causal GQA attention (64 q / 8 kv heads, d 128), SwiGLU, residuals"
    return cfg


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=20)
    ap.add_argument("--warmup", type=int, default=5)
    ap.add_argument("--impl", default="mine", choices=["mine", "reference"])
    ap.add_argument("--workload", default=DEFAULT_WORKLOAD, choices=sorted(wl.WORKLOADS))
    ap.add_argument("--variant", default="auto", choices=["auto", "tc", "mma_s8", "imad"])
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--cpu-budget-s", type=float, default=12.0)
    return ap.parse_args()


# ---------------------------------------------------------------------------
# clocks sampled during the timed region
# ---------------------------------------------------------------------------
class ClockSampler:
    FIELDS = ("clocks.sm,clocks.max.sm,power.draw,utilization.gpu,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, index: int):
        self.index = index
        self.proc = None
        self.lines = []

    def start(self):
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", f"--query-gpu={self.FIELDS}", "--format=csv,noheader,nounits",
                 "-i", str(self.index), "-lms", "50"],
                stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.thread = threading.Thread(target=self._read, daemon=True)
            self.thread.start()
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
        self.thread.join(timeout=2)
        sm, smax, util, reasons = [], [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for ln in self.lines:
            parts = [p.strip() for p in ln.split(",")]
            if len(parts) < 9:
                continue
            try:
                sm.append(float(parts[0])); smax.append(float(parts[1])); util.append(float(parts[3]))
            except ValueError:
                continue
            for nm, v in zip(names, parts[5:9]):
                if v.lower().startswith("active"):
                    reasons.add(nm)
        if not sm:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["no samples"], "samples": 0}
        loaded = [s for s, u in zip(sm, util) if u > 0] or sm
        return {"sm_mhz": float(np.median(loaded)), "sm_max_mhz": max(smax),
                "reasons": sorted(reasons), "samples": len(sm), "samples_under_load": len(loaded)}


# ---------------------------------------------------------------------------
# workloads
# ---------------------------------------------------------------------------
class _Timed:
    """CUDA events around the server products and the encodes of the steps
    being timed (on the launching stream)."""

    def __init__(self, stream):
        self.stream = stream
        self.active = False
        self.pairs = {"server": [], "encode": []}

    def _wrap(self, fn, key):
        import torch

        def timed(*a, **k):
            if not self.active:
                return fn(*a, **k)
            e0 = torch.cuda.Event(enable_timing=True); e1 = torch.cuda.Event(enable_timing=True)
            e0.record(self.stream)
            out = fn(*a, **k)
            e1.record(self.stream)
            self.pairs[key].append((e0, e1))
            return out
        return timed

    def wrap(self, layer):
        layer.server = self._wrap(layer.server, "server")
        layer.mask_input = self._wrap(layer.mask_input, "encode")

    def ms(self, key, steps):
        p = self.pairs[key]
        return float(np.sum([a.elapsed_time(b) for a, b in p])) / steps if p else 0.0

    def clear(self):
        for v in self.pairs.values():
            v.clear()


class _Parts:
    """mark(part) records a CUDA event where a part of the step begins; the
    time to the next mark is charged to that part."""

    def __init__(self, stream):
        self.stream = stream
        self.evs = []

    def __call__(self, name):
        import torch
        e = torch.cuda.Event(enable_timing=True)
        e.record(self.stream)
        self.evs.append((name, e))

    def totals(self):
        out = {}
        for (n, a), (_, b) in zip(self.evs[:-1], self.evs[1:]):
            if n != "end":
                out[n] = out.get(n, 0.0) + a.elapsed_time(b)
        return out


def _no_mark(name):
    return None


class LinearChain:
    """Secure linear calls in sequence, each call's decoded output feeding the
    next (attention projection: one call; FFN: up then down)."""

    def __init__(self, proto, dev, linears, l, rank, timed):
        import torch
        from paper_2607_29221_gb300 import protocol as PR
        self.l, self.rank = l, rank
        chains = {}
        self.layers, self.bufs = [], []
        for i, lin in enumerate(linears):
            n_pad = PR.pad_width(lin.n)
            if n_pad not in chains:
                chains[n_pad] = PR.Chains(proto, n_pad)
            W = torch.from_numpy(wl.weights(lin.m, lin.n, seed=wl.SEED_W + i, std=lin.w_std)).to(dev)
            b = torch.from_numpy(wl.bias(lin.m, seed=wl.SEED_B + i)).to(dev)
            layer = PR.SecureLinear(proto, W, 1 + i, chains[n_pad], bias=b)
            timed.wrap(layer)
            self.layers.append(layer)
            Sr = proto.sum_r
            self.bufs.append(dict(
                Xp=torch.empty(l, n_pad, dtype=torch.int32, device=dev),
                s_x=torch.empty(l, dtype=torch.float32, device=dev),
                Xpl=torch.empty(4, l, n_pad, dtype=torch.int16, device=dev) if layer.use_planes else None,
                Z=torch.empty(l, lin.m + Sr, dtype=torch.int32, device=dev),
                Y=torch.empty(l, lin.m, dtype=torch.float32, device=dev)))
        self.ring_macs = sum(l * (ly.m + proto.sum_r) * ly.n_pad for ly in self.layers)
        self.n_in, self.m_out = linears[0].n, linears[-1].m
        self.masks = [ly.init_x(l, 900_000 + c) for c, ly in enumerate(self.layers)]

    def step(self, x, i, mark=None, serial=False):
        mark = mark or _no_mark
        for c, (layer, bf) in enumerate(zip(self.layers, self.bufs)):
            mark("init_x")
            mp = layer.init_x(self.l, 1_000_000 * self.rank + 1000 * c + i, out=self.masks[c])
            mark("encode")
            layer.mask_input(x, mp, bf["Xp"], bf["s_x"], bf["Xpl"])
            mark("server")
            layer.server(bf["Xp"], bf["Xpl"], bf["Z"])
            mark("unmask")
            layer.unmask(bf["Z"], mp, bf["s_x"], bf["Y"])
            x = bf["Y"]
        return x

    def _pass(self, x, mps, ctr, side):
        from paper_2607_29221_gb300 import mosaic as M
        for c, (layer, bf) in enumerate(zip(self.layers, self.bufs)):
            layer.mask_input(x, mps[c], bf["Xp"], bf["s_x"], bf["Xpl"])
            layer.server(bf["Xp"], bf["Xpl"], bf["Z"])
            layer.unmask(bf["Z"], mps[c], bf["s_x"], bf["Y"])
            M.mosaic_advance_pass(ctr[c], 1, stream=side)
            x = bf["Y"]
        return x

    def graph(self, x):
        """The same step captured as one CUDA graph: each layer's pass id is
        a base plus a device counter that the graph advances, so every replay
        draws fresh masks (pass ids disjoint from the eager steps')."""
        import torch
        dev = x.device
        base = [1_000_000 * self.rank + 500_000 + 1000 * c for c in range(len(self.layers))]
        ctr = [torch.zeros(1, dtype=torch.int64, device=dev) for _ in self.layers]
        gmask = [ly.init_x(self.l, b) for ly, b in zip(self.layers, base)]   # buffers, workspace sized
        torch.cuda.synchronize()
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=side):
            mps = [ly.init_x(self.l, base[c], pass_dev=ctr[c], out=gmask[c]) for c, ly in enumerate(self.layers)]
            y = self._pass(x, mps, ctr, side)
        torch.cuda.synchronize()
        return g, y

    def graph_e2e(self, X, X_host, Y_host_prev, Y_dev_prev, Y_dev_out):
        """The step with its host copies as one CUDA graph: the copy of X in
        runs on a forked stream beside every layer's Init X (which does not
        depend on X); the previous step's result Y_dev_prev is read out to
        Y_host_prev on another forked stream beside the whole step, and this
        step's result ends in Y_dev_out (read out by the next step)."""
        import torch
        dev = X.device
        base = [1_000_000 * self.rank + 700_000 + 1000 * c for c in range(len(self.layers))]
        ctr = [torch.zeros(1, dtype=torch.int64, device=dev) for _ in self.layers]
        gmask = [ly.init_x(self.l, b) for ly, b in zip(self.layers, base)]
        torch.cuda.synchronize()
        side, copy, out = torch.cuda.Stream(), torch.cuda.Stream(), torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=side):
            copy.wait_stream(side)
            out.wait_stream(side)
            with torch.cuda.stream(copy):
                X.copy_(X_host, non_blocking=True)
            with torch.cuda.stream(out):
                Y_host_prev.copy_(Y_dev_prev, non_blocking=True)
            mps = [ly.init_x(self.l, base[c], pass_dev=ctr[c], out=gmask[c]) for c, ly in enumerate(self.layers)]
            side.wait_stream(copy)
            y = self._pass(X, mps, ctr, side)
            Y_dev_out.copy_(y, non_blocking=True)
            side.wait_stream(out)
        torch.cuda.synchronize()
        return g


class DecoderLayerRun:
    """One 70B decoder layer: four masked linears and the fp32 glue."""

    def __init__(self, proto, dev, l, rank, timed):
        from paper_2607_29221_gb300 import decoder as D
        s = D.LayerShape()
        self.layer = D.SecureDecoderLayer(proto, D.LayerWeights(s, seed=DECODER_SEED, device=dev))
        self.layers = self.layer.linears()
        for lin in self.layers:
            timed.wrap(lin)
        self.layer.alloc(l)
        self.ring_macs = sum(l * (lin.m + proto.sum_r) * lin.n_pad for lin in self.layers)
        self.n_in = self.m_out = s.hidden
        self.l, self.rank = l, rank
        self.masks = self.layer.init_x(l, 90_000)

    def step(self, x, i, mark=None, serial=False):
        """One pass; with `serial` the four Init X calls run whole, one after
        the other, before the layer (no draws beside other kernels), as the
        per-kernel rooflines are measured."""
        if serial:
            masks = self.layer.init_x(self.l, 100_000 * self.rank + i, out=self.masks)
            return self.layer.forward(x, masks, mark=mark)
        return self.layer.forward_pass(x, 100_000 * self.rank + i, self.masks, mark=mark)

    def graph(self, x):
        """The layer's step captured as one CUDA graph (fresh masks per replay
        from a device pass counter)."""
        import torch
        from paper_2607_29221_gb300 import mosaic as M
        base = 100_000 * self.rank + 50_000
        ctr = torch.zeros(1, dtype=torch.int64, device=x.device)
        gm = self.layer.init_x(self.l, base)
        torch.cuda.synchronize()
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=side):
            y = self.layer.forward_pass(x, base, gm, pass_dev=ctr)
            M.mosaic_advance_pass(ctr, 1, stream=side)
        torch.cuda.synchronize()
        return g, y

    def graph_e2e(self, X, X_host, Y_host_prev, Y_dev_prev, Y_dev_out):
        """The step with its host copies as one CUDA graph: the copy of X in
        runs on a forked stream beside the first call's Init X draws
        (independent of X); the previous step's result Y_dev_prev is read out
        to Y_host_prev on another forked stream beside the whole step, and
        this step's result ends in Y_dev_out (read out by the next step)."""
        import torch
        from paper_2607_29221_gb300 import mosaic as M
        base = 100_000 * self.rank + 70_000
        ctr = torch.zeros(1, dtype=torch.int64, device=X.device)
        gm = self.layer.init_x(self.l, base)
        torch.cuda.synchronize()
        side, copy, out = torch.cuda.Stream(), torch.cuda.Stream(), torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=side):
            copy.wait_stream(side)
            out.wait_stream(side)
            with torch.cuda.stream(copy):
                X.copy_(X_host, non_blocking=True)
            with torch.cuda.stream(out):
                Y_host_prev.copy_(Y_dev_prev, non_blocking=True)
            y = self.layer.forward_pass(X, base, gm, pass_dev=ctr, after=copy)
            M.mosaic_advance_pass(ctr, 1, stream=side)
            Y_dev_out.copy_(y, non_blocking=True)
            side.wait_stream(out)
        torch.cuda.synchronize()
        return g


def _time_steps(torch, runner, make_input, steps, warmup, flush, stream, timed, world, counter=None):
    for i in range(warmup):
        runner.step(make_input(), i)
    torch.cuda.synchronize()
    _barrier(world)
    torch.cuda.synchronize()
    evs = []
    timed.active = True
    c0 = counter() if counter else 0
    for i in range(steps):
        flush.fill_(i & 0xFF)
        x = make_input()
        s0 = torch.cuda.Event(enable_timing=True); s1 = torch.cuda.Event(enable_timing=True)
        s0.record(stream)
        runner.step(x, warmup + i)
        s1.record(stream)
        evs.append((s0, s1))
    timed.active = False
    launches = (counter() - c0) if counter else 0
    torch.cuda.synchronize()
    _barrier(world)
    step_ms = float(np.mean([a.elapsed_time(b) for a, b in evs]))
    gemm_ms = timed.ms("server", steps)
    enc_ms = timed.ms("encode", steps)
    timed.clear()
    return step_ms, gemm_ms, launches, enc_ms


class _Replay:
    def __init__(self, g):
        self.g = g

    def step(self, x_unused, i):
        self.g.replay()


def run_mine(args, rank, world):
    import torch
    import __graft_entry__ as G
    from paper_2607_29221_gb300 import mosaic as M
    from paper_2607_29221_gb300 import protocol as PR

    G.build()
    dev = torch.device("cuda", int(os.environ.get("LOCAL_RANK", 0)))
    torch.cuda.set_device(dev)
    variant = {"auto": M.GEMM_AUTO, "tc": M.GEMM_TC, "mma_s8": M.GEMM_MMA_S8, "imad": M.GEMM_IMAD}[args.variant]
    if variant == M.GEMM_AUTO:
        variant = M.GEMM_TC if M.mosaic_gemm_variant_available(M.GEMM_TC) else M.GEMM_IMAD
    proto = PR.Protocol(wl.mask_key(), M.default_params(), variant=variant)
    stream = torch.cuda.current_stream()
    timed = _Timed(stream)
    flush = torch.empty(L2_FLUSH_BYTES, dtype=torch.uint8, device=dev)
    wk = wl.WORKLOADS[args.workload]

    if args.workload == "decode_70b_sweep":
        return run_decode_sweep(args, rank, world, torch, M, PR, proto, dev, stream, timed, flush, wk,
                                variant)
    if args.workload == "matvec_sweep":
        return run_matvec_sweep(args, rank, world, torch, M, PR, proto, dev, stream, flush, wk)
    if args.workload == "sigma_sweep_7b":
        return run_sigma_sweep(args, rank, world, torch, M, PR, dev, wk, variant)
    if args.workload == "init_w_70b":
        return run_init_w(args, rank, world, torch, M, PR, proto, dev, wk)
    if args.workload == "kernels_hbm":
        return run_kernels_hbm(args, rank, world, torch, M, PR, proto, dev, stream, flush, wk)

    torch.cuda.synchronize()
    t0 = time.perf_counter()
    if args.workload == "decoder_70b_prefill_2048":
        runner = DecoderLayerRun(proto, dev, wk.l, rank, timed)
    else:
        runner = LinearChain(proto, dev, list(wk.linears), wk.l, rank, timed)
    torch.cuda.synchronize()
    init_w_s = time.perf_counter() - t0

    l = wk.l
    X_host = torch.from_numpy(wl.activations(l, runner.n_in, seed=wl.SEED_X + rank)).pin_memory()
    X = X_host.to(dev)

    sampler = ClockSampler(_smi_index(dev.index))
    sampler.start()
    time.sleep(0.3)
    # Eager steps: our kernels launched inside the timed region (the library's
    # own counter), and CUDA events around every server product and encode.
    eager_ms, gemm_ms, launches_timed, enc_ms = _time_steps(
        torch, runner, lambda: X, args.steps, args.warmup, flush, stream, timed, world,
        M.mosaic_kernel_launches)
    # The step as one CUDA graph (same kernels; replays draw fresh passes).
    g, _ = runner.graph(X)
    step_ms, _, _, _ = _time_steps(torch, _Replay(g), lambda: X, args.steps, args.warmup, flush, stream,
                                   timed, world)
    del g
    # Where the step's time goes: CUDA events where each part begins (eager).
    part_steps = max(3, args.steps // 4)
    parts = _Parts(stream)
    for i in range(part_steps):
        flush.fill_(i & 0xFF)
        runner.step(X, 20_000 + i, mark=parts)
        parts("end")
    torch.cuda.synchronize()
    part_ms = {k: round(v / part_steps, 4) for k, v in parts.totals().items()}
    # Per-kernel device time of eager steps (the library's own event pair
    # around each launch, so not inside the timed steps above): the client
    # kernels' rooflines.  These steps run every kernel alone (serial Init X),
    # so that a kernel's time is not shared with the overlapped draws.
    M.mosaic_kernel_times(reset=True)
    M.mosaic_kernel_timing(True)
    for i in range(part_steps):
        flush.fill_(i & 0xFF)
        runner.step(X, 30_000 + i, serial=True)
    torch.cuda.synchronize()
    M.mosaic_kernel_timing(False)
    ktimes = M.mosaic_kernel_times(reset=True)
    # The device's rate of the ChaCha20 add / xor / rotate mix: the draws' ALU peak
    # (8 x 256 threads per SM, one scratch word each; 256 SMs' worth) ...
    mix_scratch = torch.empty(8 * 256 * 256, dtype=torch.int32, device=dev)
    alu_rate = M.mosaic_int_mix_rate(mix_scratch)
    # ... and its shared-memory read rate with the gather's access: the gathers' peak.
    smem_rate = M.mosaic_smem_read_rate(mix_scratch)
    del mix_scratch

    # End to end through the public API with host buffers: the copy of X in
    # and of Y out inside the timed region, every step.
    Y_host = torch.empty(l, runner.m_out, dtype=torch.float32).pin_memory()
    e2e_steps = max(3, args.steps // 2)

    def _e2e(step_fn):
        ev = []
        for i in range(e2e_steps):
            flush.fill_(i & 0xFF)
            a = torch.cuda.Event(enable_timing=True); c = torch.cuda.Event(enable_timing=True)
            a.record(stream)
            step_fn(i)
            c.record(stream)
            ev.append((a, c))
        torch.cuda.synchronize()
        return float(np.mean([a.elapsed_time(c) for a, c in ev]))

    def _eager_e2e(i):
        X.copy_(X_host, non_blocking=True)
        Y = runner.step(X, 10_000 + i)
        Y_host.copy_(Y, non_blocking=True)
    e2e_eager_ms = _e2e(_eager_e2e)
    # The graph form pipelines the read-out: step k copies X in and reads out
    # step k - 1's result while it computes (two graphs alternate the device
    # buffer of the result); the last step's result is read inside the last
    # step's timed region.
    Y_dev = [torch.empty(l, runner.m_out, dtype=torch.float32, device=dev) for _ in range(2)]
    Y_hosts = [Y_host, torch.empty(l, runner.m_out, dtype=torch.float32).pin_memory()]
    ges = [runner.graph_e2e(X, X_host, Y_hosts[1 - p], Y_dev[1 - p], Y_dev[p]) for p in (0, 1)]
    for i in range(4):
        ges[i % 2].replay()
    torch.cuda.synchronize()

    def _graph_e2e(i):
        ges[i % 2].replay()
        if i == e2e_steps - 1:
            Y_hosts[i % 2].copy_(Y_dev[i % 2], non_blocking=True)
    e2e_ms = _e2e(_graph_e2e)
    del ges
    clocks = sampler.stop()
    M.mosaic_device_status()

    step_ms_max = _max_over_ranks(step_ms, world, dev)
    eager_ms_max = _max_over_ranks(eager_ms, world, dev)
    e2e_ms_max = _max_over_ranks(e2e_ms, world, dev)
    e2e_eager_ms_max = _max_over_ranks(e2e_eager_ms, world, dev)
    if rank != 0:
        return

    hbm, bf16, bf16_sus, peak_src = _peaks()
    tokens_s = world * l / (step_ms_max / 1e3)
    ring_tops = 2 * runner.ring_macs / (gemm_ms / 1e3) / 1e12
    roof = _roofline(variant, M, runner.ring_macs, gemm_ms, bf16, peak_src,
                     _traffic("ring_gemm_tc", args.workload) if variant == M.GEMM_TC else None)
    roof["per"] = (f"the {len(runner.layers)} server-product launches of one step"
                   if len(runner.layers) > 1 else "one server-product launch")
    if variant == M.GEMM_TC:
        roof["frac_of_sustained"] = round(roof["achieved"] / bf16_sus, 4)
    enc_bytes = sum(l * (4 * ly.n + (16 if ly.use_planes and l > M.STREAMW_MAX_M else 8) * ly.n_pad)
                    for ly in runner.layers)
    # The encode's time from the serial per-kernel steps (its launches alone),
    # the CUDA events around the encodes of the timed steps otherwise.
    enc_kt = sum(v[1] for k, v in ktimes.items() if k.startswith("encode:")) / part_steps
    if enc_kt > 0:
        enc_ms = enc_kt
    enc_gbs = enc_bytes / (enc_ms / 1e3) / 1e9 if enc_ms > 0 else 0.0
    rooflines = [dict(roof, kernel=roof["kernel"]),
                 {"kernel": "fwht_kernel (encode: rotate, quantise, + U_x, digit planes)", "bound": "hbm",
                  "achieved": round(enc_gbs, 1), "peak": hbm, "unit": "GB/s", "frac": round(enc_gbs / hbm, 4),
                  "traffic": None, "bytes_per_step": enc_bytes, "ms_per_step": round(enc_ms, 4),
                  "peak_source": f"{peak_src} copy bandwidth"}]
    rooflines += _client_rooflines(ktimes, part_steps, runner.layers, proto, l, bf16, peak_src,
                                   float(clocks.get("sm_mhz") or clocks.get("sm_max_mhz") or 2070.0), alu_rate,
                                   smem_rate)
    out = {
        "metric": METRIC, "value": round(tokens_s, 1), "unit": "tokens/s", "n_gpus": world,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": round(step_ms_max, 4),
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "u32",
        "data": "synthetic (seeded N(0,1) activations, N(0,0.02) weights)",
        "config": _config(wk, world),
        "implementation": {"gemm_variant": {M.GEMM_TC: "tc", M.GEMM_MMA_S8: "mma_s8",
                                            M.GEMM_IMAD: "imad"}[variant],
                           "launch": "one CUDA graph per step (fresh pass ids from a device counter)"},
        "ms_per_step_eager": round(eager_ms_max, 4),
        "parts_ms_per_step": part_ms,
        "ring_tops": round(ring_tops, 2),
        "gemm_ms": round(gemm_ms, 4),
        "init_w_s": round(init_w_s, 3),
        "roofline": roof,
        "rooflines": rooflines,
        "e2e": {"value": round(world * l / (e2e_ms_max / 1e3), 1), "unit": "tokens/s",
                "h2d_bytes_per_step": l * runner.n_in * 4, "d2h_bytes_per_step": l * runner.m_out * 4,
                "launch": "one CUDA graph per step: the copy of X in beside Init X, the previous step's "
                          "result read out beside the whole step (the last step's inside its own timing)",
                "value_eager": round(world * l / (e2e_eager_ms_max / 1e3), 1)},
        "gpu_launches": int(launches_timed),
        "kernel_ms_per_step": {k: round(v[1] / part_steps, 4) for k, v in sorted(ktimes.items())},
        "kernel_ms_note": "per-kernel event times of eager steps with the Init X calls run whole and serially",
        "clocks": clocks,
    }
    if world == 1 and not args.no_cpu_baseline:
        out["cpu_baseline"] = cpu_baseline(wk, args.cpu_budget_s)
    print(json.dumps(out), flush=True)


# Derived peaks of the client kernels that neither copy bandwidth nor the
# tensor cores bound (152 SMs at the median SM clock seen under load):
# ChaCha20 draws against 64 32-bit integer ops per clock per SM (four
# partitions of 16 INT32 lanes), the tiled gathers against one 128-byte
# shared-memory wavefront per clock per SM.
GB300_SMS = 152
INT_OPS_PER_CLK_SM = 64
SMEM_BYTES_PER_CLK_SM = 128
CHACHA_OPS_PER_BLOCK = 20 * 4 * 12 + 16   # 80 quarter rounds of 12 add/xor/rotate, 16 final adds


def _client_rooflines(kt, steps, layers, proto, l, bf16, peak_src, sm_mhz, alu_measured=None, smem_measured=None):
    """Rooflines of the client kernels from the library's per-kernel event
    times (`kt`: {"<role>:<kernel>": (launches, ms)} over `steps` eager steps).
    Algorithmic work per step, summed over the step's secure linears:
      draws   ChaCha20 blocks: R (l r_d words, 16 a block), the T lists (one
              round of 32 blocks per token and level), E_x (l n_pad samples,
              8 a block);
      gathers one 4-byte shared-memory word per gathered MAC: Init X
              l (n_pad + m) t_i per level, the unmask m l t_i per level;
      K = r_d products 20 flops (10 bf16 digit pairs) per ring MAC: Init X
              l (n_pad + m) r_d, the unmask l m r_d."""
    p = proto.params
    d = int(p.d)
    r = [int(p.r[i]) for i in range(d)]
    t = [int(p.t[i]) for i in range(d)]
    nested = int(p.act_nested) != 0
    r_act = r[d - 1] if nested else r[0]
    act_lv = list(range(1, d)) if nested else []
    w_lv = list(range(1, d))
    clk = sm_mhz * 1e6
    alu_peak = GB300_SMS * INT_OPS_PER_CLK_SM * clk / 1e12
    alu_src = "derived int32 ALU peak"
    if alu_measured:
        # The device's measured rate of the same add / xor / rotate mix.
        alu_peak = alu_measured / 1e12
        alu_src = "measured ChaCha20 mix rate (mosaic_int_mix_rate)"
    smem_peak = GB300_SMS * SMEM_BYTES_PER_CLK_SM * clk / 1e9
    smem_src = "derived shared-memory wavefront peak"
    if smem_measured:
        # The device's measured shared-memory read rate with the gather's access
        # (whole 128-byte lines, 16-byte loads, several lines a warp access).
        smem_peak = smem_measured / 1e9
        smem_src = "measured shared-memory read rate (mosaic_smem_read_rate)"
    blocks = sum(-(-l * r_act // 16) + len(act_lv) * l * 32 + -(-l * ly.n_pad // 8) for ly in layers)
    gx = sum(l * (ly.n_pad + ly.m) * t[i] for ly in layers for i in act_lv)
    gu = sum(ly.m * l * t[i] for ly in layers for i in w_lv)
    fx = sum(20 * l * (ly.n_pad + ly.m) * r_act for ly in layers)
    fu = sum(20 * l * ly.m * r[d - 1] for ly in layers)
    rows = [("init_x:initx_draw", "initx_draw_kernel (Init X draws: R, T lists, E_x; ChaCha20)", "alu",
             blocks * CHACHA_OPS_PER_BLOCK / 1e12, alu_peak, "Tops/s", alu_src),
            ("init_x:pgather", "pgather_kernel (Init X LPN terms of U_x and K)", "smem",
             gx * 4 / 1e9, smem_peak, "GB/s", smem_src),
            ("unmask:pgather", "pgather_kernel (unmask LPN terms + decode)", "smem",
             gu * 4 / 1e9, smem_peak, "GB/s", smem_src),
            ("init_x:ring_gemm_tc", "ring_gemm_tc_kernel (Init X: R [C_d; J_d]^T, K = r_d)", "tensor",
             fx / 1e12, bf16, "TFLOP/s", f"{peak_src} bf16 dense burst"),
            ("unmask:ring_gemm_tc", "ring_gemm_tc_kernel (unmask: Y' - K - Q_d L^T, K = r_d)", "tensor",
             fu / 1e12, bf16, "TFLOP/s", f"{peak_src} bf16 dense burst")]
    out = []
    for key, name, bound, work, peak, unit, src in rows:
        n, ms = kt.get(key, (0, 0.0))
        if n == 0 or ms <= 0.0 or work <= 0.0:
            continue
        ms_step = ms / steps
        achieved = work / (ms_step / 1e3)
        out.append({"kernel": name, "bound": bound, "achieved": round(achieved, 2), "peak": round(peak, 3),
                    "unit": unit, "frac": round(achieved / peak, 4), "traffic": None,
                    "ms_per_step": round(ms_step, 4), "launches_per_step": round(n / steps, 2),
                    "peak_source": src})
    return out


def _roofline(variant, M, ring_macs, gemm_ms, bf16, peak_src, traffic):
    ring_tops = 2 * ring_macs / (gemm_ms / 1e3) / 1e12
    if variant == M.GEMM_TC:
        achieved = 10 * 2 * ring_macs / (gemm_ms / 1e3) / 1e12      # bf16 digit-pair flops
        return {"bound": "tensor", "achieved": round(achieved, 2), "peak": bf16, "unit": "TFLOP/s",
                "frac": round(achieved / bf16, 4), "traffic": traffic,
                "kernel": "ring_gemm_tc (10 bf16 digit-pair products per ring MAC)",
                "peak_source": f"{peak_src} bf16 dense burst"}
    if variant == M.GEMM_MMA_S8:
        achieved = 10 * 2 * ring_macs / (gemm_ms / 1e3) / 1e12      # int8 digit-pair ops
        peak = 2 * bf16                                            # nominal int8 : bf16 = 2 : 1
        return {"bound": "tensor", "achieved": round(achieved, 2), "peak": round(peak, 3), "unit": "TOPS",
                "frac": round(achieved / peak, 4), "traffic": traffic,
                "kernel": "ring_gemm_s8 (mma.sync m16n8k32, 10 int8 digit-pair products per ring MAC)",
                "peak_source": f"{peak_src} bf16 dense burst x 2 (nominal int8 ratio)"}
    imad_peak = 152 * 64 * 2 * 2.07e9 / 1e12               # ring-ops/s: 64 IMAD/clk/SM, 2 ops each
    return {"bound": "alu", "achieved": round(ring_tops, 3), "peak": round(imad_peak, 2),
            "unit": "TOPS", "frac": round(ring_tops / imad_peak, 4), "traffic": None,
            "kernel": "ring_gemm_imad", "peak_source": "derived: 152 SMs x 64 IMAD/clk x 2070 MHz"}


def run_decode_sweep(args, rank, world, torch, M, PR, proto, dev, stream, timed, flush, wk, variant):
    """Every linear of one 70B layer at 1..256 tokens per step against
    pre-masked weights.  Init X does not depend on the input, so the masks of
    all the timed steps' tokens are drawn by one Init X call per linear before
    the steps (timed apart and charged to the steps pro rata); each step runs
    the online part: encode + mask-add, server product, unmask + decode."""
    hbm, bf16, _, peak_src = _peaks()
    t0 = time.perf_counter()
    layers = [LinearChain(proto, dev, [lin], 1, rank, timed).layers[0] for lin in wk.linears]
    init_w_s = time.perf_counter() - t0
    sweep = []
    sampler = ClockSampler(_smi_index(dev.index))
    sampler.start()
    time.sleep(0.3)
    nsteps = args.warmup + args.steps
    for l in wk.decode_batches:
        bufs = [dict(Xp=torch.empty(l, ly.n_pad, dtype=torch.int32, device=dev),
                     s_x=torch.empty(l, dtype=torch.float32, device=dev),
                     Xpl=(torch.empty(4, l, ly.n_pad, dtype=torch.int16, device=dev)
                          if ly.use_planes and l > M.STREAMW_MAX_M else None),
                     Z=torch.empty(l, ly.m + proto.sum_r, dtype=torch.int32, device=dev),
                     Y=torch.empty(l, ly.m, dtype=torch.float32, device=dev)) for ly in layers]
        xs = [torch.from_numpy(wl.activations(l, ly.n, seed=wl.SEED_X + l)).to(dev) for ly in layers]
        # Init X for every step's tokens at once (fresh randomness per token).
        flush.fill_(0)
        a = torch.cuda.Event(enable_timing=True); b = torch.cuda.Event(enable_timing=True)
        a.record(stream)
        masks = [ly.init_x(l * nsteps, 1_000_000 * (rank + 1) + 10_000 * l + i) for i, ly in enumerate(layers)]
        b.record(stream)
        torch.cuda.synchronize()
        initx_ms = a.elapsed_time(b) / nsteps

        class _Online:
            ring_macs = sum(l * (ly.m + proto.sum_r) * ly.n_pad for ly in layers)

            def step(self, x_unused, i):
                k = i % nsteps
                for ly, bf, mp, x in zip(layers, bufs, masks, xs):
                    part = PR.PassMask(mp.pass_id, l, mp.Ux[k * l:(k + 1) * l], mp.K[k * l:(k + 1) * l])
                    ly.mask_input(x, part, bf["Xp"], bf["s_x"], bf["Xpl"])
                    ly.server(bf["Xp"], bf["Xpl"], bf["Z"])
                    ly.unmask(bf["Z"], part, bf["s_x"], bf["Y"])

        runner = _Online()
        eager_ms, gemm_ms, launches, _ = _time_steps(torch, runner, lambda: None, args.steps, args.warmup, flush,
                                                  stream, timed, world, M.mosaic_kernel_launches)
        # The same steps as CUDA graphs (one per step: each reads its own rows
        # of the drawn masks), replayed without the Python launch overhead.
        graphs = []
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        for k in range(nsteps):
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=side):
                runner.step(None, k)
            graphs.append(g)
        torch.cuda.synchronize()

        class _StepReplay:
            def step(self, x_unused, i):
                graphs[i % nsteps].replay()

        online_ms, _, _, _ = _time_steps(torch, _StepReplay(), lambda: None, args.steps, args.warmup, flush, stream,
                                      timed, world)
        del graphs
        # The step's server products alone, as one CUDA graph (no host launch
        # gaps between them): the figure the HBM fraction is computed from.
        gsrv = torch.cuda.CUDAGraph()
        with torch.cuda.graph(gsrv, stream=side):
            for ly, bf in zip(layers, bufs):
                ly.server(bf["Xp"], bf["Xpl"], bf["Z"])
        torch.cuda.synchronize()
        srv = []
        for i in range(args.warmup + args.steps):
            flush.fill_(i & 0xFF)
            e0 = torch.cuda.Event(enable_timing=True); e1 = torch.cuda.Event(enable_timing=True)
            e0.record(stream); gsrv.replay(); e1.record(stream)
            if i >= args.warmup:
                srv.append((e0, e1))
        torch.cuda.synchronize()
        server_ms = float(np.mean([a.elapsed_time(b) for a, b in srv]))
        del gsrv
        # Per-kernel device time of a few eager online steps (the library's own
        # event pair around each launch): the server kernel's time alone.
        kt_steps = 3
        M.mosaic_kernel_times(reset=True)
        M.mosaic_kernel_timing(True)
        for i in range(kt_steps):
            flush.fill_(i & 0xFF)
            runner.step(None, i)
        torch.cuda.synchronize()
        M.mosaic_kernel_timing(False)
        kt = M.mosaic_kernel_times(reset=True)
        step_ms = online_ms + initx_ms
        del masks
        w_bytes = sum((ly.m + proto.sum_r) * ly.n_pad * 4 for ly in layers)
        # up to STREAMW_MAX_M tokens the server streams uint32 W' (4 B an element:
        # CUDA cores up to 8 tokens, tensor cores from 9), beyond that
        # the tensor cores read its bf16 digit planes (8 B an element)
        skinny = variant != M.GEMM_IMAD and l <= M.SKINNY_MAX_M
        streamw = variant != M.GEMM_IMAD and M.SKINNY_MAX_M < l <= M.STREAMW_MAX_M
        read_bytes = w_bytes if skinny or streamw or variant == M.GEMM_IMAD else 2 * w_bytes
        sweep.append({"l": l, "ms_per_step": round(step_ms, 4), "tokens_s": round(world * l / (step_ms / 1e3), 1),
                      "online_ms": round(online_ms, 4), "online_ms_eager": round(eager_ms, 4),
                      "init_x_ms_per_step": round(initx_ms, 4),
                      "gpu_launches_per_step": int(round(launches / args.steps)),
                      "gemm_ms_eager": round(gemm_ms, 4), "server_ms": round(server_ms, 4),
                      "ring_tops": round(2 * runner.ring_macs / (server_ms / 1e3) / 1e12, 2),
                      "server_kernel": "ring_gemm_skinny" if skinny else "ring_gemm_tcw" if streamw else
                                       ("ring_gemm_imad" if variant == M.GEMM_IMAD else "ring_gemm_tc"),
                      "w_prime_bytes": w_bytes, "server_read_bytes": read_bytes,
                      "server_read_gbs": round(read_bytes / (server_ms / 1e3) / 1e9, 1),
                      "server_hbm_frac": round(read_bytes / (server_ms / 1e3) / 1e9 / hbm, 4),
                      "kernel_ms_per_step": {k: round(v[1] / kt_steps, 4) for k, v in sorted(kt.items())}})
        skey = "ring_gemm:" + sweep[-1]["server_kernel"]
        if skey in kt and kt[skey][1] > 0:
            kms = kt[skey][1] / kt_steps
            sweep[-1]["server_kernel_ms"] = round(kms, 4)
            sweep[-1]["server_kernel_hbm_frac"] = round(read_bytes / (kms / 1e3) / 1e9 / hbm, 4)
    clocks = sampler.stop()
    M.mosaic_device_status()
    if rank != 0:
        return
    first = sweep[0]
    out = {"metric": METRIC, "value": first["tokens_s"], "unit": "tokens/s", "n_gpus": world,
           "steps": args.steps, "warmup": args.warmup, "ms_per_step": first["ms_per_step"],
           "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "u32",
           "data": "synthetic (seeded N(0,1) activations, N(0,0.02) weights)",
           "config": {"workload": args.workload, "batches": list(wk.decode_batches),
                      "linears": [{"name": x.name, "m": x.m, "n": x.n} for x in wk.linears],
                      "params": "Example 3.1", "l2": "flushed between timed steps (256 MiB write)",
                      "step": "online part (encode, server product, unmask) of every linear, one CUDA "
                              "graph per step, + Init X of the step's tokens, drawn ahead for all steps in "
                              "one call per linear and charged pro rata"},
           "init_w_s": round(init_w_s, 3), "sweep": sweep,
           "gpu_launches": first["gpu_launches_per_step"] * args.steps,
           "roofline": {"bound": "hbm", "achieved": first["server_read_gbs"], "peak": hbm, "unit": "GB/s",
                        "frac": first["server_hbm_frac"], "traffic": None, "peak_source": peak_src,
                        "kernel": first["server_kernel"] + " at %d token(s): reads of the server operand"
                                  % first["l"]},
           "clocks": clocks}
    print(json.dumps(out), flush=True)


def run_matvec_sweep(args, rank, world, torch, M, PR, proto, dev, stream, flush, wk):
    """Secure mat-vec (one token) per n x n: device time of Init X, encode,
    server product and unmask, each bracketed by CUDA events on the stream."""
    hbm, _, _, peak_src = _peaks()
    sweep = []
    sampler = ClockSampler(_smi_index(dev.index))
    sampler.start()
    for lin in wk.linears:
        n_pad = PR.pad_width(lin.n)
        ch = PR.Chains(proto, n_pad)
        W = torch.from_numpy(wl.weights(lin.m, lin.n)).to(dev)
        layer = PR.SecureLinear(proto, W, 1, ch, planes=False)   # one token: no digit planes
        del W
        X = torch.from_numpy(wl.activations(1, lin.n, seed=wl.SEED_X + rank)).to(dev)
        Sr = proto.sum_r
        Xp = torch.empty(1, n_pad, dtype=torch.int32, device=dev)
        s_x = torch.empty(1, dtype=torch.float32, device=dev)
        Z = torch.empty(1, lin.m + Sr, dtype=torch.int32, device=dev)
        Y = torch.empty(1, lin.m, dtype=torch.float32, device=dev)
        parts = []
        for i in range(args.warmup + args.steps):
            flush.fill_(i & 0xFF)
            ev = [torch.cuda.Event(enable_timing=True) for _ in range(5)]
            ev[0].record(stream)
            mp = layer.init_x(1, 1_000_000 * rank + i)
            ev[1].record(stream)
            layer.mask_input(X, mp, Xp, s_x, None)
            ev[2].record(stream)
            layer.server(Xp, None, Z)
            ev[3].record(stream)
            layer.unmask(Z, mp, s_x, Y)
            ev[4].record(stream)
            if i >= args.warmup:
                parts.append(ev)
        torch.cuda.synchronize()
        ms = np.mean([[a.elapsed_time(b) for a, b in zip(ev[:-1], ev[1:])] for ev in parts], axis=0)
        w_bytes = (lin.m + Sr) * n_pad * 4
        sweep.append({"n": lin.n, "n_pad": n_pad, "init_x_ms": round(ms[0], 4), "encode_ms": round(ms[1], 4),
                      "server_ms": round(ms[2], 4), "unmask_ms": round(ms[3], 4),
                      "client_online_ms": round(ms[1] + ms[3], 4), "step_ms": round(float(ms.sum()), 4),
                      "server_gbs": round(w_bytes / (ms[2] / 1e3) / 1e9, 1),
                      "server_hbm_frac": round(w_bytes / (ms[2] / 1e3) / 1e9 / hbm, 4),
                      "server_ring_gops": round(2 * lin.m * lin.n / (ms[2] / 1e3) / 1e9, 1)})
        del layer, ch, Xp, Z, Y
        torch.cuda.empty_cache()
    clocks = sampler.stop()
    M.mosaic_device_status()
    if rank != 0:
        return
    first = sweep[0]
    out = {"metric": METRIC, "value": round(world * 1e3 / first["step_ms"], 1), "unit": "tokens/s",
           "n_gpus": world, "steps": args.steps, "warmup": args.warmup, "ms_per_step": first["step_ms"],
           "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "u32",
           "data": "synthetic (seeded N(0,1) activation vector, N(0,0.02) weights)",
           "config": {"workload": wk.name, "l": 1, "sizes": [x.n for x in wk.linears],
                      "params": "Example 3.1", "l2": "flushed between steps (256 MiB write)",
                      "note": "parts timed by CUDA events between the launches; Init X is "
                              "independent of the input and can be precomputed"},
           "sweep": sweep,
           "roofline": {"bound": "hbm", "achieved": first["server_gbs"], "peak": hbm, "unit": "GB/s",
                        "frac": first["server_hbm_frac"], "traffic": None, "peak_source": peak_src,
                        "kernel": "ring_gemm_skinny (server product, n = %d)" % first["n"]},
           "clocks": clocks}
    print(json.dumps(out), flush=True)


def run_sigma_sweep(args, rank, world, torch, M, PR, dev, wk, variant):
    """Relative l2 error of one secure linear call against the fp64 product
    W X + b, per sigma and activation-mask variant (the paper's single-layer
    error table, on synthetic weights with outlier channels)."""
    sigmas = (0.0, 0.5, 0.7, 1.0, 1.5, 2.0)
    key = wl.mask_key()
    base = PR.Protocol(key, M.default_params(), variant=variant)
    chains = {}
    data = []
    for i, lin in enumerate(wk.linears):
        n_pad = PR.pad_width(lin.n)
        if n_pad not in chains:
            chains[n_pad] = PR.Chains(base, n_pad)
        W = wl.outlier_weights(lin.m, lin.n, seed=wl.SEED_W + i)
        X = wl.spike_activations(wk.l, lin.n, seed=wl.SEED_X + i, outlier=20.0, channels=4)
        b = wl.bias(lin.m, seed=wl.SEED_B + i)
        Wd, Xd, bd = (torch.from_numpy(a).to(dev) for a in (W, X, b))
        ref = Xd.double() @ Wd.double().T + bd.double()[None, :]
        data.append((lin, Wd, Xd, bd, ref, n_pad))
    rows = []
    t0 = time.perf_counter()
    for act_nested in (1, 0):
        for sigma in sigmas:
            proto = PR.Protocol(key, M.default_params(sigma=sigma, act_nested=act_nested), variant=variant)
            errs = []
            for i, (lin, Wd, Xd, bd, ref, n_pad) in enumerate(data):
                ch = chains[n_pad]
                ch.proto = proto
                layer = PR.SecureLinear(proto, Wd, 100 + i, ch, bias=bd)
                mp = layer.init_x(wk.l, 7 + i)
                Y = layer.forward(Xd, mp)
                err = torch.linalg.vector_norm(Y.double() - ref) / torch.linalg.vector_norm(ref)
                errs.append(100.0 * float(err))
                del layer, mp, Y
            rows.append({"act_nested": act_nested, "sigma": sigma,
                         "rel_l2_pct": {"mean": round(float(np.mean(errs)), 4),
                                        "median": round(float(np.median(errs)), 4),
                                        "max": round(float(np.max(errs)), 4)},
                         "per_linear_pct": {lin.name: round(e, 4) for (lin, *_), e in zip(data, errs)}})
    M.mosaic_device_status()
    if rank != 0:
        return
    out = {"metric": "single secure linear relative l2 error (%) vs fp64 W X + b",
           "value": rows[1]["rel_l2_pct"]["mean"], "unit": "%", "n_gpus": world, "steps": 1, "warmup": 0,
           "higher_is_better": False, "scaling": "weak", "vs_baseline": None, "dtype": "u32",
           "data": "synthetic: N(0,0.02) weights with 8 outlier input channels (10x), N(0,1) "
                   "activations with 4 outlier channels (20x), N(0,0.02) bias",
           "config": {"workload": wk.name, "l": wk.l,
                      "linears": [{"name": x.name, "m": x.m, "n": x.n} for x in wk.linears],
                      "sigmas": list(sigmas), "value_is": "mean over linears at sigma 0.5, nested mask"},
           "sweep": rows, "wall_s": round(time.perf_counter() - t0, 2)}
    print(json.dumps(out), flush=True)


def run_kernels_hbm(args, rank, world, torch, M, PR, proto, dev, stream, flush, wk):
    """The memory-bound client kernels alone: CUDA events around each launch,
    L2 flushed (256 MiB write) before each; bytes are the algorithmic HBM
    traffic per launch."""
    hbm, _, _, peak_src = _peaks()
    key = M.make_key(wl.mask_key())
    rows = []
    sampler = ClockSampler(_smi_index(dev.index))
    sampler.start()
    # Two batches per width: the workload's, and 4x as many rows, where the
    # fixed cost of a launch (a few us) no longer hides the streaming rate.
    shapes = []
    for lin in wk.linears:
        n_pad = PR.pad_width(lin.n)
        l0 = wk.l if n_pad <= 16384 else wk.l // 2
        shapes += [(n_pad, l0), (n_pad, 4 * l0)]
    for n_pad, l in shapes:
        x = torch.from_numpy(wl.activations(l, n_pad, seed=wl.SEED_X)).to(dev)
        y = torch.empty_like(x)
        mask = torch.randint(-2**31, 2**31 - 1, (l, n_pad), dtype=torch.int32, device=dev)
        out = torch.empty(l, n_pad, dtype=torch.int32, device=dev)
        planes = torch.empty(4, l, n_pad, dtype=torch.int16, device=dev)
        scale = torch.empty(l, dtype=torch.float32, device=dev)
        signs = torch.randint(-2**31, 2**31 - 1, (n_pad // 32,), dtype=torch.int32, device=dev)
        qmax = M.mosaic_qmax(n_pad, 16)
        elems = l * n_pad
        cases = [
            ("mosaic_hadamard", 8, lambda: M.mosaic_hadamard(x, n_pad, y, l, n_pad, n_pad, signs)),
            ("mosaic_encode (rotate, quantise, + U_x)", 12,
             lambda: M.mosaic_encode(x, n_pad, l, n_pad, n_pad, qmax, 1, signs, mask, n_pad, out, n_pad, scale)),
            ("mosaic_encode (+ digit planes)", 20,
             lambda: M.mosaic_encode(x, n_pad, l, n_pad, n_pad, qmax, 1, signs, mask, n_pad, out, n_pad, scale,
                                     planes)),
            ("mosaic_prg_gaussian (E_x, ChaCha20)", 4,
             lambda: M.mosaic_prg_gaussian(key, M.TAG_EX, 5, 20, 0.5, elems, out)),
        ]
        for name, bpe, fn in cases:
            for _ in range(args.warmup):
                fn()
            evs = []
            for i in range(args.steps):
                flush.fill_(i & 0xFF)
                a = torch.cuda.Event(enable_timing=True); b = torch.cuda.Event(enable_timing=True)
                a.record(stream); fn(); b.record(stream)
                evs.append((a, b))
            torch.cuda.synchronize()
            ms = float(np.median([a.elapsed_time(b) for a, b in evs]))
            gbs = bpe * elems / (ms / 1e3) / 1e9
            rows.append({"kernel": name, "l": l, "n_pad": n_pad, "bytes_per_elem": bpe, "us": round(ms * 1e3, 2),
                         "gbs": round(gbs, 1), "hbm_frac": round(gbs / hbm, 4)})
        del x, y, mask, out, planes
        torch.cuda.empty_cache()
    clocks = sampler.stop()
    M.mosaic_device_status()
    if rank != 0:
        return
    enc = [r for r in rows if r["kernel"].startswith("mosaic_encode (rotate")]
    best = max(enc, key=lambda r: r["gbs"])
    out = {"metric": "memory-bound client kernels: achieved HBM GB/s", "value": best["gbs"], "unit": "GB/s",
           "n_gpus": world, "steps": args.steps, "warmup": args.warmup, "higher_is_better": True,
           "scaling": "weak", "vs_baseline": None, "dtype": "f32/u32", "data": "synthetic N(0,1) rows",
           "config": {"workload": wk.name, "shapes": [[r["l"], r["n_pad"]] for r in rows[::4]],
                      "l2": "flushed before each launch (256 MiB write)", "timing": "median of steps"},
           "kernels": rows,
           "roofline": {"bound": "hbm", "achieved": best["gbs"], "peak": hbm, "unit": "GB/s",
                        "frac": best["hbm_frac"], "traffic": None, "peak_source": peak_src,
                        "kernel": "fwht_kernel encode mode (%d x %d)" % (best["l"], best["n_pad"])},
           "clocks": clocks}
    print(json.dumps(out), flush=True)


def run_init_w(args, rank, world, torch, M, PR, proto, dev, wk):
    """One-time Init W of a 70B layer: the public chains per rotation width
    (shared by every layer) and the four matrices' masking, extrapolated to
    an 80-layer model (the paper quotes about 55 s per 70B model)."""
    layers = 80
    chains_s, chains = {}, {}
    for lin in wk.linears:
        n_pad = PR.pad_width(lin.n)
        if n_pad in chains:
            continue
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        chains[n_pad] = PR.Chains(proto, n_pad)
        torch.cuda.synchronize()
        chains_s[n_pad] = time.perf_counter() - t0
    mats = []
    Sr, rd = proto.sum_r, proto.ranks[-1]
    for i, lin in enumerate(wk.linears):
        n_pad = PR.pad_width(lin.n)
        W = torch.from_numpy(wl.weights(lin.m, lin.n, seed=wl.SEED_W + i)).to(dev)
        PR.SecureLinear(proto, W[:64].contiguous(), 999, chains[n_pad])      # warm-up of every kernel
        times = []
        for rep in range(2):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            layer = PR.SecureLinear(proto, W, 1 + i, chains[n_pad])
            torch.cuda.synchronize()
            times.append(time.perf_counter() - t0)
            del layer
        server_b = (lin.m + Sr) * n_pad * 4
        client_b = lin.m * (Sr + rd) * 4 + proto.sparse_words(lin.m) * 8 + lin.m * 4 + n_pad // 8
        mats.append({"name": lin.name, "m": lin.m, "n": lin.n, "n_pad": n_pad, "init_w_s": round(min(times), 4),
                     "server_state_bytes": server_b, "server_plane_bytes": 2 * server_b,
                     "client_state_bytes": client_b})
        del W
        torch.cuda.empty_cache()
    M.mosaic_device_status()
    if rank != 0:
        return
    layer_s = sum(x["init_w_s"] for x in mats)
    ch_s = sum(chains_s.values())
    model_s = ch_s + layers * layer_s
    out = {"metric": "Init W time of a 70B model (s), extrapolated from one layer",
           "value": round(model_s, 2), "unit": "s", "n_gpus": world, "steps": 1, "warmup": 1,
           "higher_is_better": False, "scaling": "weak", "vs_baseline": round(model_s / 55.0, 3),
           "dtype": "u32", "data": "synthetic N(0,0.02) weights",
           "config": {"workload": wk.name, "layers": layers, "params": "Example 3.1",
                      "linears": [{"name": x.name, "m": x.m, "n": x.n} for x in wk.linears]},
           "chains_s": {str(k): round(v, 3) for k, v in chains_s.items()},
           "layer_s": round(layer_s, 4), "matrices": mats,
           "paper_s": 55.0}
    print(json.dumps(out), flush=True)


def _smi_index(dev_index: int) -> int:
    vis = os.environ.get("CUDA_VISIBLE_DEVICES", "")
    parts = [p for p in vis.split(",") if p.strip()]
    if parts and all(p.strip().isdigit() for p in parts) and dev_index < len(parts):
        return int(parts[dev_index])
    return dev_index


def _barrier(world):
    if world > 1:
        import torch.distributed as dist
        dist.barrier()


def _max_over_ranks(v, world, dev):
    if world == 1:
        return v
    import torch
    import torch.distributed as dist
    t = torch.tensor([v], dtype=torch.float64, device=dev)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


# ---------------------------------------------------------------------------
# CPU oracle as baseline / reference arm
# ---------------------------------------------------------------------------
ORACLE_TOKENS = 16           # tokens per sampled oracle step
ORACLE_ROWS = 256            # output rows per linear where Init W in full is out of reach
ORACLE_FULL_INIT_MACS = 6e10  # Init W (J = (W_hat + E_w) C) up to this many MACs runs on every row


def _linear_weights_seed(wk, i):
    """Seed and std of linear i's float weights, as the GPU arm draws them."""
    if wk.name == "decoder_70b_prefill_2048":
        return DECODER_SEED + i, 0.02
    return wl.SEED_W + i, wk.linears[i].w_std


def _oracle_setup(wk, tokens):
    """One-time oracle state of every linear of the workload: the public chains
    in full, and Init W on all rows or on ORACLE_ROWS evenly spaced rows
    (oracle.sampled).  Not timed (the GPU arm's Init W is timed apart too)."""
    import oracle as O
    from oracle import sampled as OS
    key = wl.mask_key()
    p = O.Params()
    chains = {}
    plan = []
    t0 = time.perf_counter()
    for i, lin in enumerate(wk.linears):
        n_pad = 1 << max(5, (lin.n - 1).bit_length())
        if n_pad not in chains:
            chains[n_pad] = O.chains(key, p, n_pad)
        P, C = chains[n_pad]
        if lin.m * n_pad * sum(p.r) <= ORACLE_FULL_INIT_MACS:
            rows = np.arange(lin.m)
        else:
            rows = np.unique(np.linspace(0, lin.m - 1, ORACLE_ROWS).astype(np.int64))
        seed, std = _linear_weights_seed(wk, i)
        W_rows = wl.weight_rows(lin.m, lin.n, rows, seed=seed, std=std)
        wr = OS.weight_rows(key, p, W_rows, rows, 1 + i, P, C, n_pad)
        X = wl.activations(tokens, lin.n, seed=wl.SEED_X + i)
        b = wl.bias(lin.m, seed=wl.SEED_B + i)[rows]
        plan.append(dict(lin=lin, n_pad=n_pad, P=P, C=C, wr=wr, X=X, b=b, rows=rows))
    return O, OS, key, p, plan, time.perf_counter() - t0


def _oracle_step(O, OS, key, p, plan, pass_id):
    """One sampled oracle step: every linear's Init X, encode + mask-add, server
    product, unmask and decode for the sample's tokens, over the sampled rows.
    Returns the seconds the whole step (all rows) takes for those tokens: the
    per-token part (Init X draws and U_x, encode, Q_i = P_i X') as measured,
    the per-(row, token) part (K, Y', unmask, decode) scaled by m / rows."""
    total = 0.0
    for st in plan:
        k = st["X"].shape[0]
        wr = st["wr"]
        t0 = time.perf_counter()
        tc = OS.token_cols(key, p, st["X"], np.arange(k), pass_id, wr.sign_words, wr.qmax, st["C"], st["n_pad"])
        Q = OS.server_q(tc, st["P"])
        t1 = time.perf_counter()
        K = OS.k_entries(p, wr, tc)
        Ym = OS.server_rows(wr, tc)
        Yh = OS.unmask_entries(p, wr, K, Ym, Q)
        O.decode(Yh, wr.s_w, tc.s_x, st["b"])
        t2 = time.perf_counter()
        total += (t1 - t0) + (t2 - t1) * st["lin"].m / len(st["rows"])
    return total


def _oracle_sample_text(wk, plan, k, extra=""):
    rows = ", ".join(f"{st['lin'].name} {len(st['rows'])}/{st['lin'].m}" for st in plan)
    glue = "; fp32 glue not included" if wk.name == "decoder_70b_prefill_2048" else ""
    return (f"{k} of {wk.l} tokens per step through every linear (rows computed: {rows}); "
            f"per-token work (Init X draws, U_x, encode, Q_i = P_i X') timed as run, per-(row, token) "
            f"work (K, Y', unmask, decode) scaled by m / rows computed{glue}; seeded N(0,1) inputs of "
            f"each linear's width; one-time chains + Init W excluded like the GPU value{extra}")


def cpu_baseline(wk, budget_s):
    O, OS, key, p, plan, init_s = _oracle_setup(wk, ORACLE_TOKENS)
    k = ORACLE_TOKENS
    done, secs, t0 = 0, 0.0, time.perf_counter()
    while True:
        secs += _oracle_step(O, OS, key, p, plan, 500 + done)
        done += 1
        if time.perf_counter() - t0 >= budget_s:
            break
    return {"value": round(done * k / secs, 3), "unit": "tokens/s", "cores": O.num_threads(),
            "kind": "oracle",
            "sample": _oracle_sample_text(wk, plan, k, f" ({done} sampled steps, {init_s:.1f} s of setup)"),
            "init_w_s": round(init_s, 2)}


def run_reference(args, rank, world):
    """The reference arm: the oracle as it stands, on the host cores, on the
    same workload, metric and config as the GPU arm; each step one sampled
    oracle step (rank 0 only)."""
    if rank != 0:
        return
    wk = wl.WORKLOADS[args.workload]
    if not wk.linears or wk.l < 1 or wk.name in ("decode_70b_sweep", "matvec_sweep", "sigma_sweep_7b",
                                                  "kernels_hbm", "init_w_70b"):
        print(json.dumps({"impl": "reference", "unavailable": f"no oracle step for workload {wk.name}"}))
        return
    O, OS, key, p, plan, init_s = _oracle_setup(wk, ORACLE_TOKENS)
    k = ORACLE_TOKENS
    for i in range(args.warmup):
        _oracle_step(O, OS, key, p, plan, 900 + i)
    secs = [_oracle_step(O, OS, key, p, plan, 950 + i) for i in range(args.steps)]
    val = k / float(np.mean(secs))
    out = {"impl": "reference", "metric": METRIC, "value": round(val, 3), "unit": "tokens/s",
           "n_gpus": world, "steps": args.steps, "warmup": args.warmup,
           "ms_per_step": round(wk.l / val * 1e3, 3), "higher_is_better": True, "scaling": "weak",
           "vs_baseline": None, "dtype": "u32", "data": "synthetic",
           "config": _config(wk, world),
           "cpu_baseline": {"value": round(val, 3), "unit": "tokens/s", "cores": O.num_threads(),
                            "kind": "oracle", "sample": _oracle_sample_text(wk, plan, k,
                                                                            f" ({init_s:.1f} s of setup)")},
           "e2e": {"value": round(val, 3), "unit": "tokens/s", "h2d_bytes_per_step": 0,
                   "d2h_bytes_per_step": 0}}
    print(json.dumps(out), flush=True)


def main():
    args = parse()
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    if args.impl == "reference":
        run_reference(args, rank, world)
        return
    if world > 1:
        import torch
        import torch.distributed as dist
        torch.cuda.set_device(int(os.environ.get("LOCAL_RANK", 0)))
        dist.init_process_group("nccl")
    try:
        run_mine(args, rank, world)
    finally:
        if world > 1:
            import torch.distributed as dist
            dist.destroy_process_group()


if __name__ == "__main__":
    main()
