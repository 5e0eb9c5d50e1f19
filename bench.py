#!/usr/bin/env python
"""Benchmark of the streaming span-retrieval attention path on B200.

A step is one `ltri_prefill_chunk` call: one chunk of the workload's stream through every
layer (append, evict + index, local attention, local-map pass, segmentation, scoring +
top-k, gather + retrieved attention).  The timed steps are the LAST K chunks of the
context, so the reported prefill throughput is the one at full context length; the chunks
before them are streamed untimed as set-up.  After the prefill measurement the workload's
decode steps are timed the same way and reported under "decode".

    python bench.py [--gpus N] [--steps K] [--warmup W] [--config C] [--impl ltri|reference]

With N > 1 (launched by torchrun, one rank per GPU) every rank streams its own replica of
the workload; nothing is exchanged (the path does not shard: replicas only).
"""
from __future__ import annotations

import argparse
import json
import os
import statistics
import subprocess
import sys
import threading
import time

import numpy as np
import torch

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

from paper_2412_04757_b200 import inputs  # noqa: E402

METRIC = "streamed prefill tok/s at full context (decode tok/s and roofline fractions alongside)"


def measured_peaks():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(path):
        with open(path) as f:
            p = json.load(f)
        return {"hbm_gbs": p["hbm_gbs"], "bf16_tflops": p["bf16_tflops"],
                "bf16_tflops_sustained": p.get("bf16_tflops_sustained", p["bf16_tflops"]), "source": "measured"}
    return {"hbm_gbs": 6650.0, "bf16_tflops": 1590.0, "bf16_tflops_sustained": 1400.0, "source": "fallback"}


class ClockSampler:
    """Samples SM clocks and throttle reasons while the timed region runs (read-only NVML queries every 20 ms;
    falls back to `nvidia-smi -lms 200` when the NVML binding is missing)."""

    Q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,clocks_event_reasons.hw_slowdown,"
         "clocks_event_reasons.hw_thermal_slowdown,clocks_event_reasons.sw_thermal_slowdown,"
         "clocks_event_reasons.sw_power_cap")

    def __init__(self, index: int):
        self.index = index
        self.proc = None
        self.lines = []
        self.samples = []       # (sm_mhz, reasons bitmask, power W)
        self.stop_flag = False
        self.nvml = None
        self.thread = None

    def start(self):
        try:
            import pynvml
            pynvml.nvmlInit()
            self.nvml = pynvml
            vis = os.environ.get("CUDA_VISIBLE_DEVICES")
            phys = self.index
            if vis:
                try:
                    phys = int(vis.split(",")[self.index])
                except ValueError:
                    phys = self.index
            self.handle = pynvml.nvmlDeviceGetHandleByIndex(phys)
            self.sm_max = pynvml.nvmlDeviceGetMaxClockInfo(self.handle, pynvml.NVML_CLOCK_SM)
            self.thread = threading.Thread(target=self._poll, daemon=True)
            self.thread.start()
            return
        except Exception:
            self.nvml = None
        try:
            self.proc = subprocess.Popen(["nvidia-smi", f"--id={self.index}", f"--query-gpu={self.Q}",
                                          "--format=csv,noheader,nounits", "-lms", "200"],
                                         stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.thread = threading.Thread(target=self._read, daemon=True)
            self.thread.start()
        except Exception:
            self.proc = None

    def _poll(self):
        n = self.nvml
        while not self.stop_flag:
            try:
                mhz = n.nvmlDeviceGetClockInfo(self.handle, n.NVML_CLOCK_SM)
                reasons = n.nvmlDeviceGetCurrentClocksEventReasons(self.handle)
                watts = n.nvmlDeviceGetPowerUsage(self.handle) / 1000.0
                self.samples.append((mhz, reasons, watts))
            except Exception:
                pass
            time.sleep(0.02)

    def _read(self):
        for line in self.proc.stdout:
            self.lines.append(line.strip())

    def mark(self):
        """Index of the next sample (to restrict the summary to a window)."""
        return len(self.samples)

    def stop(self, lo=0, hi=None):
        if self.nvml is not None:
            self.stop_flag = True
            self.thread.join(timeout=2)
            n = self.nvml
            win = self.samples[lo:hi] or self.samples
            sm = [s[0] for s in win]
            names = {"hw_slowdown": n.nvmlClocksEventReasonHwSlowdown,
                     "hw_thermal_slowdown": n.nvmlClocksEventReasonHwThermalSlowdown,
                     "sw_thermal_slowdown": n.nvmlClocksEventReasonSwThermalSlowdown,
                     "sw_power_cap": n.nvmlClocksEventReasonSwPowerCap}
            reasons = sorted(k for k, bit in names.items() if any(s[1] & bit for s in win))
            return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": float(self.sm_max),
                    "samples": len(sm), "power_w_max": max((s[2] for s in win), default=None), "reasons": reasons,
                    "source": "nvml, 20 ms"}
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["no clock source available"]}
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except Exception:
            self.proc.kill()
        sm, smax, reasons = [], [], set()
        for ln in self.lines:
            f = [x.strip() for x in ln.split(",")]
            if len(f) < 9:
                continue
            try:
                sm.append(float(f[1]))
                smax.append(float(f[2]))
            except ValueError:
                continue
            for name, val in zip(["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"], f[5:9]):
                if val.lower().startswith("active"):
                    reasons.add(name)
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": max(smax) if smax else None,
                "samples": len(sm), "reasons": sorted(reasons), "source": "nvidia-smi -lms 200"}


def dist_setup(n_gpus):
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    world = int(os.environ.get("WORLD_SIZE", "1"))
    if world > 1:
        import torch.distributed as dist
        os.environ.setdefault("MASTER_ADDR", "127.0.0.1")
        dist.init_process_group("nccl" if torch.cuda.is_available() else "gloo")
    return rank, local, world


def barrier(world):
    if world > 1:
        import torch.distributed as dist
        dist.barrier()


def max_over_ranks(x: float, world, device):
    if world == 1:
        return x
    import torch.distributed as dist
    t = torch.tensor([x], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def sum_over_ranks(x: float, world, device):
    if world == 1:
        return x
    import torch.distributed as dist
    t = torch.tensor([x], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.SUM)
    return float(t.item())


# ------------------------------------------------------------------------------------------------
def oracle_sample(cfg, steps, warmup):
    """Time the CPU oracle, as it stands, on a bounded sample of the workload: layer 0 of the first
    prefill calls of the stream until the window is full, then `steps` timed calls.  Returns tok/s
    extrapolated to all layers, the cores it ran on and a description of the sample."""
    from oracle import ltri_oracle as orc  # test infrastructure: only this CPU-baseline leg touches it

    one = inputs.StreamConfig(**{**cfg.__dict__, "n_layers": 1, "n_seqs": 1})
    st = inputs.SyntheticStream(one)
    fill = (cfg.window + cfg.chunk - 1) // cfg.chunk + 1
    need = (fill + warmup + steps) * cfg.chunk
    o = orc.OracleStream(cfg.n_q_heads, cfg.n_kv_heads, cfg.head_dim, cfg.chunk, cfg.window, cfg.n_sink, cfg.top_k,
                         need + 8, reps_per_span=cfg.reps_per_span, max_spans_per_region=cfg.max_spans_per_region,
                         theta_mode=cfg.theta_mode, theta=cfg.layer_theta[0] if cfg.layer_theta else cfg.theta,
                         rep_mode=cfg.rep_mode, ratio_kind=cfg.ratio_kind, min_reps=cfg.min_reps, max_reps=cfg.max_reps,
                         rep_lambda=cfg.layer_rep_lambda[0] if cfg.layer_rep_lambda else cfg.rep_lambda,
                         unit_tokens=cfg.unit_tokens, persist_decode=int(cfg.persist_decode),
                         nms_iou_milli=cfg.layer_nms_iou_milli[0] if cfg.layer_nms_iou_milli else cfg.nms_iou_milli,
                         ret_head=cfg.retrieval_head[0] if cfg.retrieval_head else -1,
                         head_weight=cfg.retrieval_head_score[0] if cfg.retrieval_head_score else 1.0,
                         collab_vote=int(cfg.collab_vote), segment_per_unit=int(cfg.segment_per_unit))
    times = []
    for ci in range(fill + warmup + steps):
        q, k, v = st.tokens(ci * cfg.chunk, cfg.chunk)
        t = time.perf_counter()
        if ci < fill:
            o.prefill_local(q[0], k[0], v[0])      # state only: fills the window and the index
            o.prefill_retrieve()
        else:
            o.prefill_chunk(q[0], k[0], v[0])
        dt = time.perf_counter() - t
        if ci >= fill + warmup:
            times.append(dt)
    per_call_layer = sum(times) / len(times)
    toks = cfg.chunk / (per_call_layer * cfg.n_layers)
    cores = min(cfg.n_q_heads, os.cpu_count() or 1)
    sample = (f"layer 0 of {cfg.name}: {steps} full prefill calls of {cfg.chunk} tokens with the {cfg.window}-token "
              f"window full (after {fill} state-only calls), time x {cfg.n_layers} layers")
    return toks, cores, sample, per_call_layer


def run_reference(args, cfg):
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return
    steps = max(1, min(args.steps, 4))
    warm = min(args.warmup, 1)
    toks, cores, sample, per = oracle_sample(cfg, steps, warm)
    # a step of this arm is what the oracle was actually timed on: one 512-token call of ONE layer; the all-layer
    # figure is that time x layers and lives in `value` / `sample` only
    line = {
        "impl": "reference", "metric": METRIC, "value": toks, "unit": "tok/s", "n_gpus": args.gpus,
        "steps": steps, "warmup": warm, "ms_per_step": per * 1e3, "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "f32", "data": "synthetic",
        "config": {**workload_config(cfg, 1, 1), "timed": "layer 0 only; value = chunk / (ms_per_step x layers)"},
        "cpu_baseline": {"value": toks, "unit": "tok/s", "cores": cores, "kind": "oracle", "sample": sample},
        "e2e": {"value": toks, "unit": "tok/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }
    print(json.dumps(line))


def workload_config(cfg, world, nseq):
    return {"workload": cfg.name, "layers": cfg.n_layers, "q_heads": cfg.n_q_heads, "kv_heads": cfg.n_kv_heads,
            "context": cfg.context, "chunk": cfg.chunk, "window": cfg.window, "sink": cfg.n_sink, "top_k": cfg.top_k,
            "parallelism": "replicas only" if world > 1 else "single GPU", "sequences": nseq}


# ------------------------------------------------------------------------------------------------
# DRAM traffic measured by Nsight Compute on small cases of the same kernels, expressed per unit so that it can be
# scaled to the launch this run times (traffic grows in proportion to these units):
#  * local attention (k_attn_tc phase 0), Llama-3-8B geometry, chunk 512, window 4096 full, sink 64: DRAM read +
#    write of one launch over 4 layers at 16K context -> bytes per layer of a launch
ATTN_LOCAL_DRAM_BYTES_PER_LAYER = {(32, 8, 512, 4096, 64): (93.74e6 + 6.56e6) / 4}
#  * decode retrieval + attention: 240.0 MB measured against 237.8 MB of algorithmic bytes for an 8-layer step at
#    64K: every byte is read once, nothing is re-read
DECODE_DRAM_PER_ALGORITHMIC_BYTE = 240.0 / 237.8
NOMINAL_BF16_TFLOPS = 2250.0   # dense bf16, per GPU
NOMINAL_HBM_GBS = 8000.0


def local_keys(cfg, t0, n, E):
    """Keys a row of the call sees in the local part, averaged over the rows: sink + local + causal current."""
    return min(cfg.n_sink, t0) + (t0 - min(E, t0)) + (n + 1) / 2.0


def attn_local_flops(cfg, t0, n, E):
    """Algorithmic flops of the local attention kernel for one call (all layers): QK^T + PV over
    sink + local + causal current keys."""
    return 4.0 * n * cfg.n_q_heads * cfg.head_dim * local_keys(cfg, t0, n, E) * cfg.n_layers


def map_pass_flops(cfg, t0, n, E):
    """Algorithmic flops of the local-map pass for one call (all layers): QK^T over local + causal current keys."""
    return 2.0 * n * cfg.n_q_heads * cfg.head_dim * ((t0 - min(E, t0)) + (n + 1) / 2.0) * cfg.n_layers


def tensor_roofline(tflops, peaks, clocks):
    """Fractions of one achieved TFLOP/s figure against every denominator on record, and which measured peak the
    run's clocks call for: the burst figure when the SM clock stayed at (>= 95 % of) its maximum with no power cap
    active while the kernels ran, the sustained one otherwise."""
    sm, smax = clocks.get("sm_mhz"), clocks.get("sm_max_mhz")
    at_max = bool(sm and smax and sm >= 0.95 * smax and "sw_power_cap" not in clocks.get("reasons", []))
    peak = peaks["bf16_tflops"] if at_max else peaks["bf16_tflops_sustained"]
    return {"achieved": tflops, "peak": peak, "unit": "TFLOP/s", "frac": tflops / peak if tflops else None,
            "frac_burst": tflops / peaks["bf16_tflops"] if tflops else None,
            "frac_sustained": tflops / peaks["bf16_tflops_sustained"] if tflops else None,
            "frac_nominal": tflops / NOMINAL_BF16_TFLOPS if tflops else None,
            "of": f"{peaks['source']} ({'burst' if at_max else 'sustained'}: SM clock {sm} of {smax} MHz under load)"}


def needle_recall(lt, st, seq, cfg):
    """Share of the planted needle's tokens that the selection of the last call covers, per (layer, KV head):
    a property of the generator (reported, not a parity gate).  None when the needle is not fully indexed."""
    rng = st.needle_range()
    if rng is None:
        return None
    a, b = rng
    full, cover, units = 0, 0.0, 0
    for layer in range(cfg.n_layers):
        if lt.ltri_get_stats(seq, layer).evicted_end < b:
            return None
        spans = lt.ltri_get_spans(seq, layer)
        sel = lt.ltri_get_selected(seq, layer)
        for g in range(cfg.n_kv_heads):
            ids = sel[g][sel[g] >= 0]
            if cfg.unit_tokens > 0:   # the ids are unit numbers: tokens [id * U, (id + 1) * U)
                lo = np.maximum(ids * cfg.unit_tokens, a)
                hi = np.minimum((ids + 1) * cfg.unit_tokens, b)
            else:
                lo = np.maximum(spans[ids, 0], a)
                hi = np.minimum(spans[ids, 0] + spans[ids, 1], b)
            c = float(np.clip(hi - lo, 0, None).sum()) / (b - a)
            cover += c
            full += c >= 1.0
            units += 1
    return {"needle_tokens": [int(a), int(b)], "mean_coverage": cover / units, "fully_retrieved": full / units}


def params_of(cfg, nseq, binding):
    return binding.make_params(cfg.n_layers, cfg.n_q_heads, cfg.n_kv_heads, cfg.max_tokens, cfg.chunk, cfg.window,
                               cfg.n_sink, cfg.top_k, head_dim=cfg.head_dim, max_seqs=nseq,
                               reps_per_span=cfg.reps_per_span, max_spans_per_region=cfg.max_spans_per_region,
                               theta_mode=cfg.theta_mode, theta=cfg.theta, rep_mode=cfg.rep_mode,
                               ratio_kind=cfg.ratio_kind, min_reps=cfg.min_reps, max_reps=cfg.max_reps,
                               rep_lambda=cfg.rep_lambda,
                               flags=(binding.FLAG_PERSIST_DECODE if cfg.persist_decode else 0) |
                                     (binding.FLAG_COLLAB_VOTE if cfg.collab_vote else 0) |
                                     (binding.FLAG_SEGMENT_PER_UNIT if cfg.segment_per_unit else 0) |
                                     (binding.FLAG_HOST_KV if cfg.host_kv else 0),
                               cache_units=cfg.cache_units, score_decay=cfg.score_decay,
                               unit_tokens=cfg.unit_tokens, nms_iou_milli=cfg.nms_iou_milli,
                               retrieval_head=cfg.retrieval_head, retrieval_head_score=cfg.retrieval_head_score,
                               layer_theta=cfg.layer_theta, layer_nms_iou_milli=cfg.layer_nms_iou_milli,
                               layer_rep_lambda=cfg.layer_rep_lambda)


def measure(cfg, K, W, rank, local, world, dev, peaks, want_e2e=True, per_layer_calls=False):
    """Streams the workload of `cfg` up to its last W + K prefill calls, times those K calls (and the workload's decode
    steps) with the inputs resident in HBM and, if asked, once more through the host-buffer entry.  Returns a dict
    with everything the report lines are made of."""
    from paper_2412_04757_b200 import binding

    L, n = cfg.n_layers, cfg.chunk
    chunks = list(inputs.prefill_calls(cfg))
    if K + W > len(chunks):   # tiny workloads: fewer calls exist than were asked for
        W = min(W, max(0, len(chunks) // 2 - 1))
        K = len(chunks) - W
    first_timed = len(chunks) - K
    first_warm = first_timed - W

    NSEQ = cfg.n_seqs
    streams = [inputs.SyntheticStream(cfg, seq=rank * NSEQ + s, device=dev) for s in range(NSEQ)]
    st = streams[-1]        # the timed prefill steps run on the last sequence; the others are streamed as set-up
    SQ = NSEQ - 1
    p = params_of(cfg, NSEQ, binding)

    def stream_until(lt, upto, keep_from):
        for s in range(NSEQ - 1):
            for (t0, cnt) in chunks:
                q, k, v = streams[s].tokens(t0, cnt)
                lt.ltri_prefill_chunk(s, 0, L, q, k, v)
        kept = []
        for ci, (t0, cnt) in enumerate(chunks[:upto]):
            q, k, v = st.tokens(t0, cnt)
            if ci >= keep_from:
                kept.append((q, k, v))
            else:
                lt.ltri_prefill_chunk(SQ, 0, L, q, k, v)
        return kept

    def call(lt, qkv, out):
        q, k, v = qkv
        if not per_layer_calls:
            lt.ltri_prefill_chunk(SQ, 0, L, q, k, v, out=out)
        else:   # one layer per call, in order: what a model whose layers depend on each other has to do
            for l in range(L):
                lt.ltri_prefill_chunk(SQ, l, 1, q[l:l + 1], k[l:l + 1], v[l:l + 1], out=out[l:l + 1])

    lt = binding.Ltri(p, device=dev)
    # set-up: stream everything before the warm-up chunks, generate (and keep) warm-up + timed inputs
    kept = stream_until(lt, len(chunks), first_warm)
    outs = [torch.empty_like(kept[0][0]) for _ in range(2)]

    def decode_inputs(step):
        parts = [sx.tokens(cfg.context + step, 1, kind=1) for sx in streams]
        return tuple(torch.cat([pp[i].permute(1, 0, 2, 3) for pp in parts]).contiguous() for i in range(3))

    dec_in = [decode_inputs(s) for s in range(cfg.decode_steps)]
    seq_ids = list(range(NSEQ))
    torch.cuda.synchronize(dev)

    # ---- device-resident timing ------------------------------------------------------------
    # (the library's per-class CUDA events are on during the timed steps: they give kernel_ms_per_step and the
    # rooflines from the very launches that `value` is made of; they cost about 1 % and keep consecutive kernel
    # classes from overlapping their launches)
    for i in range(W):
        call(lt, kept[i], outs[i & 1])
    torch.cuda.synchronize(dev)
    lt.ltri_profile_read()                      # clears counters
    lt.ltri_profile_enable(True)
    miss_before_timed = sum(lt.ltri_debug_read(binding.BUF_CACHE_STATS, SQ, l) for l in range(L))[1] if cfg.host_kv else 0
    sampler = ClockSampler(local)
    sampler.start()
    launches0 = lt.ltri_launch_count()
    barrier(world)
    torch.cuda.synchronize(dev)
    clk_lo = sampler.mark()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record()
    for i in range(K):
        call(lt, kept[W + i], outs[i & 1])
    e1.record()
    torch.cuda.synchronize(dev)
    clk_hi = sampler.mark()
    barrier(world)
    ms = e0.elapsed_time(e1)
    launches = lt.ltri_launch_count() - launches0
    prof = lt.ltri_profile_read()
    lt.ltri_profile_enable(False)
    assert lt.ltri_sync_status() == 0, "device-side status word reports an error"
    stats = lt.ltri_get_stats(SQ, 0)
    # retrieved tokens of the last timed call, summed over KV heads and layers (the continuation kernel's work)
    retrieved_all = sum(lt.ltri_get_stats(SQ, l).retrieved_tokens for l in range(L))
    pager = None
    if cfg.host_kv:
        # unit-cache traffic of all layers since the stream began (prefill calls only so far)
        hm = sum(lt.ltri_debug_read(binding.BUF_CACHE_STATS, SQ, l) for l in range(L))
        unit_bytes = cfg.unit_tokens * cfg.head_dim * 2 * 2     # K and V rows of one unit
        pager = {"cache_units": cfg.cache_units, "score_decay": cfg.score_decay, "unit_hits": int(hm[0]),
                 "unit_misses": int(hm[1]), "hit_rate": float(hm[0] / max(1, hm[0] + hm[1])),
                 "host_to_device_bytes_per_call": float(hm[1]) * unit_bytes / max(1, len(chunks)),
                 "device_to_host_bytes_per_call": float(L * cfg.n_kv_heads * cfg.chunk * cfg.head_dim * 2 * 2),
                 "note": "prefill calls of the whole stream; the mirror gets every evicted row once",
                 "arena_bytes": int(lt.arena_bytes), "slab_slides": int(stats.slab_slides)}
        p_res = binding.LtriParams.from_buffer_copy(p)
        p_res.flags &= ~binding.FLAG_HOST_KV
        pager["resident_arena_bytes"] = int(binding.ltri_arena_bytes(p_res))
        # the pulls of the timed calls against the bus: bytes the top-k kernels asked for (misses of the timed calls,
        # taken from the counters) over the time the pull kernels were running, next to a plain pinned-memory copy
        miss_timed = float(hm[1]) - float(miss_before_timed)
        src = torch.empty(256 << 20, dtype=torch.uint8).pin_memory()
        dst = torch.empty_like(src, device=dev)
        best = None
        for _ in range(4):
            b0, b1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            b0.record()
            dst.copy_(src, non_blocking=True)
            b1.record()
            torch.cuda.synchronize(dev)
            best = min(best, b0.elapsed_time(b1)) if best else b0.elapsed_time(b1)
        bus = src.numel() / (best * 1e-3) / 1e9
        del src, dst
        pager["roofline"] = {"bound": "bus", "pulled_bytes": miss_timed * unit_bytes, "peak": bus, "unit": "GB/s",
                             "note": "host-to-device bytes of the timed calls' missing units over the run time of "
                                     "the pull kernels; peak = a 256 MiB copy from pinned memory on this box"}
    recall = {"final_chunk": needle_recall(lt, st, SQ, cfg)} if cfg.needle and rank == 0 else None
    ms = max_over_ranks(ms, world, dev)
    tokens = K * n
    prefill_tps = sum_over_ranks(tokens / (ms * 1e-3), world, dev) if world > 1 else tokens / (ms * 1e-3)

    # ---- decode (state is now at full context) ----------------------------------------------
    dec = None
    if cfg.decode_steps > 0:
        dout = torch.empty_like(dec_in[0][0])
        dw = min(3, cfg.decode_steps // 2)
        for s in range(dw):
            lt.ltri_decode_step(seq_ids, 0, L, *dec_in[s], out=dout)
        torch.cuda.synchronize(dev)
        # first half of the steps plain (tok/s), second half with the per-class events on (kernel times)
        half = dw + max(1, (cfg.decode_steps - dw) // 2)
        d0, d1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        barrier(world)
        d0.record()
        for s in range(dw, half):
            lt.ltri_decode_step(seq_ids, 0, L, *dec_in[s], out=dout)
        d1.record()
        torch.cuda.synchronize(dev)
        dms = max_over_ranks(d0.elapsed_time(d1), world, dev)
        lt.ltri_profile_read()
        lt.ltri_profile_enable(True)
        for s in range(half, cfg.decode_steps):
            lt.ltri_decode_step(seq_ids, 0, L, *dec_in[s], out=dout)
        torch.cuda.synchronize(dev)
        dprof = lt.ltri_profile_read()
        lt.ltri_profile_enable(False)
        psteps = max(1, cfg.decode_steps - half)
        dsteps = half - dw
        dst = lt.ltri_get_stats(SQ, 0)
        ret_tok = dst.retrieved_tokens / cfg.n_kv_heads
        keys = cfg.n_sink + ret_tok + (dst.tokens - dst.evicted_end)
        # algorithmic bytes per step: index scan + K and V rows once per KV head
        bytes_step = NSEQ * L * (cfg.n_kv_heads * dst.n_spans * cfg.head_dim * 2 +
                                 2 * cfg.n_kv_heads * cfg.head_dim * 2 * keys)
        k_ms = dprof["decode_retrieve"][0] + dprof["decode_attn"][0]
        gbs = bytes_step * psteps / (k_ms * 1e-3) / 1e9 if k_ms > 0 else None
        dec = {"value": world * NSEQ * dsteps / (dms * 1e-3), "unit": "tok/s", "steps": dsteps, "sequences": NSEQ,
               "ms_per_step": dms / dsteps,
               "keys_per_head": keys, "index_spans": dst.n_spans,
               "roofline": {"bound": "hbm", "achieved": gbs, "peak": peaks["hbm_gbs"], "unit": "GB/s",
                            "frac": gbs / peaks["hbm_gbs"] if gbs else None,
                            "frac_nominal": gbs / NOMINAL_HBM_GBS if gbs else None,
                            "frac_whole_step": bytes_step / (dms / dsteps * 1e-3) / 1e9 / peaks["hbm_gbs"],
                            "traffic": bytes_step * DECODE_DRAM_PER_ALGORITHMIC_BYTE,
                            "traffic_note": "bytes per step, scaled from an ncu capture of an 8-layer 64K case",
                            "kernels": "decode score+top-k and split-KV attention+merge",
                            "of": peaks["source"]},
               "kernel_ms_per_step": {k: v[0] / psteps for k, v in dprof.items() if v[1]}}
        if recall is not None:
            recall["last_decode_step"] = needle_recall(lt, st, SQ, cfg)
    clocks = sampler.stop(clk_lo, clk_hi)
    if pager is not None:
        pull_ms = prof["pager_pull"][0]
        gbs = pager["roofline"]["pulled_bytes"] / (pull_ms * 1e-3) / 1e9 if pull_ms > 0 else None
        pager["roofline"].update({"achieved": gbs, "frac": gbs / pager["roofline"]["peak"] if gbs else None})

    # ---- end-to-end: same steps with host buffers ---------------------------------------------
    e2e = None
    if want_e2e:
        lt.close()
        del lt
        torch.cuda.empty_cache()
        p_host = binding.LtriParams.from_buffer_copy(p)
        p_host.flags |= binding.FLAG_HOST_STAGING
        lt = binding.Ltri(p_host, device=dev)
        stream_until(lt, first_warm, len(chunks))
        host = [tuple(x.cpu().pin_memory() for x in kept[i]) for i in range(W + K)]
        h2d = sum(x.numel() * 2 for x in host[0])
        shape = kept[0][0].shape
        del kept
        # The library's host-buffer entry: q, k, v in pinned host memory, output back to pinned host memory.  It
        # carries a call out in layer groups (the layers are independent): a group's inputs go up on a copy stream
        # while the previous group computes and the one before sends its output down; two staging sets alternate
        # between calls.
        hout = [torch.empty(shape, dtype=torch.bfloat16).pin_memory() for _ in range(2)]
        d2h = hout[0].numel() * 2

        def step(i):
            lt.ltri_prefill_chunk_host(SQ, 0, L, host[i][0], host[i][1], host[i][2], hout[i & 1])

        torch.cuda.synchronize(dev)
        for i in range(W):
            step(i)
        lt.ltri_host_outputs_ready()
        torch.cuda.synchronize(dev)
        barrier(world)
        g0, g1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        t0 = time.perf_counter()
        g0.record()
        for i in range(K):
            step(W + i)
        lt.ltri_host_outputs_ready()                  # the stream now waits for the last output copy
        g1.record()
        torch.cuda.synchronize(dev)                   # every output of every timed step is in host memory
        wall = (time.perf_counter() - t0) * 1e3
        ems = max_over_ranks(max(g0.elapsed_time(g1), wall), world, dev)
        ngrp = min(4, L)
        assert lt.ltri_sync_status() == 0, "device-side status word reports an error"
        e2e = {"value": world * tokens / (ems * 1e-3), "unit": "tok/s", "h2d_bytes_per_step": h2d,
               "d2h_bytes_per_step": d2h, "ms_per_step": ems / K, "layer_groups": ngrp,
               "api": "ltri_prefill_chunk_host",
               "timing": "max of device events (first call -> last output copy done) and the host clock"}
    lt.close()
    del lt
    torch.cuda.empty_cache()

    # ---- rooflines of the dense kernels, live CUDA-event times ---------------------------------
    timed = chunks[first_timed:]
    E_of = lambda t0: max(cfg.n_sink, t0 - cfg.window - (t0 % cfg.chunk))
    f_loc = sum(attn_local_flops(cfg, t0, cnt, E_of(t0)) for (t0, cnt) in timed)
    f_map = sum(map_pass_flops(cfg, t0, cnt, E_of(t0)) for (t0, cnt) in timed)
    # continuation over the retrieved tokens: G query heads x n rows x R keys per (layer, KV head); R taken from
    # the last timed call and assumed for all of them
    G = cfg.n_q_heads // cfg.n_kv_heads
    f_ret = sum(4.0 * cnt * G * cfg.head_dim * retrieved_all for (_, cnt) in timed)
    a_ms, a_cnt = prof["attn_local"]
    r_ms, _ = prof["attn_retrieved"]
    per_layer = ATTN_LOCAL_DRAM_BYTES_PER_LAYER.get((cfg.n_q_heads, cfg.n_kv_heads, cfg.chunk, cfg.window, cfg.n_sink))
    window_full = timed[0][0] >= cfg.window + cfg.chunk
    traffic = per_layer * L / max(1, a_cnt // K) if per_layer and window_full else None
    roof = {"bound": "tensor",
            **tensor_roofline(f_loc / (a_ms * 1e-3) / 1e12 if a_ms > 0 else None, peaks, clocks),
            "traffic": traffic,
            "traffic_note": "DRAM bytes per launch, ncu capture of a 4-layer case of the same geometry x layers / 4",
            "kernel": "k_attn_tc, local part (sink | local | current)",
            "launches": a_cnt, "ms_per_launch": a_ms / max(a_cnt, 1),
            "timing": "CUDA events of the library around the launch"}
    roof_attn = {"bound": "tensor",
                 **tensor_roofline((f_loc + f_ret) / ((a_ms + r_ms) * 1e-3) / 1e12 if a_ms > 0 else None, peaks, clocks),
                 "kernels": "k_attn_tc local part + continuation over the retrieved spans (the chunked-prefill "
                            "attention as a whole)",
                 "ms_per_step": (a_ms + r_ms) / K, "flops_per_step": (f_loc + f_ret) / K}
    roof_call = {"bound": "tensor",
                 **tensor_roofline((f_loc + f_ret + f_map) / (ms * 1e-3) / 1e12, peaks, clocks),
                 "kernels": "all dense work of a call (attention, continuation, local-map pass) over the whole step time",
                 "flops_per_step": (f_loc + f_ret + f_map) / K}
    return {"cfg": cfg, "K": K, "W": W, "ms": ms, "value": prefill_tps, "launches": launches, "prof": prof,
            "stats": stats, "retrieved_per_kv_head": retrieved_all / (L * cfg.n_kv_heads), "pager": pager,
            "recall": recall, "decode": dec, "clocks": clocks, "e2e": e2e, "roofline": roof,
            "roofline_prefill_attention": roof_attn, "roofline_call": roof_call,
            "timed_positions": [timed[0][0], cfg.context], "nseq": NSEQ,
            "kernel_ms_per_step": {k: v[0] / K for k, v in prof.items() if v[1]}}


def brief(m):
    """The short form of a measurement, for the extra workloads reported beside the headline."""
    d = m["decode"]
    out = {"workload": m["cfg"].name, "prefill_tok_s": m["value"], "ms_per_step": m["ms"] / m["K"], "steps": m["K"],
           "frac_attn_local": m["roofline"]["frac"], "frac_prefill_attention": m["roofline_prefill_attention"]["frac"],
           "peak_tflops": m["roofline"]["peak"], "index_spans": m["stats"].n_spans,
           "retrieved_tokens_per_kv_head": m["retrieved_per_kv_head"], "gpu_launches": m["launches"],
           "kernel_ms_per_step": m["kernel_ms_per_step"]}
    if d:
        out.update({"decode_tok_s": d["value"], "decode_ms_per_step": d["ms_per_step"],
                    "decode_frac_hbm": d["roofline"]["frac"]})
    if m["recall"]:
        out["needle_recall"] = m["recall"]
    if m["pager"]:
        out["pager"] = m["pager"]
    return out


def paper_setting(cfg):
    """The paper's own setting of the optional modes on the same workload: 128-token memory units (Eq. 8 as
    printed), dynamic representative counts with the row ratio and lambda = 3 (Sec. 3.3.2), NMS threshold 0.1
    (App. "NMS Input Filtration"), persistent mechanism in decode (Sec. 3.5)."""
    import dataclasses
    c = dataclasses.replace(cfg, unit_tokens=128, rep_mode=1, ratio_kind=0, rep_lambda=3.0, min_reps=1, max_reps=4,
                            nms_iou_milli=100, persist_decode=True)
    c.name += "[paper-setting: unit=128,dynamic-reps,nms-iou=0.1,persist-decode]"
    return c


def run_ltri(args, cfg):
    from paper_2412_04757_b200 import build

    if not torch.cuda.is_available():
        raise SystemExit("bench.py needs a CUDA device: the path has no CPU fallback")
    rank, local, world = dist_setup(args.gpus)
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    build.build()
    peaks = measured_peaks()
    m = measure(cfg, args.steps, args.warmup, rank, local, world, dev, peaks, want_e2e=not args.no_e2e)
    extras = {}
    if args.extras and world == 1:
        # beside the headline: the same workload in the paper's own setting, the other single-GPU workloads, and
        # the headline workload submitted one layer per call; few steps each, no host-buffer leg
        ks, ws = min(8, args.steps), min(3, args.warmup)
        extras["paper_setting"] = brief(measure(paper_setting(cfg), ks, ws, rank, local, world, dev, peaks, False))
        if args.config == 2 and cfg.name == inputs.config(2).name:
            extras["other_configs"] = [brief(measure(inputs.config(c), ks, ws, rank, local, world, dev, peaks, False))
                                       for c in (1, 3, 4)]
        pl = measure(cfg, ks, ws, rank, local, world, dev, peaks, False, per_layer_calls=True)
        extras["per_layer_calls"] = {**brief(pl), "note": "every layer of a chunk submitted as its own call "
                                                          "(layer_count = 1), as a model with dependent layers must"}
    if rank != 0:
        return
    cpu = None
    if not args.no_cpu_baseline:
        ctoks, cores, sample, _ = oracle_sample(cfg, 2, 0)
        cpu = {"value": ctoks, "unit": "tok/s", "cores": cores, "kind": "oracle", "sample": sample}
    K = m["K"]
    line = {
        "metric": METRIC, "value": m["value"], "unit": "tok/s", "n_gpus": world, "steps": K, "warmup": m["W"],
        "ms_per_step": m["ms"] / K, "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "bf16",
        "data": "synthetic",
        "config": {**workload_config(cfg, world, m["nseq"]), "timed_positions": m["timed_positions"],
                   "l2": "inputs of every step are distinct and larger than L2 (no flush needed)",
                   "index_spans": m["stats"].n_spans, "retrieved_tokens_per_kv_head": m["retrieved_per_kv_head"]},
        "clocks": m["clocks"], "gpu_launches": m["launches"], "e2e": m["e2e"], "decode": m["decode"],
        "roofline": m["roofline"], "roofline_prefill_attention": m["roofline_prefill_attention"],
        "roofline_call": m["roofline_call"], "cpu_baseline": cpu,
        "needle_recall": m["recall"], "pager": m["pager"], "kernel_ms_per_step": m["kernel_ms_per_step"],
        **extras,
    }
    print(json.dumps(line))


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=32)
    ap.add_argument("--warmup", type=int, default=4)
    ap.add_argument("--config", type=int, default=2, help="workload index 0..4 (2 = 128K needle, the headline)")
    ap.add_argument("--impl", default="ltri", choices=["ltri", "reference"])
    ap.add_argument("--layers", type=int, default=0, help="override the layer count (profiling of small cases)")
    ap.add_argument("--context", type=int, default=0, help="override the context length (profiling of small cases)")
    ap.add_argument("--decode-steps", type=int, default=-1, help="override the number of decode steps")
    ap.add_argument("--dynamic-reps", action="store_true",
                    help="dynamic span index vectors (rep_mode 1; row ratio and lambda 3 as in the paper's "
                         "implementation details, 1..4 per span)")
    ap.add_argument("--unit-tokens", type=int, default=0,
                    help="retrieval granularity: fixed units of this many tokens instead of spans (the paper's 128)")
    ap.add_argument("--nms-iou", type=float, default=0.0,
                    help="IoU threshold of the segmenter's NMS (0: spans never overlap; the paper lists 0.1 / 0.01)")
    ap.add_argument("--persist-decode", action="store_true",
                    help="decode keeps the spans selected by the last prefill call (persistent mechanism)")
    ap.add_argument("--host-kv", type=int, default=0, metavar="CACHE_UNITS",
                    help="host-memory pager: mirror evicted rows in pinned host memory and read retrieved units from a "
                         "device cache of this many units per (layer, KV head) (the paper's 32); needs --unit-tokens. "
                         "The mirror takes 2 x layers x KV heads x context x 256 bytes of pinned memory")
    ap.add_argument("--segment-per-unit", action="store_true",
                    help="segment every memory unit on its own, four spans kept per unit (the paper's 'Span' column); "
                         "needs --unit-tokens")
    ap.add_argument("--layer-tables", action="store_true",
                    help="per-layer theta (quantile levels spread over 0.88..0.95), phi (0.1 / 0.01 alternating) and "
                         "lambda (20 for the first four layers, 3 after them, as in the paper's implementation "
                         "details); the theta and phi values are made up within the paper's ranges")
    ap.add_argument("--retrieval-heads", action="store_true",
                    help="give 14 of every 32 layers a retrieval head (a made-up table: which heads these are belongs "
                         "to a trained model); such a layer locates evidence with that head alone")
    ap.add_argument("--collab-vote", action="store_true",
                    help="collaborative voting over the layers' ballots (needs --retrieval-heads and --unit-tokens)")
    ap.add_argument("--p-self", type=float, default=-1.0,
                    help="generator: probability that a prefill token targets its own segment (default 0.5; 0 = the "
                         "literal 'earlier segment' reading)")
    ap.add_argument("--no-e2e", action="store_true")
    ap.add_argument("--extras", dest="extras", action="store_true", default=None,
                    help="also measure the paper's own setting, the other single-GPU workloads and per-layer calls "
                         "(default: on for the plain default run, off when any workload option is given)")
    ap.add_argument("--no-extras", dest="extras", action="store_false")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    args = ap.parse_args()
    if args.extras is None:
        workload_flags = ("--layers", "--context", "--decode-steps", "--dynamic-reps", "--unit-tokens", "--nms-iou",
                          "--persist-decode", "--host-kv", "--segment-per-unit", "--layer-tables", "--retrieval-heads",
                          "--collab-vote", "--p-self", "--config", "--no-e2e", "--no-cpu-baseline")
        args.extras = not any(a.split("=")[0] in workload_flags for a in sys.argv[1:])
    cfg = inputs.config(args.config)
    if args.layers > 0 or args.context > 0 or args.decode_steps >= 0:
        import dataclasses
        cfg = dataclasses.replace(cfg, n_layers=args.layers or cfg.n_layers, context=args.context or cfg.context,
                                  decode_steps=cfg.decode_steps if args.decode_steps < 0 else args.decode_steps)
        cfg.name += f"[layers={cfg.n_layers},context={cfg.context},decode={cfg.decode_steps}]"
    if args.dynamic_reps:
        import dataclasses
        cfg = dataclasses.replace(cfg, rep_mode=1, ratio_kind=0, rep_lambda=3.0, min_reps=1, max_reps=4)
        cfg.name += "[dynamic-reps]"
    if args.p_self >= 0:
        import dataclasses
        cfg = dataclasses.replace(cfg, p_self=args.p_self)
        cfg.name += f"[p_self={args.p_self:g}]"
    if args.unit_tokens > 0:
        import dataclasses
        cfg = dataclasses.replace(cfg, unit_tokens=args.unit_tokens)
        cfg.name += f"[unit={args.unit_tokens}]"
    if args.nms_iou > 0:
        import dataclasses
        cfg = dataclasses.replace(cfg, nms_iou_milli=int(round(args.nms_iou * 1000)))
        cfg.name += f"[nms-iou={args.nms_iou:g}]"
    if args.persist_decode:
        import dataclasses
        cfg = dataclasses.replace(cfg, persist_decode=True)
        cfg.name += "[persist-decode]"
    if args.host_kv > 0:
        import dataclasses
        if args.unit_tokens <= 0:
            ap.error("--host-kv needs --unit-tokens")
        cfg = dataclasses.replace(cfg, host_kv=True, cache_units=args.host_kv, score_decay=0.1)
        cfg.name += f"[host-kv,cache={args.host_kv}]"
    if args.segment_per_unit:
        import dataclasses
        if args.unit_tokens <= 0:
            ap.error("--segment-per-unit needs --unit-tokens")
        cfg = dataclasses.replace(cfg, segment_per_unit=True, max_spans_per_region=4)
        cfg.name += "[segment-per-unit]"
    if args.layer_tables:
        import dataclasses
        L = cfg.n_layers
        cfg = dataclasses.replace(
            cfg, layer_theta=tuple(0.88 + 0.07 * ((l * 13) % 8) / 7 for l in range(L)),
            layer_nms_iou_milli=tuple(100 if l % 2 == 0 else 10 for l in range(L)),
            layer_rep_lambda=tuple(20.0 if l < 4 else 3.0 for l in range(L)))
        cfg.name += "[layer-tables]"
    if args.retrieval_heads:
        import dataclasses
        has = [(l * 7) % 16 < 7 for l in range(cfg.n_layers)]
        cfg = dataclasses.replace(
            cfg, retrieval_head=tuple((l * 5 + 3) % cfg.n_q_heads if has[l] else -1 for l in range(cfg.n_layers)),
            retrieval_head_score=tuple(0.1 + 0.4 * ((l * 37) % 17) / 16 if has[l] else 0.0 for l in range(cfg.n_layers)),
            collab_vote=args.collab_vote)
        cfg.name += "[retrieval-heads" + (",vote]" if args.collab_vote else "]")
    elif args.collab_vote:
        ap.error("--collab-vote needs --retrieval-heads and --unit-tokens")
    if args.impl == "reference":
        run_reference(args, cfg)
    else:
        run_ltri(args, cfg)


if __name__ == "__main__":
    main()
