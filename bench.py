#!/usr/bin/env python
"""Benchmark of the BAPS fused attention forward on B200.

    python bench.py [--gpus N] [--steps K] [--warmup W] [--workload NAME] [--impl reference]

A step is one pass of the whole hot path (one ``baps_attention_fwd`` call) over one batch of
seeded synthetic input.  The default workload is the largest single-GPU configuration, the
long-context prefill (B=1, H=32, Hkv=8, S=32768, D=128, causal); the other attention configurations
and the standalone sweep are reported under ``extra``.  Rank 0 prints ONE JSON line.  With N > 1 (launched
through ``torch.distributed.run``) every rank runs an independent replica of the workload on
its own GPU -- the path has no exchange step -- and the value is the sum over ranks divided by
the slowest rank's time.

``--impl reference`` times the CPU checker (``oracle/``) on the host cores, on a bounded sample
of the same workload.
"""
from __future__ import annotations

import argparse
import json
import os
import sys
import threading
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

import numpy as np
import torch

from paper_2602_02071_b200 import replicas, workloads

METRIC = "BAPS attention fwd TFLOP/s"
UNIT = "TFLOP/s"
DEFAULT_WORKLOAD = "c5_long_context"
NOMINAL_DENSE_BF16_TFLOPS = 2250.0      # vendor figure for dense bf16 on one B200, for context
FALLBACK_PEAKS = {"hbm_gbs": 6650.0, "bf16_tflops": 1590.0, "bf16_tflops_sustained": 1400.0}

# From the committed ncu captures (profiles/): DRAM bytes read + written by one launch of the fused
# kernel, and the fraction of cycles its tensor pipe was active (a clock-independent counter).
# None where no capture of that workload exists.
NCU_CAPTURES = {
    # profiles/paired_attention_tc_kernel_c5_long_context_dram.txt: one launch of the full workload
    # (405.4 MB read + 235.5 MB written, 52.7 % of cycles)
    "c5_long_context": {"traffic": 640.9e6, "tensor_pipe_active_pct": 52.7},
    # profiles/paired_attention_tc_kernel_c2_llm_prefill_mha.txt: 143.3 MB read + 13.7 MB written
    "c2_llm_prefill_mha": {"traffic": 157.0e6, "tensor_pipe_active_pct": 43.3},
}

# Thread instructions per score element of the fused kernels, from smsp__inst_executed.sum of the committed
# captures (profiles/paired_attention_tc_kernel_long_causal_s16384.txt: 9.24; configuration 2 with its outlier keys
# 9.64; profiles/attention_d64_kernel_vit_b8_s1024.txt: 11.13), and the issue peak of the part: 148 SMs x 4 schedulers x
# 32 lanes per clock.
INSTR_PER_SCORE = {128: 9.2, 64: 11.1}
ISSUE_LANES_PER_CLOCK = 148 * 4 * 32


def issue_roofline(w, ms, sm_mhz):
    """The same launch against the instruction-issue peak (what bounds the kernel where the tensor core
    idles: D = 64, and the softmax side of every configuration).  Context beside the tensor roofline."""
    scores = w.B * w.H * (w.S * (w.S + 128) // 2 if w.causal else w.S * w.S)   # causal: whole diagonal tiles
    ipe = INSTR_PER_SCORE.get(w.D)
    if not ipe or not sm_mhz:
        return None
    achieved = scores * ipe / (ms * 1e-3)
    peak = ISSUE_LANES_PER_CLOCK * sm_mhz * 1e6
    return {"bound": "alu", "achieved": achieved / 1e12, "peak": peak / 1e12, "unit": "T thread-instructions/s",
            "frac": achieved / peak, "instr_per_score_ncu": ipe,
            "peak_kind": "148 SMs x 128 lanes x the SM clock sampled during the run"}


def load_peaks():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(path):
        with open(path) as f:
            return json.load(f), "measured"
    return dict(FALLBACK_PEAKS), "fallback"


class ClockSampler:
    """Samples SM clock and throttle reasons through NVML while the timed region runs."""

    def __init__(self, index: int, period_s: float = 0.002):
        self.samples, self.reasons, self.max_mhz = [], set(), None
        self._stop = threading.Event()
        self._thread = None
        self.period = period_s
        try:
            import pynvml
            pynvml.nvmlInit()
            self.nv = pynvml
            self.h = pynvml.nvmlDeviceGetHandleByIndex(index)
            self.max_mhz = int(pynvml.nvmlDeviceGetMaxClockInfo(self.h, pynvml.NVML_CLOCK_SM))
        except Exception:
            self.nv = None

    def _loop(self):
        nv = self.nv
        names = {
            "hw_slowdown": getattr(nv, "nvmlClocksThrottleReasonHwSlowdown", 0x8),
            "hw_thermal_slowdown": getattr(nv, "nvmlClocksThrottleReasonHwThermalSlowdown", 0x40),
            "sw_thermal_slowdown": getattr(nv, "nvmlClocksThrottleReasonSwThermalSlowdown", 0x20),
            "sw_power_cap": getattr(nv, "nvmlClocksThrottleReasonSwPowerCap", 0x4),
        }
        while not self._stop.is_set():
            try:
                self.samples.append(int(nv.nvmlDeviceGetClockInfo(self.h, nv.NVML_CLOCK_SM)))
                r = int(nv.nvmlDeviceGetCurrentClocksThrottleReasons(self.h))
                for k, bit in names.items():
                    if r & bit:
                        self.reasons.add(k)
            except Exception:
                pass
            time.sleep(self.period)

    def __enter__(self):
        if self.nv is not None:
            self._thread = threading.Thread(target=self._loop, daemon=True)
            self._thread.start()
        return self

    def __exit__(self, *a):
        self._stop.set()
        if self._thread is not None:
            self._thread.join()

    def summary(self):
        med = float(np.median(self.samples)) if self.samples else None
        return {"sm_mhz": med, "sm_max_mhz": self.max_mhz, "reasons": sorted(self.reasons),
                "samples": len(self.samples)}


def dist_info():
    return replicas.dist_env()


def oracle_sample_time(w, q, k, v, tiles):
    """Seconds the CPU checker needs for the given query tiles, and the flops they stand for."""
    import oracle
    qf, kf, vf = (t.float().numpy() for t in (q, k, v))
    oracle.attention(qf, kf, vf, causal=w.causal, block_q=w.block_q, block_k=w.block_k,
                     tiles=np.array(tiles[:1], dtype=np.int32))        # warm (builds tables)
    t0 = time.perf_counter()
    oracle.attention(qf, kf, vf, causal=w.causal, block_q=w.block_q, block_k=w.block_k,
                     tiles=np.array(tiles, dtype=np.int32))
    dt = time.perf_counter() - t0
    flops = 0.0
    for (_, _, i) in tiles:
        nkeys = (i + 1) * w.block_q if w.causal else w.S
        # causal tiles: the diagonal tile is counted as half
        if w.causal:
            nkeys = i * w.block_q + w.block_q / 2.0
        flops += 4.0 * w.block_q * nkeys * w.D
    return dt, flops, oracle.num_threads()


def bounded_sample_tiles(w, target_flops=2.5e10):
    """An evenly strided subset of all query tiles (every batch, head and position class is hit)
    whose total work is about target_flops; all tiles if the workload is smaller than that."""
    nq = w.S // w.block_q
    allt = [(b, h, i) for b in range(w.B) for h in range(w.H) for i in range(nq)]
    if w.flops <= target_flops:
        return allt
    n = max(1, int(round(len(allt) * target_flops / w.flops)))
    # a stride co-prime with the tile count per head so that positions are covered evenly
    step = max(1, len(allt) // n)
    while step > 1 and (nq % step == 0 or step % nq == 0):
        step -= 1
    return allt[::step][:max(n, 1)] if step > 1 else allt[:n]


def error_sample_tiles(w, n_min=24, seed=2):
    """Query tiles on which the GPU result is compared with the checker inside the benchmark: first,
    second, middle and last tile spread over one query head of every kv group and every batch, plus
    random ones, at least n_min in total (all tiles if the workload has fewer)."""
    nq = w.S // w.block_q
    if w.n_query_tiles <= n_min:
        return [(b, h, i) for b in range(w.B) for h in range(w.H) for i in range(nq)]
    gsz = w.H // w.Hkv
    picks = [0, min(1, nq - 1), nq // 2, nq - 1]
    out = set()
    for b in range(w.B):
        for g in range(w.Hkv):
            h = g * gsz + (g % gsz)
            out.add((b, h, picks[(2 * g) % 4])); out.add((b, h, picks[(2 * g + 1) % 4]))
    gen = torch.Generator().manual_seed(seed)
    while len(out) < n_min:
        out.add((int(torch.randint(0, w.B, (1,), generator=gen)), int(torch.randint(0, w.H, (1,), generator=gen)),
                 int(torch.randint(0, nq, (1,), generator=gen))))
    return sorted(out)


def run_reference(args):
    """Reference arm: the CPU checker, as it stands, on the host cores."""
    rank, world, _ = dist_info()
    if rank != 0:
        return 0
    w = workloads.WORKLOADS[args.workload]
    q, k, v = workloads.make_qkv(w)
    tiles = bounded_sample_tiles(w, target_flops=2.0e10)
    times, flops, cores = [], 0.0, 1
    for s in range(args.warmup + args.steps):
        dt, flops, cores = oracle_sample_time(w, q, k, v, tiles)
        if s >= args.warmup:
            times.append(dt)
    mean = float(np.mean(times))
    value = flops / mean / 1e12
    sample = f"{len(tiles)} of {w.n_query_tiles} query tiles per step (spread over heads and positions)"
    line = {
        "impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": args.gpus,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": mean * 1e3, "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "config": {"workload": w.name, "B": w.B, "H": w.H, "Hkv": w.Hkv, "S": w.S, "D": w.D,
                   "causal": w.causal, "block": [w.block_q, w.block_k]},
        "cpu_baseline": {"value": value, "unit": UNIT, "cores": cores, "kind": "oracle", "sample": sample},
        "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
        "gpu_launches": 0,
    }
    print(json.dumps(line), flush=True)
    return 0


def time_attention(w, q, k, v, steps, warmup, flush_buf):
    """Device-resident timing: per-step CUDA events around the call, L2 flushed between steps."""
    from paper_2602_02071_b200 import binding
    out = torch.empty_like(q)
    evs = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True))
           for _ in range(steps)]
    for _ in range(warmup):
        flush_buf.zero_()
        binding.baps_attention_fwd(q, k, v, causal=w.causal, block_q=w.block_q, block_k=w.block_k, out=out)
    torch.cuda.synchronize()
    n0 = binding.launch_count()
    for s in range(steps):
        flush_buf.zero_()
        evs[s][0].record()
        binding.baps_attention_fwd(q, k, v, causal=w.causal, block_q=w.block_q, block_k=w.block_k, out=out)
        evs[s][1].record()
    torch.cuda.synchronize()
    launches = binding.launch_count() - n0
    binding.poll_async_error()
    return [a.elapsed_time(b) for a, b in evs], launches


def time_e2e(w, qh, kh, vh, steps, warmup):
    """End to end through the public call with HOST buffers: every step copies q, k, v from pinned
    host memory to the device, runs the kernel and copies the output back to pinned host memory,
    all inside the timed region.  The steps are double-buffered over three streams (copy in,
    compute, copy out) as a serving loop would do it, so the copy of step i + 1 overlaps the kernel
    and the read-back of step i; the time is that of the whole sequence of `steps` steps."""
    from paper_2602_02071_b200 import binding
    dev = torch.device("cuda", torch.cuda.current_device())
    s_in, s_k, s_out = torch.cuda.Stream(dev), torch.cuda.Stream(dev), torch.cuda.Stream(dev)
    bufs = []
    for _ in range(2):
        bufs.append(dict(q=torch.empty(qh.shape, dtype=qh.dtype, device=dev),
                         k=torch.empty(kh.shape, dtype=kh.dtype, device=dev),
                         v=torch.empty(vh.shape, dtype=vh.dtype, device=dev),
                         o=torch.empty(qh.shape, dtype=qh.dtype, device=dev),
                         oh=torch.empty(qh.shape, dtype=qh.dtype).pin_memory(),
                         ev_in=torch.cuda.Event(), ev_k=torch.cuda.Event(), ev_out=torch.cuda.Event()))

    def run(nsteps):
        for s in range(nsteps):
            b = bufs[s % 2]
            with torch.cuda.stream(s_in):
                s_in.wait_event(b["ev_k"])            # the kernel that last read these inputs is done
                b["q"].copy_(qh, non_blocking=True); b["k"].copy_(kh, non_blocking=True); b["v"].copy_(vh, non_blocking=True)
                b["ev_in"].record(s_in)
            with torch.cuda.stream(s_k):
                s_k.wait_event(b["ev_in"])
                s_k.wait_event(b["ev_out"])           # the read-back of this output buffer is done
                binding.baps_attention_fwd(b["q"], b["k"], b["v"], causal=w.causal, block_q=w.block_q,
                                           block_k=w.block_k, out=b["o"])
                b["ev_k"].record(s_k)
            with torch.cuda.stream(s_out):
                s_out.wait_event(b["ev_k"])
                b["oh"].copy_(b["o"], non_blocking=True)
                b["ev_out"].record(s_out)

    run(max(warmup, 2))
    torch.cuda.synchronize()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record(s_in)
    run(steps)
    e1.record(s_out)                                  # after the last read-back
    torch.cuda.synchronize()
    total_ms = e0.elapsed_time(e1)
    binding.poll_async_error()
    h2d = sum(t.numel() * t.element_size() for t in (qh, kh, vh))
    d2h = bufs[0]["oh"].numel() * bufs[0]["oh"].element_size()
    return [total_ms / steps] * steps, h2d, d2h


def extra_measurements(peaks, flush_buf, skip, steps=10, warmup=3):
    """Supplementary numbers (not the headline): the other attention configurations and the
    standalone encode / row-softmax sweep, device resident."""
    from paper_2602_02071_b200 import binding
    extra = {}
    for name in ("c2_llm_prefill_mha", "c3_llm_prefill_gqa", "c4_vit_encoder", "c5_long_context"):
        if name == skip:
            continue
        w = workloads.WORKLOADS[name]
        q, k, v = workloads.make_qkv(w, device="cuda")
        with ClockSampler(torch.cuda.current_device()) as cs:
            ts, _ = time_attention(w, q, k, v, max(steps, 20 if w.flops < 1e12 else steps), warmup, flush_buf)
        ms = float(np.mean(ts))
        tf = w.flops / (ms * 1e-3) / 1e12
        clk = cs.summary()
        extra[name] = {"ms": ms, "best_ms": float(np.min(ts)), "tflops": tf,
                       "frac_of_bf16_burst": tf / peaks["bf16_tflops"],
                       "frac_of_bf16_sustained": tf / peaks.get("bf16_tflops_sustained", peaks["bf16_tflops"]),
                       "frac_of_nominal_dense_bf16": tf / NOMINAL_DENSE_BF16_TFLOPS,
                       "ms_x_sm_mhz": ms * clk["sm_mhz"] if clk["sm_mhz"] else None, "clocks": clk,
                       "issue_roofline": issue_roofline(w, ms, clk["sm_mhz"])}
        cap = NCU_CAPTURES.get(name)
        if cap:
            extra[name]["ncu"] = cap
        if w.causal:
            extra[name]["restart_rates_lambda_1"] = restart_rates_both_b0(w, q, k, v)
        if w.D == 128 and name != "c5_long_context":
            extra[name]["fp8_qk"] = fp8_study(w, q, k, v, flush_buf)
        del q, k, v
    sweep = {}
    n = 1 << 28
    g = torch.Generator(device="cuda"); g.manual_seed(0)
    x = torch.randn(n, device="cuda", generator=g) * 2.0
    codes = torch.empty(n, dtype=torch.uint8, device="cuda")
    probs = torch.empty(n, dtype=torch.float32, device="cuda")

    def timeit(fn):
        for _ in range(warmup):
            fn()
        torch.cuda.synchronize()
        ts = []
        for _ in range(steps):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record(); fn(); b.record(); torch.cuda.synchronize()
            ts.append(a.elapsed_time(b))
        return float(np.median(ts))

    ms = timeit(lambda: binding.baps_hif8_encode(x, codes))
    sweep["encode"] = {"ms": ms, "gbs": 5.0 * n / (ms * 1e-3) / 1e9}
    ms = timeit(lambda: binding.baps_hif8_decode(codes, probs))
    sweep["decode"] = {"ms": ms, "gbs": 5.0 * n / (ms * 1e-3) / 1e9}
    codes2 = torch.empty_like(codes)
    ms = timeit(lambda: binding.baps_exp2_hif8(codes, codes2))
    sweep["exp2_map"] = {"ms": ms, "gbs": 2.0 * n / (ms * 1e-3) / 1e9}
    del codes2
    for cols in (1024, 2048, 4096, 8192, 16384, 32768, 65536):
        xr = x.view(n // cols, cols)
        pr = probs.view(n // cols, cols)
        ms = timeit(lambda: binding.baps_softmax_rows(xr, 128, pr))
        sweep[f"softmax_rows_{cols}"] = {"ms": ms, "gbs": 8.0 * n / (ms * 1e-3) / 1e9}
    for cols in (1024, 8192, 65536):
        xr = x.view(n // cols, cols)
        ms = timeit(lambda: binding.baps_softmax_rows_codes(xr, 128))
        sweep[f"softmax_rows_codes_{cols}"] = {"ms": ms, "gbs": 5.0 * n / (ms * 1e-3) / 1e9}
    for v_ in sweep.values():
        v_["frac_of_hbm"] = v_["gbs"] / peaks["hbm_gbs"]
    extra["sweep_2p28_fp32"] = sweep
    return extra


def restart_rates_both_b0(w, q, k, v, lam=1):
    """ARR / PRR of Table 4 from the per-query-tile restart counters, for B0 = {first} and for
    B0 = {first, last visible tile}; 8-bit tiles per query tile = visible key tiles minus |B0|."""
    from paper_2602_02071_b200 import binding
    nq = w.S // 128
    vis = (torch.arange(nq) + 1) if w.causal else torch.full((nq,), nq)
    out = {}
    for key, b0_last in (("b0_first", False), ("b0_first_last", True)):
        st = binding.baps_attention_fwd_ex(q, k, v, causal=w.causal, block_q=128, block_k=128, lam=lam, b0_last=b0_last)
        cnt = st.restarts.cpu().to(torch.float64)                       # [B, H, nq]
        t8 = (vis - torch.clamp(vis, max=2 if b0_last else 1)).to(torch.float64)
        ratio = torch.where(t8 > 0, cnt / torch.clamp(t8, min=1), torch.zeros_like(cnt))
        out[key] = {"ARR": float(cnt.sum() / (t8.sum() * w.B * w.H)), "PRR": float(ratio.max())}
        del st
    return out


def fp8_study(w, q, k, v, flush_buf, steps=10):
    """Quantised-input variant: Q and K as E4M3 with one power-of-two scale per 128-row tile (quantised here,
    on the device, from the bf16 inputs).  Reports its rate and how far its output is from the bf16
    path's on the same inputs (the price of the quantisation; parity with the checker is a test)."""
    from paper_2602_02071_b200 import binding
    q8, qs, _ = workloads.quantize_e4m3_tiles(q)
    k8, ks, _ = workloads.quantize_e4m3_tiles(k)
    out = torch.empty_like(q)
    fn = lambda: binding.baps_attention_fwd_fp8(q8, k8, v, qs, ks, causal=w.causal, want_stats=False, out=out)
    for _ in range(3):
        fn()
    torch.cuda.synchronize()
    ts = []
    for _ in range(steps):
        flush_buf.zero_()
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record(); fn(); b.record(); torch.cuda.synchronize(); ts.append(a.elapsed_time(b))
    ref = binding.baps_attention_fwd(q, k, v, causal=w.causal)
    diff = (out.float() - ref.float()).abs()
    ms = float(np.mean(ts))
    return {"ms": ms, "tflops": w.flops / (ms * 1e-3) / 1e12,
            "vs_bf16_path": {"max_abs": float(diff.max()), "mean_abs": float(diff.mean())}}


def fig2_experiment(lengths=(1024, 2048, 4096, 8192, 16384, 32768), heads=2):
    """Section 3.3 / Fig. 2: error that accumulates in the rescale factors.  On inputs whose row
    maximum rises a little with every key tile (workloads.make_rising_max_qkv) the real-valued running
    max of the "Exp2 HiF8" setup moves at every tile and each move multiplies the accumulators by an
    8-bit, non-integer power of two, while Algorithm 1's integer max moves once in twenty tiles and
    its factors are exact.  Reported per sequence length: number of max updates, and the error of
    both setups against Eq. (1) (double precision, from the checker) on the first query tile of every
    head -- for the CUDA kernels and, as a cross-check, for the checker's own versions of the setups."""
    import oracle
    from paper_2602_02071_b200 import binding
    out = {}
    for S in lengths:
        q, k, v = workloads.make_rising_max_qkv(S, H=heads)
        qd, kd, vd = q.cuda(), k.cuda(), v.cuda()
        qf, kf, vf = (t.float().numpy() for t in (q, k, v))
        tiles = np.array([(0, h, 0) for h in range(heads)], dtype=np.int32)
        kw = dict(causal=False, block_q=128, block_k=128, tiles=tiles)
        ex = oracle.attention(qf, kf, vf, mode=oracle.MODE_EXACT, **kw)
        row = {"max_updates_real_valued": S // 128 - 1}
        for key, gmode, omode in (("e2e_hif8", binding.MODE_E2E_HIF8, oracle.MODE_E2E_HIF8),
                                  ("exp2_hif8", binding.MODE_EXP2_HIF8, oracle.MODE_EXP2_HIF8)):
            st = binding.baps_attention_fwd_ex(qd, kd, vd, causal=False, block_q=128, block_k=128, mode=gmode)
            got = np.stack([st.out_f32[0, h, :128].cpu().numpy() for h in range(heads)])
            ref = oracle.attention(qf, kf, vf, mode=omode, **kw)
            row[key] = {"gpu_vs_eq1": {"max_abs": float(np.abs(got - ex.out).max()), "mean_abs": float(np.abs(got - ex.out).mean())},
                        "oracle_vs_eq1": {"max_abs": float(np.abs(ref.out - ex.out).max()), "mean_abs": float(np.abs(ref.out - ex.out).mean())},
                        "gpu_vs_oracle_max_abs": float(np.abs(got - ref.out).max())}
            if key == "e2e_hif8":
                m0 = np.ceil((qf[0, :, :128].astype(np.float64) @ np.swapaxes(kf[0, :, :128].astype(np.float64), 1, 2)).max(axis=2)
                             * 1.4426950408889634 / np.sqrt(qf.shape[-1]))
                row["max_updates_integer"] = float((ref.row_m - m0).mean())
            del st
        out[str(S)] = row
        del qd, kd, vd
    return out


PROFILE_CASES = {
    # small cases of the same kernels, sized so that a multi-pass ncu capture ends in a minute
    "attn_d128": workloads.AttnWorkload("profile_attn_d128", 1, 16, 4, 4096, 128, True, 128, 128),
    "attn_d128_long": workloads.AttnWorkload("profile_attn_d128_long", 1, 8, 2, 16384, 128, True, 128, 128),
    "attn_c2": workloads.WORKLOADS["c2_llm_prefill_mha"],
    "attn_c3": workloads.WORKLOADS["c3_llm_prefill_gqa"],
    "attn_c4": workloads.WORKLOADS["c4_vit_encoder"],
    "attn_c5": workloads.WORKLOADS["c5_long_context"],
    "attn_one_tile": workloads.AttnWorkload("profile_attn_one_tile", 1, 8, 8, 4096, 128, True, 128, 128),
    "attn_fp8": workloads.AttnWorkload("profile_attn_fp8", 1, 8, 2, 16384, 128, True, 128, 128),      # 8-bit Q / K
    "attn_d64": workloads.AttnWorkload("profile_attn_d64", 8, 16, 16, 1024, 64, False, 128, 128, key_bias_var=0.5),
}


def run_profile_case(name: str, launches: int = 3, warmup: int = 3):
    """Launch one kernel a few times on a small case (the command ncu captures)."""
    import __graft_entry__ as entry
    entry.build()
    from paper_2602_02071_b200 import binding
    torch.cuda.set_device(0)
    if name in PROFILE_CASES:
        w = PROFILE_CASES[name]
        q, k, v = workloads.make_qkv(w, device="cuda")
        out = torch.empty_like(q)
        fn = lambda: binding.baps_attention_fwd(q, k, v, causal=w.causal, out=out)
        if name == "attn_fp8":
            (q8, qs, _), (k8, ks, _) = (workloads.quantize_e4m3_tiles(t) for t in (q, k))
            fn = lambda: binding.baps_attention_fwd_fp8(q8, k8, v, qs, ks, causal=w.causal, want_stats=False, out=out)
        work, unit = w.flops / 1e12, "TFLOP/s"
    elif name in ("encode", "decode", "exp2_map") or name.startswith("softmax_rows_"):   # softmax_rows[_codes]_<cols>
        n = 1 << 27                                      # 512 MB of fp32: larger than L2
        x = workloads.make_rows(n // 16384, 16384, device="cuda").reshape(-1)
        codes = torch.empty(n, dtype=torch.uint8, device="cuda")
        y = torch.empty(n, dtype=torch.float32, device="cuda")
        if name == "encode":
            fn, work = (lambda: binding.baps_hif8_encode(x, codes)), 5.0 * n / 1e9
        elif name == "decode":
            binding.baps_hif8_encode(x, codes)
            fn, work = (lambda: binding.baps_hif8_decode(codes, y)), 5.0 * n / 1e9
        elif name == "exp2_map":
            binding.baps_hif8_encode(x, codes)
            codes2 = torch.empty_like(codes)
            fn, work = (lambda: binding.baps_exp2_hif8(codes, codes2)), 2.0 * n / 1e9
        elif name.startswith("softmax_rows_codes_"):
            cols = int(name.rsplit("_", 1)[1])
            xr = x[:n // cols * cols].view(-1, cols)
            fn, work = (lambda: binding.baps_softmax_rows_codes(xr, 128)), 5.0 * xr.numel() / 1e9
        else:
            cols = int(name.rsplit("_", 1)[1])
            xr, yr = x[:n // cols * cols].view(-1, cols), y[:n // cols * cols].view(-1, cols)
            fn, work = (lambda: binding.baps_softmax_rows(xr, 128, yr)), 8.0 * xr.numel() / 1e9
        unit = "GB/s"
    else:
        raise SystemExit(f"unknown profile case {name}")
    for _ in range(warmup):
        fn()
    torch.cuda.synchronize()
    ts = []
    for _ in range(launches):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record(); fn(); b.record(); torch.cuda.synchronize()
        ts.append(a.elapsed_time(b))
    binding.poll_async_error()
    print(json.dumps({"profile_case": name, "ms": ts, "rate": work / (min(ts) * 1e-3), "unit": unit}))
    return 0


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--profile-case", default=None,
                    help="launch one kernel a few times on a small case and exit (for ncu)")
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=20)
    ap.add_argument("--warmup", type=int, default=5)
    ap.add_argument("--workload", default=DEFAULT_WORKLOAD, choices=sorted(
        k for k, w in workloads.WORKLOADS.items() if w.dtype == "bf16"))
    ap.add_argument("--impl", default="baps", choices=["baps", "reference"])
    ap.add_argument("--no-extra", action="store_true", help="skip the supplementary measurements")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    args = ap.parse_args()
    args.warmup = max(args.warmup, 3) if args.impl == "baps" else args.warmup

    if args.profile_case:
        return run_profile_case(args.profile_case)
    if args.impl == "reference":
        return run_reference(args)

    rank, world, local = dist_info()
    if not torch.cuda.is_available():
        raise SystemExit("bench.py needs a CUDA device (there is no CPU fallback)")
    torch.cuda.set_device(local)
    use_dist = world > 1
    if use_dist:
        import torch.distributed as dist
        dist.init_process_group("nccl", device_id=torch.device("cuda", local))

    import __graft_entry__ as entry
    if rank == 0:
        entry.build()
    if use_dist:
        dist.barrier()
    from paper_2602_02071_b200 import binding
    binding.load()

    peaks, peak_kind = load_peaks()
    w = workloads.WORKLOADS[args.workload]
    qh, kh, vh = workloads.make_qkv(w)
    qh, kh, vh = qh.pin_memory(), kh.pin_memory(), vh.pin_memory()
    q, k, v = qh.cuda(non_blocking=True), kh.cuda(non_blocking=True), vh.cuda(non_blocking=True)
    flush_buf = torch.empty(256 << 20, dtype=torch.uint8, device="cuda")    # > 126 MB L2
    torch.cuda.synchronize()

    # ---- device-resident timing ---------------------------------------------------------------
    if use_dist:
        dist.barrier()
    torch.cuda.synchronize()
    with ClockSampler(local) as cs:
        times, launches = time_attention(w, q, k, v, args.steps, args.warmup, flush_buf)
    torch.cuda.synchronize()
    total_ms = replicas.max_over_ranks(float(np.sum(times)), device="cuda")
    ms_per_step = total_ms / args.steps
    value = replicas.whole_job_rate(w.flops, ms_per_step, world) / 1e12

    # ---- end to end with host buffers -----------------------------------------------------------
    e2e_times, h2d, d2h = time_e2e(w, qh, kh, vh, max(3, args.steps // 3), 3)
    e2e_ms = replicas.max_over_ranks(float(np.sum(e2e_times)), device="cuda")
    e2e_value = replicas.whole_job_rate(w.flops, e2e_ms / len(e2e_times), world) / 1e12

    if rank != 0:
        if use_dist:
            dist.barrier(); dist.destroy_process_group()
        return 0

    # ---- roofline of the dominant (only) kernel ----------------------------------------------------
    kernel_ms = float(np.mean(times))
    achieved = w.flops / (kernel_ms * 1e-3) / 1e12
    cap = NCU_CAPTURES.get(w.name) or {}
    clocks = cs.summary()
    roofline = {
        "bound": "tensor", "achieved": achieved, "peak": peaks["bf16_tflops"], "unit": "TFLOP/s",
        "frac": achieved / peaks["bf16_tflops"], "peak_kind": f"{peak_kind} bf16 burst (kernel timed alone)",
        "frac_of_sustained": achieved / peaks.get("bf16_tflops_sustained", peaks["bf16_tflops"]),
        # context: the same rate against the vendor's dense bf16 figure, and the clock-independent
        # tensor-pipe-active counter of the committed ncu capture of this workload
        "frac_of_nominal_dense_bf16": achieved / NOMINAL_DENSE_BF16_TFLOPS,
        "tensor_pipe_active_pct_ncu": cap.get("tensor_pipe_active_pct"),
        "traffic": cap.get("traffic"),
        "algorithmic_bytes": float(2 * (2 * w.B * w.H + 2 * w.B * w.Hkv) * w.S * w.D),
        "kernel": "attention_d64_kernel" if w.D == 64 else "paired_attention_tc_kernel<false>", "best_ms": float(np.min(times)),
        "median_ms": float(np.median(times)),
        "ms_x_sm_mhz": kernel_ms * clocks["sm_mhz"] if clocks["sm_mhz"] else None,
        "issue_roofline": issue_roofline(w, kernel_ms, clocks["sm_mhz"]),
    }

    # ---- error against the checker and against exact attention (sampled tiles) ------------------
    import oracle
    tiles = error_sample_tiles(w)
    qf, kf, vf = (t.float().numpy() for t in (qh, kh, vh))
    st = binding.baps_attention_fwd_ex(q, k, v, causal=w.causal, block_q=w.block_q, block_k=w.block_k)
    got = np.stack([st.out_f32[b, h, i * 128:(i + 1) * 128].cpu().numpy() for b, h, i in tiles])
    ref = oracle.attention(qf, kf, vf, causal=w.causal, block_q=w.block_q, block_k=w.block_k,
                           tiles=np.array(tiles, dtype=np.int32))
    ex = oracle.attention(qf, kf, vf, causal=w.causal, block_q=w.block_q, block_k=w.block_k,
                          tiles=np.array(tiles, dtype=np.int32), mode=oracle.MODE_EXACT)
    errors = {
        "tiles_checked": len(tiles),
        "gpu_vs_oracle": {"max_abs": float(np.abs(got - ref.out).max()), "mean_abs": float(np.abs(got - ref.out).mean())},
        "gpu_vs_exact": {"max_abs": float(np.abs(got - ex.out).max()), "mean_abs": float(np.abs(got - ex.out).mean())},
        "oracle_vs_exact": {"max_abs": float(np.abs(ref.out - ex.out).max()), "mean_abs": float(np.abs(ref.out - ex.out).mean())},
        "restart_rate_sampled": float(ref.restarts.sum() / max(1, (ref.n_tiles - 1).sum())),
    }
    # the three setups of Section 4.1 on the same inputs, each against Eq. (1) evaluated by the checker
    # in double precision (Default = Eq. (2) with fp32 exponentials and bf16 P on the tensor core)
    def _err(a, b_):
        return {"max_abs": float(np.abs(a - b_).max()), "mean_abs": float(np.abs(a - b_).mean())}
    ref2 = oracle.attention(qf, kf, vf, causal=w.causal, block_q=w.block_q, block_k=w.block_k,
                            tiles=np.array(tiles, dtype=np.int32), mode=oracle.MODE_EXP2_HIF8)
    setups = {"e2e_hif8": _err(got, ex.out)}
    for key, mode in (("default", binding.MODE_EXACT), ("exp2_hif8", binding.MODE_EXP2_HIF8)):
        stm = binding.baps_attention_fwd_ex(q, k, v, causal=w.causal, block_q=w.block_q, block_k=w.block_k, mode=mode)
        gm = np.stack([stm.out_f32[b, h, i * 128:(i + 1) * 128].cpu().numpy() for b, h, i in tiles])
        setups[key] = _err(gm, ex.out)
        if mode == binding.MODE_EXP2_HIF8:
            errors["exp2_gpu_vs_oracle"] = _err(gm, ref2.out)
        t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        t0.record()
        for _ in range(3):
            binding.baps_attention_fwd_ex(q, k, v, causal=w.causal, block_q=w.block_q, block_k=w.block_k,
                                          mode=mode, want_stats=False)
        t1.record(); torch.cuda.synchronize()
        setups[key]["tflops"] = w.flops / (t0.elapsed_time(t1) / 3 * 1e-3) / 1e12
        del stm
    errors["setups_vs_eq1"] = setups
    # the comparison setups of Section 4.2 (Table 1), evaluated by the checker alone (CPU) on a subset of
    # the sampled tiles, each against Eq. (1): which 8-bit format feeds / leaves the exponential, and
    # what casting the scores before the subtraction ("Naive E2E") costs
    ftiles = np.array(tiles[::3][:8], dtype=np.int32)
    fex = oracle.attention(qf, kf, vf, causal=w.causal, block_q=w.block_q, block_k=w.block_k, tiles=ftiles,
                           mode=oracle.MODE_EXACT)
    formats = {"tiles_checked": int(len(ftiles)), "computed_by": "checker (CPU)"}
    for key, mode in (("e2e_hif8", oracle.MODE_E2E_HIF8), ("exp2_hif8", oracle.MODE_EXP2_HIF8),
                      ("exp2_e4m3", oracle.MODE_EXP2_E4M3), ("exp2_e5m2", oracle.MODE_EXP2_E5M2),
                      ("exp2_e4m3xe5m2", oracle.MODE_EXP2_E4M3_E5M2), ("naive_e2e", oracle.MODE_NAIVE_E2E)):
        fo = oracle.attention(qf, kf, vf, causal=w.causal, block_q=w.block_q, block_k=w.block_k, tiles=ftiles, mode=mode)
        formats[key] = _err(fo.out, fex.out)
    errors["formats_vs_eq1"] = formats
    # restart rates of the whole workload (Table 4's ARR / PRR) for lambda = 0, 1, 2
    rr = {}
    for lam in (0, 1, 2):
        _, rates = binding.baps_attention_restart_rates(q, k, v, causal=w.causal, lam=lam)
        arr_, prr_ = rates.cpu().tolist()
        rr[f"lambda_{lam}"] = {"ARR": arr_, "PRR": prr_}
    errors["restart_rates_gpu"] = rr
    errors["restart_rates_lambda_1_by_b0"] = restart_rates_both_b0(w, q, k, v)
    if world == 1 and not args.no_extra:
        errors["fig2"] = fig2_experiment()

    # ---- CPU baseline: the checker on a bounded sample ------------------------------------------------
    cpu = None
    if not args.no_cpu_baseline:
        btiles = bounded_sample_tiles(w, target_flops=4.0e11)
        dt, fl, cores = oracle_sample_time(w, qh, kh, vh, btiles)
        cpu = {"value": fl / dt / 1e12, "unit": UNIT, "cores": cores, "kind": "oracle",
               "sample": f"{len(btiles)} of {w.n_query_tiles} query tiles (evenly strided over heads and "
                         f"positions), {dt:.1f} s; rate = their flops / that time",
               "extrapolated_full_workload_s": dt * w.flops / fl,
               "note": "full-workload time is extrapolated from the sample by flops"}

    extra = None
    if not args.no_extra and world == 1:
        del q, k, v
        torch.cuda.empty_cache()
        extra = extra_measurements(peaks, flush_buf, skip=w.name)

    line = {
        "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": ms_per_step, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "bf16", "data": "synthetic",
        "config": {"workload": w.name, "B": w.B, "H": w.H, "Hkv": w.Hkv, "S": w.S, "D": w.D,
                   "causal": w.causal, "block": [w.block_q, w.block_k], "lambda": 1,
                   "l2": "flushed between steps (256 MB write)", "multi_gpu": "independent replicas"},
        "roofline": roofline, "cpu_baseline": cpu, "clocks": clocks,
        "e2e": {"value": e2e_value, "unit": UNIT, "h2d_bytes_per_step": h2d, "d2h_bytes_per_step": d2h,
                "ms_per_step": e2e_ms / len(e2e_times),
                "pipeline": "double-buffered over three streams (copy in, compute, copy out)"},
        "gpu_launches": int(launches), "errors": errors, "extra": extra,
    }
    print(json.dumps(line), flush=True)
    if use_dist:
        dist.barrier(); dist.destroy_process_group()
    return 0


if __name__ == "__main__":
    sys.exit(main())
