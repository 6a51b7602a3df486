#!/usr/bin/env python
"""Benchmark of the HiFA4 hot path on B200: one step = Smooth-QK + HIF4 quantization of Q/K/V
followed by the fused 4-bit-operand attention forward (Algorithm 1) over one batch of synthetic
prefill activations.  Prints ONE JSON line: metric, value (whole-job TFLOP/s over the timed steps),
roofline (attention launch against the measured BF16 tensor peak), quantize split, end-to-end figures
with host buffers (FP16 and FP32 output), clocks sampled during the timed region, CPU-oracle baseline,
dense GEMM peaks measured in the same run (BF16, FP8), context numbers and a sweep over the other
configurations and variants.

    python bench.py [--gpus N] [--steps K] [--warmup W] [--workload C2] [--impl ours|reference]

N > 1 is launched by torch.distributed.run, one rank per GPU; every rank processes its own copy
of the workload (independent batches: the path has no exchange step), so scaling is weak.
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

import torch

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

from paper_2607_04302_b200 import synth  # noqa: E402

METRIC = "4-bit attention prefill TFLOPS on 1 B200; % of dense 4-bit tensor peak"
UNIT = "TFLOP/s"
NOMINAL = {"fp4": 9000.0, "fp8": 4500.0, "bf16": 2250.0}      # dense TFLOP/s, context only
# executed warp instructions per 32 scores and DRAM bytes per launch (ncu), from profiles/attention_pair_and_sm_pairs.md
NCU_INSTR_PER_WARP_SCORE = {"attention_fwd_pair_kernel<0, 0>": 10.3, "attention_fwd_pair_kernel<0, 1>": 10.3,
                            "attention_fwd_cta2_kernel<0>": 11.7, "attention_fwd_ws64_kernel<128, fp32 P>": 11.3}
NCU_TRAFFIC_BYTES = {("C2-qwen3-8b-4k", 64): 68.99e6, ("C2-qwen3-8b-4k", 128): 70.12e6, ("C4-gemma2-9b-8k", 64): 232.8e6}
# Issue slots the method itself needs per score on this machine (per 32 scores one warp instruction each), with P quantized
# on packed FP16 pairs: exponential 1, scale-subtract FMA 0.5 (packed), FP16 conversion 0.5, row maximum 0.5, scale 0.5,
# subgroup maxima 0.6, shift selection 0.8, scale and round 0.5, BF16 image 0.5, rescale of the history about 0.7, per-row
# scalars and tensor-memory traffic about 0.6: 6.7.
ALGORITHMIC_SLOTS_PER_SCORE = 6.7


def attn_flops(cfg) -> float:
    f = 4.0 * cfg.B * cfg.Hq * cfg.N * cfg.N * cfg.d
    return f / 2 if cfg.causal else f


def two_blocks_chosen(cfg, sms: int, qmean: bool = False) -> bool:
    """Whether the library runs this d = 128 workload in the two-block kernel (csrc/hifa4_dispatch.h)."""
    unit, units = (cfg.N + 127) // 128 * (cfg.Hq // cfg.Hkv), cfg.Hkv * cfg.B
    blocks, pairs = unit * units, (unit + 1) // 2 * units
    waves, pairs_per_sm = -(-pairs // sms), ((blocks + 1) // 2) / sms
    if cfg.Bc == 128:
        if cfg.causal and cfg.N > 128:
            return pairs_per_sm >= min(0.6 + (cfg.N - 256) / 1000.0, 1.37 if qmean else 1.5)
        tiles = (cfg.N + 127) // 128 * 2
        return 2.9 + (1.63 if qmean else 1.72) * waves * tiles <= -(-blocks // sms) * (tiles + (2.0 if qmean else 1.5))
    if cfg.causal and cfg.N > 320:
        return pairs_per_sm >= min(1.05 + (cfg.N - 512) / 4200.0, 1.42)
    full, rest = divmod(blocks, 2 * sms)
    tiles = (cfg.N + 63) // 64
    waves64 = full + (0 if rest == 0 else (0.74 if cfg.causal else 0.44) if rest <= sms else 1)
    if cfg.causal:
        return 2.2 + 0.74 * waves * tiles <= waves64 * (tiles + 0.75)
    return 3.1 + (1.02 if qmean else 0.915) * waves * (tiles + 1.3) <= waves64 * (tiles + 4.0)


def attention_kernel(cfg, *, p_f32=False, qmean=False, f8qk=False, sms=148) -> str:
    """Name of the attention kernel that the timed step launches."""
    qm = int(bool(qmean))
    if f8qk:
        return "attention_fwd_ws64_kernel<128, f8f6f4 experiment> + 2 x f8_image_kernel"
    if cfg.d == 128 and not p_f32 and two_blocks_chosen(cfg, sms, qmean):
        return f"attention_fwd_pair_kernel<{qm}, {int(cfg.Bc == 128)}>"
    blocks = (cfg.N + 127) // 128 * cfg.Hq * cfg.B
    if cfg.d == 256 and cfg.Bc == 64 and not p_f32 and blocks > sms:
        return f"attention_fwd_cta2_kernel<{qm}>"
    if cfg.Bc == 64:
        return f"attention_fwd_ws64_kernel<{cfg.d}{', fp32 P' if p_f32 else ''}>"
    return "attention_fwd_ws_kernel<4>" if cfg.d == 128 else f"attention_fwd_kernel<{cfg.d},{cfg.Bc}>"


def measured_peaks():
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(p):
        d = json.load(open(p))
        return dict(hbm=d["hbm_gbs"], bf16=d["bf16_tflops"], bf16_sustained=d["bf16_tflops_sustained"],
                    source="measured")
    return dict(hbm=6650.0, bf16=1590.0, bf16_sustained=1400.0, source="fallback")


class ClockSampler:
    """Samples SM clocks and throttle reasons with nvidia-smi while the GPU is under load.

    nvidia-smi needs ~100 ms per sample, so a short timed region yields few samples; the sampler is
    started before warm-up and the benchmark keeps the GPU busy (same step function) until at least
    a few samples fall inside the marked window."""
    Q = ("clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,clocks_event_reasons.hw_slowdown,"
         "clocks_event_reasons.hw_thermal_slowdown,clocks_event_reasons.sw_thermal_slowdown,"
         "clocks_event_reasons.sw_power_cap")

    def __init__(self, index: int):
        self.index, self.rows, self.proc, self.thr = index, [], None, None
        self.t0 = self.t1 = None

    def start(self):
        try:
            self.proc = subprocess.Popen(["nvidia-smi", "-i", str(self.index), f"--query-gpu={self.Q}",
                                          "--format=csv,noheader,nounits", "-lms", "50"],
                                         stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
        except OSError:
            return
        self.thr = threading.Thread(target=self._read, daemon=True)
        self.thr.start()

    def _read(self):
        for line in self.proc.stdout:
            self.rows.append((time.perf_counter(), [c.strip() for c in line.split(",")]))

    def mark_begin(self):
        self.t0 = time.perf_counter()

    def mark_end(self):
        self.t1 = time.perf_counter()

    def samples_in_window(self):
        if self.t0 is None:
            return 0
        t1 = self.t1 if self.t1 is not None else time.perf_counter()
        return sum(1 for t, _ in self.rows if self.t0 <= t <= t1)

    def stop(self):
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except subprocess.TimeoutExpired:
            self.proc.kill()
        sm, mx, reasons, power = [], None, set(), []
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for t, r in self.rows:
            if self.t0 is None or not (self.t0 <= t <= (self.t1 or t)):
                continue
            try:
                sm.append(float(r[0])); mx = float(r[1]); power.append(float(r[2]))
            except (ValueError, IndexError):
                continue
            for n, v in zip(names, r[4:8]):
                if v.lower().startswith("active"):
                    reasons.add(n)
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": mx,
                "reasons": sorted(reasons), "samples": len(sm),
                "power_w_max": max(power) if power else None,
                "window": "timed steps plus identical untimed steps run until 8 samples were taken"}


def max_over_ranks(dist, ms: float, device) -> float:
    """Device time of the slowest rank (the job is as slow as its slowest rank)."""
    if dist is None:
        return ms
    t = torch.tensor([ms], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def whole_job_tflops(cfg, world: int, steps: int, total_ms: float) -> float:
    """Aggregate over all ranks: every rank processes its own copy of the workload (weak scaling)."""
    return world * attn_flops(cfg) * steps / (total_ms * 1e-3) / 1e12


def measure_gemm_peaks(dev):
    """Dense GEMM throughput measured in this run (8192^3, best of 5): BF16 through torch.matmul, FP8 (e4m3) and
    FP4 (e2m1 with one e4m3 scale per 16 elements, the block-scaled 4-bit format the tensor cores take) through
    torch._scaled_mm; each is null where the installed torch does not expose it."""
    res = {"bf16_tflops": None, "fp8_tflops": None, "fp4_tflops": None}
    n = 8192
    try:
        a = torch.randn((n, n), device=dev, dtype=torch.bfloat16)
        b = torch.randn((n, n), device=dev, dtype=torch.bfloat16)

        def best(fn):
            for _ in range(2):
                fn()
            torch.cuda.synchronize()
            t = []
            for _ in range(5):
                e0 = torch.cuda.Event(enable_timing=True); e1 = torch.cuda.Event(enable_timing=True)
                e0.record(); fn(); e1.record()
                torch.cuda.synchronize()
                t.append(e0.elapsed_time(e1))
            return 2.0 * n ** 3 / (min(t) * 1e-3) / 1e12

        res["bf16_tflops"] = best(lambda: torch.matmul(a, b))
        a8 = a.to(torch.float8_e4m3fn)
        b8 = b.to(torch.float8_e4m3fn).t().contiguous().t()          # column-major second operand
        one = torch.ones((), device=dev, dtype=torch.float32)
        res["fp8_tflops"] = best(lambda: torch._scaled_mm(a8, b8, scale_a=one, scale_b=one, out_dtype=torch.bfloat16))
    except Exception as e:                                             # context only: never fail the bench on it
        res["error"] = str(e)[:160]
    try:
        # random 4-bit codes, all block scales 1.0 in the 128 x 4 tiled layout the block-scaled GEMM reads
        a4 = torch.randint(0, 256, (n, n // 2), dtype=torch.uint8, device=dev).view(torch.float4_e2m1fn_x2)
        b4 = torch.randint(0, 256, (n, n // 2), dtype=torch.uint8, device=dev).view(torch.float4_e2m1fn_x2)
        sc = torch.ones((n * (n // 16),), device=dev, dtype=torch.float32).to(torch.float8_e4m3fn)
        res["fp4_tflops"] = best(lambda: torch._scaled_mm(a4, b4.t(), scale_a=sc, scale_b=sc, out_dtype=torch.bfloat16))
    except Exception as e:
        res["fp4_error"] = str(e)[:160]
    return res


def time_workload(hb, cfg, dev, steps, warmup, flush_l2, s=None, inv_s=None, qmean=False, p_f32=False, fused_q=False,
                  f8qk=False):
    """Device-resident timing of one configuration: per-step time of quantize + attention (events around each
    step, L2 flushed between steps) and, from a second pass with one more event, the attention launch alone.
    fused_q: K and V through the quantizer, Q quantized inside the attention kernel (hifa4_attention_fwd_qraw).
    f8qk: the kind::f8f6f4 experiment (hifa4_attention_fwd_f8qk; its two operand-image launches count as attention)."""
    q, k, v = synth.make_qkv_device(cfg, dev)
    dt = hb._DT[q.dtype]
    qkv = hb.alloc_qkv(cfg.B, cfg.Hq, cfg.Hkv, cfg.N, cfg.d, dt, dev, qmean=qmean)
    out = torch.empty((cfg.B, cfg.Hq, cfg.N, cfg.d), dtype=torch.float32, device=dev)
    status = torch.zeros(1, dtype=torch.int32, device=dev)
    f8_ws = None
    if f8qk:
        import ctypes
        sh_ = hb._shape(cfg.B, cfg.Hq, cfg.Hkv, cfg.N, cfg.d, dt, None)
        f8_ws = torch.empty(int(hb.lib().hifa4_f8qk_workspace_bytes(ctypes.byref(sh_))), dtype=torch.uint8, device=dev)

    def step(split):
        hb.quantize_qkv(None if fused_q else q, k, v, s, inv_s, out=qkv, d_status=status, qmean=qmean, Hq=cfg.Hq)
        mid = None
        if split:
            mid = torch.cuda.Event(enable_timing=True)
            mid.record()
        if f8qk:
            hb.attention_fwd_f8qk(qkv, cfg.causal, out_dtype=hb.F32, out=out, workspace=f8_ws, d_status=status)
        elif fused_q:
            hb.attention_fwd_qraw(q, s, qkv, cfg.causal, out_dtype=hb.F32, out=out, d_status=status,
                                  p_dtype=hb.F32 if p_f32 else hb.F16)
        else:
            hb.attention_fwd(qkv, cfg.causal, Bc=cfg.Bc, out_dtype=hb.F32, out=out, d_status=status,
                             p_dtype=hb.F32 if p_f32 else hb.F16, qmean=qmean)
        return mid

    for _ in range(warmup):
        flush_l2(); step(False)
    torch.cuda.synchronize()
    ev, ev2 = [], []
    for _ in range(steps):
        flush_l2()
        a = torch.cuda.Event(enable_timing=True); b = torch.cuda.Event(enable_timing=True)
        a.record(); step(False); b.record()
        ev.append((a, b))
    for _ in range(steps):
        flush_l2()
        a = torch.cuda.Event(enable_timing=True); b = torch.cuda.Event(enable_timing=True)
        a.record(); m = step(True); b.record()
        ev2.append((a, m, b))
    torch.cuda.synchronize()
    assert int(status.item()) == 0, f"device status {int(status.item())}"
    ms = sum(a.elapsed_time(b) for a, b in ev) / steps
    attn = sum(m.elapsed_time(b) for _, m, b in ev2) / steps
    quant = sum(a.elapsed_time(m) for a, m, _ in ev2) / steps
    fl = attn_flops(cfg)
    return {"ms_per_step": ms, "tflops": fl / (ms * 1e-3) / 1e12, "attention_ms": attn,
            "attention_tflops": fl / (attn * 1e-3) / 1e12, "quantize_ms": quant}


def oracle_time(cfg, q, k, v, s, inv_s, heads):
    """Time the CPU oracle, as it stands, on whole heads of the workload (batch 0)."""
    from oracle import hifa4_oracle as orc
    import numpy as np
    dt = orc.F16 if cfg.dtype == "fp16" else orc.BF16
    idx = np.arange(cfg.N, dtype=np.int32)
    grp = cfg.Hq // cfg.Hkv
    t0 = time.perf_counter()
    for h in heads:
        g = h // grp
        orc.attention_rows(q[0, h], idx, k[0, g], v[0, g], None if s is None else s[g],
                           None if inv_s is None else inv_s[g], causal=cfg.causal, Bc=cfg.Bc, in_dtype=dt)
    return time.perf_counter() - t0, orc.num_threads()


def head_flops(cfg) -> float:
    f = 4.0 * cfg.N * cfg.N * cfg.d
    return f / 2 if cfg.causal else f


def host_inputs(cfg):
    q, k, v = synth.make_qkv(cfg)
    return q, k, v


def oracle_scales(cfg):
    """Smooth-QK factors from the oracle's own calibration (used by the CPU legs only)."""
    if cfg.smooth_mode == 0:
        return None, None
    from oracle import hifa4_oracle as orc
    small = synth.config(cfg.name.split("-")[0], cal_samples=min(cfg.cal_samples, 4), cal_tokens=min(cfg.cal_tokens, 256))
    qc, kc = synth.make_calibration(small)
    cal = orc.smooth_calibrate(qc.float().numpy(), kc.float().numpy(), cfg.smooth_mode)
    return cal["s"], cal["inv_s"]


def config_dict(cfg, args, world):
    """The `config` object of the JSON line (the same for both arms, so that they can be matched)."""
    return {"workload": cfg.name, "B": cfg.B, "Hq": cfg.Hq, "Hkv": cfg.Hkv, "N": cfg.N, "d": cfg.d,
            "causal": cfg.causal, "Br": 128, "Bc": cfg.Bc, "in_dtype": cfg.dtype, "out_dtype": "f32",
            "p_dtype": "f32 (variant)" if args.p_f32 else "f16", "qmean": bool(args.qmean),
            "smooth_mode": cfg.smooth_mode, "step": "hifa4_quantize_qkv + hifa4_attention_fwd",
            "l2": "flushed between steps (256 MiB write, then a 256 MiB read that drains the dirty lines), outside the per-step events",
            "parallelism": f"replicated batches x{world}"}


def run_reference(args, cfg, rank):
    """--impl reference: the CPU oracle, as it stands, on a bounded sample per step."""
    if rank != 0:
        return
    from oracle import hifa4_oracle as orc
    orc.build()
    q, k, v = (t.float().numpy() for t in host_inputs(cfg))
    s, inv_s = oracle_scales(cfg)
    t1, cores = oracle_time(cfg, q, k, v, s, inv_s, [0])
    # the whole run (warm-up included) gets about two minutes of CPU work, at most 8 s per step
    per_step = min(8.0, 120.0 / max(args.steps + args.warmup, 1))
    n_heads = max(1, min(cfg.Hq, int(per_step / max(t1, 1e-3))))
    heads = [int(i * cfg.Hq / n_heads) for i in range(n_heads)]
    for _ in range(args.warmup):
        oracle_time(cfg, q, k, v, s, inv_s, heads[:1])
    tot = 0.0
    for _ in range(args.steps):
        t, cores = oracle_time(cfg, q, k, v, s, inv_s, heads)
        tot += t
    val = n_heads * head_flops(cfg) * args.steps / tot / 1e12
    sample = f"{n_heads} of {cfg.B * cfg.Hq} (batch, head) slices of {cfg.name}, all {cfg.N} rows each, per step"
    line = {"impl": "reference", "metric": METRIC, "value": val, "unit": UNIT, "n_gpus": args.gpus,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": tot / args.steps * 1e3,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
            "data": "synthetic", "config": config_dict(cfg, args, int(os.environ.get("WORLD_SIZE", "1"))),
            "cpu_baseline": {"value": val, "unit": UNIT, "cores": cores, "kind": "oracle", "sample": sample},
            "e2e": {"value": val, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
            "gpu_launches": 0}
    print(json.dumps(line), flush=True)


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=100)
    ap.add_argument("--warmup", type=int, default=10)
    ap.add_argument("--workload", default="C2", help="C2 (headline), C3, C4, C5 or C5@<N>")
    ap.add_argument("--noncausal", action="store_true")
    ap.add_argument("--Bc", type=int, default=0, help="key-tile width (default: the configuration's, 64)")
    ap.add_argument("--p-f32", action="store_true",
                    help="variant: quantize the FP32 exponential (not the method's FP16 P; for comparison only)")
    ap.add_argument("--qmean", action="store_true", help="with the Q-Mean auxiliary (Algorithm 1 lines 2 and 6)")
    ap.add_argument("--f8qk", action="store_true",
                    help="experiment: Q K^T as kind::f8f6f4 with one accumulator per HIF4 group (d = 128, Bc = 64)")
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-context", action="store_true", help="skip the torch SDPA / N=8192 context numbers")
    ap.add_argument("--no-sweep", action="store_true",
                    help="skip the sweep over the other configurations and variants (headline workload only)")
    args = ap.parse_args()
    args.warmup = max(args.warmup, 3) if args.impl == "ours" else args.warmup

    rank = int(os.environ.get("RANK", "0"))
    local_rank = int(os.environ.get("LOCAL_RANK", "0"))
    world = int(os.environ.get("WORLD_SIZE", "1"))

    name, _, n_over = args.workload.partition("@")
    over = {}
    if n_over:
        over["N"] = int(n_over)
    if args.noncausal:
        over["causal"] = False
    if args.Bc:
        over["Bc"] = args.Bc
    cfg = synth.config(name, **over)

    if args.impl == "reference":
        run_reference(args, cfg, rank)
        return

    from paper_2607_04302_b200 import binding as hb
    hb.lib()                                  # fail loudly if the CUDA library is missing
    torch.cuda.set_device(local_rank)
    dev = torch.device("cuda", local_rank)
    dist = None
    if world > 1:
        import torch.distributed as dist_mod
        dist = dist_mod
        os.environ.setdefault("MASTER_ADDR", "127.0.0.1")
        dist.init_process_group("nccl", device_id=dev)

    # ---- inputs (resident in HBM) and offline calibration
    big = cfg.B * cfg.Hq * cfg.N * cfg.d > (1 << 28)
    if big:
        q, k, v = synth.make_qkv_device(cfg, dev)
        qh = kh = vh = None
    else:
        qh, kh, vh = host_inputs(cfg)
        q, k, v = qh.to(dev), kh.to(dev), vh.to(dev)
    s = inv_s = None
    if cfg.smooth_mode:
        qc, kc = synth.make_calibration(cfg, samples=min(cfg.cal_samples, 8), tokens=min(cfg.cal_tokens, 512))
        s, inv_s = hb.smooth_calibrate(qc.to(dev), kc.to(dev), cfg.smooth_mode)
    dt = hb._DT[q.dtype]
    qkv = hb.alloc_qkv(cfg.B, cfg.Hq, cfg.Hkv, cfg.N, cfg.d, dt, dev, qmean=args.qmean)
    out = torch.empty((cfg.B, cfg.Hq, cfg.N, cfg.d), dtype=torch.float32, device=dev)
    status = torch.zeros(1, dtype=torch.int32, device=dev)
    flush = torch.empty(256 << 20, dtype=torch.uint8, device=dev)       # > 126 MB of L2
    flush_rd = torch.zeros(64 << 20, dtype=torch.float32, device=dev)   # 256 MiB that are only read

    f8_ws = None
    if args.f8qk:
        import ctypes
        sh_ = hb._shape(cfg.B, cfg.Hq, cfg.Hkv, cfg.N, cfg.d, dt, None)
        f8_ws = torch.empty(int(hb.lib().hifa4_f8qk_workspace_bytes(ctypes.byref(sh_))), dtype=torch.uint8, device=dev)

    def flush_l2():
        # Write a buffer larger than L2, then read another one: the write evicts every line of the
        # previous step, the read pass pushes the dirty lines of the write out to HBM, so that their
        # write-back does not run inside the next step's timed region.
        flush.zero_()
        flush_rd.sum()

    def step(split=False):
        """One pass of the hot path.  split: record an event between the two launches (used only by the
        pass that attributes time to each kernel: the event keeps the attention grid, which is launched
        with programmatic stream serialization, from starting while the quantize grid drains)."""
        hb.quantize_qkv(q, k, v, s, inv_s, out=qkv, d_status=status, qmean=args.qmean)
        mid = None
        if split:
            mid = torch.cuda.Event(enable_timing=True)
            mid.record()
        if args.f8qk:
            hb.attention_fwd_f8qk(qkv, cfg.causal, out_dtype=hb.F32, out=out, workspace=f8_ws, d_status=status)
        else:
            hb.attention_fwd(qkv, cfg.causal, Bc=cfg.Bc, out_dtype=hb.F32, out=out, d_status=status,
                             p_dtype=hb.F32 if args.p_f32 else hb.F16, qmean=args.qmean)
        return mid

    def barrier():
        if dist is not None:
            dist.barrier()
        torch.cuda.synchronize()

    sampler = ClockSampler(local_rank)
    sampler.start()
    # spin-up (untimed, before the W warm-up steps): a fresh process on a fresh box starts with idle
    # clocks and unloaded modules; a quarter of a second of the same steps brings both up
    t_spin = time.perf_counter() + 0.25
    while time.perf_counter() < t_spin:
        for _ in range(10):
            flush_l2()
            step()
        torch.cuda.synchronize()
    for _ in range(args.warmup):
        flush_l2()
        step()
    barrier()
    assert int(status.item()) == 0, f"device status {int(status.item())}"

    c0 = hb.get_counters()["launches"]
    ev = []
    barrier()
    sampler.mark_begin()
    for _ in range(args.steps):
        flush_l2()                                                      # L2 flush, outside the events
        a = torch.cuda.Event(enable_timing=True)
        b = torch.cuda.Event(enable_timing=True)
        a.record()
        step()
        b.record()
        ev.append((a, b))
    barrier()
    launches = hb.get_counters()["launches"] - c0
    # second pass over the same steps with one more event per step, for the per-kernel durations
    ev_split = []
    for _ in range(args.steps):
        flush_l2()
        a = torch.cuda.Event(enable_timing=True)
        b = torch.cuda.Event(enable_timing=True)
        a.record()
        mid = step(split=True)
        b.record()
        ev_split.append((a, mid, b))
    barrier()
    # keep the same load on the GPU (untimed) until nvidia-smi has taken a few samples of it
    t_lim = time.perf_counter() + 3.0
    while sampler.proc is not None and sampler.samples_in_window() < 8 and time.perf_counter() < t_lim:
        for _ in range(20):
            flush_l2()
            step()
        torch.cuda.synchronize()
    sampler.mark_end()
    clocks = sampler.stop()
    step_ms = [a.elapsed_time(b) for a, b in ev]
    attn_ms = [m.elapsed_time(b) for _, m, b in ev_split]
    quant_ms = [a.elapsed_time(m) for a, m, _ in ev_split]
    split_step_ms = sum(a.elapsed_time(b) for a, _, b in ev_split) / len(ev_split)
    total_ms = sum(step_ms)
    total_ms = max_over_ranks(dist, total_ms, dev)
    assert int(status.item()) == 0, f"device status {int(status.item())}"

    # ---- end to end through the raw C-ABI entry point with host buffers (pinned), copies timed.  Two figures:
    # FP16 output (the method's final normalisation is FP16: Appendix, "FP16 operations") and FP32 output (the
    # dtype the parity tests judge); the FP16 one is the line's `e2e`.
    e2e = e2e_f32 = None
    if not big and not args.qmean and not args.p_f32 and not args.f8qk:
        pq, pk, pv = qh.pin_memory(), kh.pin_memory(), vh.pin_memory()
        # One problem per batch element: hifa4_attention_fwd_raw on its Q/K/V (contiguous slices).  One stream
        # carries all host-to-device copies, one all device-to-host copies, the kernels of consecutive problems
        # alternate between two more.  Device buffers come in two sets used by alternate steps, tied by events: a
        # set's inputs are overwritten only after the kernels that read them, its output only after the read-back
        # of the previous result, so consecutive steps pipeline (copy-in of step i+1 under the kernels of step i and
        # the read-back of step i-1) exactly as they would with different data in every step.  Few large copies:
        # with one problem per pair of KV head groups (twelve copies in, four out per step) the same pipeline was
        # 15 % slower.
        G = cfg.Hq // cfg.Hkv
        NB = 2
        streams = [torch.cuda.Stream(device=dev) for _ in range(2)]
        h2d_stream, d2h_stream = torch.cuda.Stream(device=dev), torch.cuda.Stream(device=dev)
        ws_bytes = hb.attention_raw_workspace_bytes(1, cfg.Hq, cfg.Hkv, cfg.N, cfg.d, dt, cfg.causal, cfg.Bc)
        ws_s = [torch.empty(ws_bytes, dtype=torch.uint8, device=dev) for _ in streams]
        in_sets = [tuple(torch.empty_like(t) for t in (q, k, v)) for _ in range(NB)]

        def fork():
            e = torch.cuda.Event()
            e.record()
            for st_i in streams + [h2d_stream, d2h_stream]:
                st_i.wait_event(e)

        def join():
            for st_i in streams + [h2d_stream, d2h_stream]:
                e = torch.cuda.Event()
                e.record(st_i)
                torch.cuda.current_stream().wait_event(e)

        def e2e_run(out_code, torch_dt):
            d_outs = [torch.empty(out.shape, dtype=torch_dt, device=dev) for _ in range(NB)]
            pos = [torch.empty(out.shape, dtype=torch_dt).pin_memory() for _ in range(NB)]
            inputs_free = [None] * NB                                  # events: kernels that read the set are done
            output_free = [None] * NB                                  # event: read-back of the set's output is done
            calls = [0]

            def e2e_step(i):
                b_i = i % NB
                dq, dk, dv = in_sets[b_i]
                kernels_done = []
                for bb in range(cfg.B):
                    st_i = streams[calls[0] % len(streams)]
                    with torch.cuda.stream(h2d_stream):
                        if bb == 0 and inputs_free[b_i] is not None:
                            for e in inputs_free[b_i]:
                                h2d_stream.wait_event(e)
                        dq[bb:bb + 1].copy_(pq[bb:bb + 1], non_blocking=True)
                        dk[bb:bb + 1].copy_(pk[bb:bb + 1], non_blocking=True)
                        dv[bb:bb + 1].copy_(pv[bb:bb + 1], non_blocking=True)
                        landed = torch.cuda.Event()
                        landed.record()
                    st_i.wait_event(landed)
                    if output_free[b_i] is not None:
                        st_i.wait_event(output_free[b_i])
                    with torch.cuda.stream(st_i):
                        hb.attention_fwd_raw(dq[bb:bb + 1], dk[bb:bb + 1], dv[bb:bb + 1], s, inv_s,
                                             cfg.causal, Bc=cfg.Bc, out_dtype=out_code, out=d_outs[b_i][bb:bb + 1],
                                             workspace=ws_s[calls[0] % len(streams)], d_status=status)
                        done = torch.cuda.Event()
                        done.record()
                    calls[0] += 1
                    kernels_done.append(done)
                    d2h_stream.wait_event(done)
                    with torch.cuda.stream(d2h_stream):
                        pos[b_i][bb:bb + 1].copy_(d_outs[b_i][bb:bb + 1], non_blocking=True)
                inputs_free[b_i] = kernels_done
                with torch.cuda.stream(d2h_stream):
                    e = torch.cuda.Event()
                    e.record()
                    output_free[b_i] = e

            fork()
            for i in range(4):
                e2e_step(i)
            join()
            barrier()
            for po in pos:
                po.zero_()
            a = torch.cuda.Event(enable_timing=True); b = torch.cuda.Event(enable_timing=True)
            n_e2e = max(4, min(args.steps, 50))                  # back-to-back steps: their copies and kernels pipeline
            a.record()
            fork()
            for i in range(n_e2e):
                e2e_step(i)
            join()
            b.record()
            barrier()
            assert int(status.item()) == 0, f"device status {int(status.item())}"
            # every host copy equals the device-resident result of the timed steps, rounded once to the output dtype
            for po in pos:
                assert torch.equal(po.to(dev), out.to(torch_dt)), "end-to-end output differs from the device result"
            e_ms = max_over_ranks(dist, a.elapsed_time(b), dev)
            h2d = (pq.numel() + pk.numel() + pv.numel()) * pq.element_size()
            return {"value": whole_job_tflops(cfg, world, n_e2e, e_ms), "unit": UNIT,
                    "h2d_bytes_per_step": h2d, "d2h_bytes_per_step": pos[0].numel() * pos[0].element_size(),
                    "ms_per_step": e_ms / n_e2e, "steps": n_e2e, "out_dtype": str(torch_dt).replace("torch.", ""),
                    "how": f"hifa4_attention_fwd_raw per batch element ({cfg.B} per step), {NB} sets of device buffers used "
                           f"by alternate steps, {len(streams)} kernel streams and two copy streams tied by events, pinned "
                           "host buffers; back-to-back steps pipeline"}

        e2e_f32 = e2e_run(hb.F32, torch.float32)
        e2e = e2e_run(hb.F16, torch.float16)

    # ---- context (not the product): torch SDPA in BF16 on the same inputs, and, for the headline
    # workload, its N = 8192 sibling (the target sentence names an 8K prefill, the configuration 4K)
    context = {}
    if rank == 0 and not args.no_context:
        import torch.nn.functional as F
        try:
            qb, kb, vb = (t.to(torch.bfloat16) for t in (q, k, v))
            for _ in range(3):
                F.scaled_dot_product_attention(qb, kb, vb, is_causal=cfg.causal, enable_gqa=True)
            torch.cuda.synchronize()
            a = torch.cuda.Event(enable_timing=True); b = torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(10):
                F.scaled_dot_product_attention(qb, kb, vb, is_causal=cfg.causal, enable_gqa=True)
            b.record()
            torch.cuda.synchronize()
            context["torch_sdpa_bf16_tflops"] = attn_flops(cfg) * 10 / (a.elapsed_time(b) * 1e-3) / 1e12
        except Exception as e:                                         # context only: never fail the bench on it
            context["torch_sdpa_bf16_tflops"] = None
            context["torch_sdpa_error"] = str(e)[:120]
        assert int(status.item()) == 0

    # ---- sweep (rank 0, headline run only): every other configuration and the variants, each timed on the
    # device like the headline (events around each step, L2 flushed between steps), under the same clock record
    sweep, gemm, sweep_clocks = None, None, None
    headline = cfg.name == synth.CONFIGS["C2"].name and cfg.N == 4096 and cfg.causal and cfg.Bc == 64 \
        and not args.qmean and not args.p_f32 and not args.f8qk
    if rank == 0 and headline and not args.no_sweep:
        gemm = measure_gemm_peaks(dev)
        del out
        sweep = {}
        sweep_sampler = ClockSampler(local_rank)
        sweep_sampler.start()
        sweep_sampler.mark_begin()

        def cal(c):
            if not c.smooth_mode:
                return None, None
            qc_, kc_ = synth.make_calibration(c, samples=min(c.cal_samples, 4), tokens=min(c.cal_tokens, 256))
            return hb.smooth_calibrate(qc_.to(dev), kc_.to(dev), c.smooth_mode)

        entries = [("C1", synth.config("C1"), {}),
                   ("C2@8192 causal (the shape the target sentence names)", synth.config("C2", N=8192), {}),
                   ("C2 non-causal", synth.config("C2", causal=False), {}),
                   ("C2 Bc=128", synth.config("C2", Bc=128), {}),
                   ("C2 Q-Mean", synth.config("C2"), {"qmean": True}),
                   ("C2 FP32-P variant", synth.config("C2"), {"p_f32": True}),
                   ("C2 Q K^T as kind::f8f6f4 with split accumulators (experiment; incl. 2 operand-image launches)",
                    synth.config("C2"), {"f8qk": True}),
                   ("C2 Q quantized inside the attention kernel", synth.config("C2"), {"fused_q": True}),
                   ("C2@8192 Q quantized inside the attention kernel", synth.config("C2", N=8192), {"fused_q": True}),
                   ("C3", synth.config("C3"), {}), ("C4", synth.config("C4"), {})]
        for n_ in (1024, 2048, 4096, 8192, 16384, 32768):
            entries.append((f"C5@{n_} causal", synth.config("C5", N=n_), {}))
            entries.append((f"C5@{n_} non-causal", synth.config("C5", N=n_, causal=False), {}))
        for label, c, kw in entries:
            big_c = c.N >= 16384
            s_c, is_c = cal(c)
            r = time_workload(hb, c, dev, steps=3 if big_c else 8, warmup=3, flush_l2=flush_l2, s=s_c, inv_s=is_c, **kw)
            r["frac_of_measured_bf16_peak"] = r["attention_tflops"] / measured_peaks()["bf16"]
            sweep[label] = {k_: (round(v_, 5) if isinstance(v_, float) else v_) for k_, v_ in r.items()}
            torch.cuda.empty_cache()
        sweep_sampler.mark_end()
        sweep_clocks = sweep_sampler.stop()
        sweep_clocks["window"] = "the whole sweep"
        assert int(status.item()) == 0

    if rank != 0:
        if dist is not None:
            dist.destroy_process_group()
        return

    peaks = measured_peaks()
    fl = attn_flops(cfg)
    value = whole_job_tflops(cfg, world, args.steps, total_ms)
    attn_avg_ms = sum(attn_ms) / len(attn_ms)
    achieved = fl / (attn_avg_ms * 1e-3) / 1e12
    kern = attention_kernel(cfg, p_f32=args.p_f32, qmean=args.qmean, f8qk=args.f8qk,
                            sms=torch.cuda.get_device_properties(dev).multi_processor_count)
    frac_measured = {"bf16_driver_measured": achieved / peaks["bf16"]}
    if gemm:
        if gemm.get("bf16_tflops"):
            frac_measured["bf16_this_run"] = achieved / gemm["bf16_tflops"]
            frac_measured["fp4_as_4x_bf16_this_run"] = achieved / (4 * gemm["bf16_tflops"])
        if gemm.get("fp8_tflops"):
            frac_measured["fp8_this_run"] = achieved / gemm["fp8_tflops"]
        if gemm.get("fp4_tflops"):
            frac_measured["fp4_this_run"] = achieved / gemm["fp4_tflops"]
    roofline = {"bound": "tensor", "kernel": kern, "achieved": achieved, "peak": peaks["bf16"],
                "unit": "TFLOP/s", "frac": achieved / peaks["bf16"], "frac_of_measured": frac_measured,
                "traffic": NCU_TRAFFIC_BYTES.get((cfg.name, cfg.Bc) if cfg.causal and not args.p_f32 and not args.qmean else None),
                "peak_source": f"{peaks['source']} cuBLAS bf16 burst (the MMA kind issued is kind::f16 on BF16 images)",
                "avg_launch_ms": attn_avg_ms,
                "timed_in": "a second pass of the same steps with one event between the two launches "
                            f"({split_step_ms:.4f} ms per step there)",
                "frac_of_nominal": {k_: achieved / v_ for k_, v_ in NOMINAL.items()}}
    # The binding resource of the attention kernel is the instruction issue of its softmax/quantizer warps, not
    # the tensor pipe.  Roofline on it: scores per second against (SMs x 4 schedulers x clock x 32 lanes) divided
    # by the issue slots the METHOD needs per score (ALGORITHMIC_SLOTS_PER_SCORE above).  Beside it, as a separate
    # figure, the issue-slot utilisation: the same rate against the warp instructions the kernel actually executes
    # per 32 scores (ncu opcode counters, polling loops included).
    n_scores = cfg.B * cfg.Hq * sum(min(cfg.N, ((qb * 128 + 127) // cfg.Bc + 1) * cfg.Bc) if cfg.causal else cfg.N
                                    for qb in range((cfg.N + 127) // 128)) * 128
    sm_count = torch.cuda.get_device_properties(dev).multi_processor_count
    sm_hz = (clocks.get("sm_mhz") or 1965.0) * 1e6
    ach_scores = n_scores / (attn_avg_ms * 1e-3)
    peak_scores = sm_count * 4 * sm_hz * 32 / ALGORITHMIC_SLOTS_PER_SCORE
    roofline_alu = {"bound": "alu", "kernel": kern, "achieved": ach_scores / 1e9, "peak": peak_scores / 1e9,
                    "unit": "Gscore/s", "frac": ach_scores / peak_scores,
                    "algorithmic_issue_slots_per_score": ALGORITHMIC_SLOTS_PER_SCORE,
                    "peak_source": f"{sm_count} SMs x 4 schedulers x {sm_hz / 1e6:.0f} MHz (sampled) x 32 lanes / "
                                   f"{ALGORITHMIC_SLOTS_PER_SCORE} issue slots per score the method needs"}
    instr_per_warp_score = NCU_INSTR_PER_WARP_SCORE.get(kern)
    if instr_per_warp_score:
        roofline_alu["issue_slot_utilisation"] = ach_scores * instr_per_warp_score / (sm_count * 4 * sm_hz * 32)
        roofline_alu["executed_instr_per_warp_score"] = instr_per_warp_score
    q_bytes = sum(t.numel() for t in (q, k, v)) * (2 + 0.5625)
    quant = {"avg_ms": sum(quant_ms) / len(quant_ms), "algorithmic_gbs": q_bytes / (sum(quant_ms) / len(quant_ms) * 1e-3) / 1e9,
             "hbm_peak_gbs": peaks["hbm"]}

    cpu = None
    if not args.no_cpu_baseline and not big:
        from oracle import hifa4_oracle as orc
        orc.build()
        qn, kn, vn = (t.float().numpy() for t in (qh, kh, vh))
        sn = None if s is None else s.cpu().numpy()
        isn = None if inv_s is None else inv_s.cpu().numpy()
        t1, cores = oracle_time(cfg, qn, kn, vn, sn, isn, [0])
        n_heads = max(1, min(cfg.Hq - 1, int(12.0 / max(t1, 1e-3))))
        heads = [1 + int(i * (cfg.Hq - 1) / n_heads) for i in range(n_heads)]
        t, cores = oracle_time(cfg, qn, kn, vn, sn, isn, heads)
        cpu = {"value": n_heads * head_flops(cfg) / t / 1e12, "unit": UNIT, "cores": cores, "kind": "oracle",
               "sample": f"{n_heads} of {cfg.B * cfg.Hq} (batch, head) slices of {cfg.name}, all {cfg.N} rows each, "
                         f"{t:.1f} s"}

    line = {"metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": total_ms / args.steps, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "bf16", "data": "synthetic",
            "config": config_dict(cfg, args, world),
            "frac_of_nominal_peak": {k_: value / world / v_ for k_, v_ in NOMINAL.items()},
            "clocks": clocks, "e2e": e2e, "e2e_f32_out": e2e_f32, "gpu_launches": launches, "roofline": roofline,
            "roofline_alu": roofline_alu, "quantize": quant, "cpu_baseline": cpu, "context": context,
            "measured_gemm_peaks_this_run": gemm, "sweep": sweep, "sweep_clocks": sweep_clocks}
    print(json.dumps(line), flush=True)
    if dist is not None:
        dist.destroy_process_group()


if __name__ == "__main__":
    main()
