#!/usr/bin/env python3
"""Benchmark: prefill-only KV selection throughput on GB300.

One step = one mmshift_select call over every layer of the workload (proxies,
two-pass proxy softmax with group-mass aggregation, coverage vote, budgeted
top-k, gather), inputs resident in HBM. Default workload: the 28-layer
Qwen2.5-VL-7B-shaped long-context stack (T = 32768 = 4 images x 8064 visual +
512 text tokens, Hq/Hkv = 28/4, d = 128, bf16, window 32, budget 2048) with the
paper's hyper-parameters (N = 512 proxies, G = 32, gamma = 10, tau = 0.95,
lambda = 1).

Metric: prompt tokens selected per second per layer (sum_b T_b * L / step
time), whole job over all ranks; plus the fraction of the HBM roofline the
step's algorithmic bytes (K read once + K/V gathered, read and written) reach.

--stats prefill takes the proxies' statistics over every prompt query instead
of the window's (Section 3.2.1): each step then also reads the L x T x Hq x d
prompt queries once (mmshift_prefill_stats) and selects with
mmshift_select_with_stats; the line adds that pass's HBM roofline.
--stats hidden builds the proxies the paper's way: statistics over the prefill
hidden states (d_model = Hq x d = 3584 features per token, 6.6 GB per step),
N proxy hidden states projected by a resident W_Q on the tensor cores
(mmshift_hidden_stats + mmshift_build_hidden_proxies), then mmshift_select
with those proxies; the line adds the statistics pass's HBM roofline and the
projection's tensor roofline.

After the timed steps the line reports the attention-mass coverage (Fig. 1b)
of the kept set for 32 synthetic decode queries per (layer, request), next to
that of the most recent tokens under the same budget (--coverage N; 0 skips).

--impl reference times the CPU oracle on the host cores instead (a bounded
sample of the same workload per step).

Multi-GPU (torchrun): every rank runs its own replica of the workload (units
are independent: no data-path collective); value sums all ranks' tokens over
the slowest rank's time.
"""
from __future__ import annotations

import argparse
import json
import math
import multiprocessing as mp
import os
import statistics
import subprocess
import sys
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

from paper_2607_22586_gb300 import synth as S  # noqa: E402

METRIC = "prompt tokens selected/sec per layer + % of GB300 HBM roofline (bytes read/time)"
SFU_EX2_PER_SM_CLK = 32          # MUFU.EX2 lanes per SM per clock on GB300 (measured ~31)

# DRAM traffic (read + write) of the two scoring kernels per launch of the
# default workload: one ncu capture of a 4-layer slice (one kernel launch each),
# scaled by 7 to the 28 layers (the passes' units grow in proportion to the
# layers; read per launch, of K's bytes: softmax pass 1.17x, mass pass 1.22x in
# the slice). It describes only the score_umma.cu it was measured on (checked by
# hash).
SCORE_TRAFFIC = {"source_sha256_16": "5acdcb67c02668ad", "workload": "qwen7b-28l-32k",
                 "proxies": "paper", "softmax_pass": 7 * (156.355328e6 + 42.547712e6),
                 "mass_pass": 7 * (163.975680e6 + 55.691008e6)}
# DRAM traffic of the prompt-query statistics pass (both kernels) per launch
# of the default workload, from one ncu capture of a 4-layer slice scaled by 7
# (partial kernel 939.564544 MB read + 9.113856 MB written, merge 11.026176 MB
# read); valid for the stats.cu it was measured on (checked by hash).
STATS_TRAFFIC = {"source_sha256_16": "4e41aed56a87fda0", "workload": "qwen7b-28l-32k",
                 "bytes": 7 * (939.564544e6 + 9.113856e6 + 11.026176e6)}
UNIT = "tokens/s/layer"
SM_COUNT = 152
FP32_LANES_PER_SM = 128


def _gen_one(args):
    wl, layer = args
    li = S.make_layer(wl, layer)
    return li.native(wl.dtype)


def gen_workload(wl, rank_seed: int, procs: int):
    """All layers of wl as stacked native arrays (K, V, Qwin), seeded."""
    wl = wl.replace(seed=wl.seed + rank_seed)
    jobs = [(wl, l) for l in range(wl.n_layers)]
    if procs > 1 and wl.n_layers > 1:
        with mp.get_context("spawn").Pool(procs) as pool:
            parts = pool.map(_gen_one, jobs)
    else:
        parts = [_gen_one(j) for j in jobs]
    return tuple(np.stack([p[i] for p in parts]) for i in range(3))


def prompt_queries_device(wl, K, Qwin, seed: int):
    """All prompt queries [L, T*Hq*d] on the device for --stats prefill, with
    the recipe of synth.make_prompt_queries (half the request's per-head key
    mean plus unit normal noise, a N(0, 1) modality offset per (head,
    dimension) on visual positions, the window queries as the last rows),
    drawn by torch's seeded device generator: the 28 x 32K x 28 x 128 stack
    is 6.6 GB, too large to draw on the host every run."""
    import torch
    L, T = wl.n_layers, wl.total_tokens
    hq, hkv, d, w = wl.n_q_heads, wl.n_kv_heads, wl.head_dim, wl.window
    g = torch.Generator(device=K.device).manual_seed(seed)
    out = torch.empty((L, T, hq, d), dtype=K.dtype, device=K.device)
    cu = wl.cu_seqlens()
    Kv = K.view(L, T, hkv, d)
    Qv = Qwin.view(L, wl.batch, w, hq, d)
    for l in range(L):
        for b, (t_len, n_vis) in enumerate(zip(wl.seq_lens, wl.n_visual)):
            lo, hi = int(cu[b]), int(cu[b + 1])
            kmean = Kv[l, lo:hi].float().mean(dim=0).repeat_interleave(hq // hkv, dim=0)
            q = torch.randn((t_len, hq, d), generator=g, device=K.device) + 0.5 * kmean
            q[:n_vis] += torch.randn((hq, d), generator=g, device=K.device)
            out[l, lo:hi] = q.to(K.dtype)
            nw = min(w, t_len)
            out[l, hi - nw:hi] = Qv[l, b, w - nw:]
    return out.view(L, -1)


def hidden_states_device(wl, d_model: int, seed: int, device):
    """Prefill hidden states [L, T*d_model] on the device for --stats hidden,
    with the recipe of synth.make_hidden_states (per-feature mean N(0, 0.5^2)
    with four massive features at +-20, scale U(0.5, 1.5), a 0.5 N(0, 1)
    modality offset on visual positions, unit noise), drawn by torch's seeded
    device generator."""
    import torch
    L, T = wl.n_layers, wl.total_tokens
    g = torch.Generator(device=device).manual_seed(seed)
    out = torch.empty((L, T, d_model), dtype=torch.bfloat16, device=device)
    cu = wl.cu_seqlens()
    for l in range(L):
        mean = torch.randn(d_model, generator=g, device=device) * 0.5
        scale = torch.rand(d_model, generator=g, device=device) + 0.5
        massive = torch.randperm(d_model, generator=g, device=device)[:4]
        mean[massive] = 20.0 * torch.sign(torch.randn(4, generator=g, device=device))
        for b, (t_len, n_vis) in enumerate(zip(wl.seq_lens, wl.n_visual)):
            h = mean + scale * torch.randn((t_len, d_model), generator=g, device=device)
            h[:n_vis] += 0.5 * torch.randn(d_model, generator=g, device=device)
            out[l, int(cu[b]):int(cu[b + 1])] = h.to(torch.bfloat16)
    return out.view(L, -1)


def query_projection_device(wl, d_model: int, seed: int, device):
    """W_Q [L, Hq*d, d_model] with N(0, 1/d_model) entries and a bias
    [L, Hq*d] N(0, 0.5^2), bf16, as synth.make_query_projection: model weights,
    resident on the device (not per-step inputs)."""
    import torch
    f = wl.n_q_heads * wl.head_dim
    g = torch.Generator(device=device).manual_seed(seed)
    w = (torch.randn((wl.n_layers, f, d_model), generator=g, device=device) / math.sqrt(d_model))
    bias = torch.randn((wl.n_layers, f), generator=g, device=device) * 0.5
    return w.to(torch.bfloat16), bias.to(torch.bfloat16)


def decode_queries_device(wl, K, n_dec: int, seed: int, spread: float = 1.5):
    """Synthetic decode queries [L, B, Hq, n_dec, d] on the device with the
    recipe of synth.make_decode_queries (half the request's per-head key mean
    plus N(0, spread^2) noise), drawn by torch's seeded device generator."""
    import torch
    L, T = wl.n_layers, wl.total_tokens
    hq, hkv, d = wl.n_q_heads, wl.n_kv_heads, wl.head_dim
    g = torch.Generator(device=K.device).manual_seed(seed)
    out = torch.empty((L, wl.batch, hq, n_dec, d), dtype=K.dtype, device=K.device)
    cu = wl.cu_seqlens()
    Kv = K.view(L, T, hkv, d)
    for l in range(L):
        for b in range(wl.batch):
            kmean = Kv[l, int(cu[b]):int(cu[b + 1])].float().mean(dim=0).repeat_interleave(hq // hkv, dim=0)
            q = 0.5 * kmean[:, None, :] + spread * torch.randn((hq, n_dec, d), generator=g, device=K.device)
            out[l, b] = q.to(K.dtype)
    return out


def measure_coverage(args, wl, shape, K, Q, out_idx, stream, seed, M, tpeak, tkind):
    """Attention-mass coverage (Fig. 1b) of the step's kept set for
    args.coverage synthetic decode queries per (layer, request), next to the
    coverage of the most recent min(C_b, T_b) tokens (a StreamingLLM-like
    window without sinks), both through mmshift_coverage; plus the time of
    one coverage call."""
    import torch
    n_dec = args.coverage
    dec = decode_queries_device(wl, K, n_dec, seed)
    nb = M.mmshift_coverage_workspace_size(shape, n_dec)
    ws = torch.zeros(nb, dtype=torch.uint8, device=K.device)
    L = wl.n_layers
    cov = torch.empty((L, wl.batch, wl.n_kv_heads, n_dec), device=K.device)
    recent = torch.empty_like(out_idx)
    off = 0
    for t_len, c in zip(wl.seq_lens, wl.budgets):
        keep = min(c, t_len)
        recent[:, off:off + keep, :] = torch.arange(t_len - keep, t_len, dtype=torch.int32,
                                                    device=K.device)[None, :, None]
        off += keep

    def run(idx, out):
        M.check(M.mmshift_coverage(shape, K, Q, dec, n_dec, 0.0, idx, out, ws, nb, stream),
                "mmshift_coverage")

    run(out_idx, cov)
    cov_recent = torch.empty_like(cov)
    run(recent, cov_recent)
    M.check(M.mmshift_poll_status(ws, stream), "coverage status")
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record(stream)
    for _ in range(3):
        run(out_idx, cov)
    e1.record(stream)
    torch.cuda.synchronize()
    ms = e0.elapsed_time(e1) / 3
    c = cov.flatten().double().cpu().numpy()
    cr = cov_recent.flatten().double().cpu().numpy()
    # the logits of every prompt key and of the kept keys: 2 d flops per (decode
    # query, query head, key)
    kept = sum(min(t, c) for t, c in zip(wl.seq_lens, wl.budgets))
    flops = 2.0 * wl.head_dim * n_dec * wl.n_q_heads * (wl.total_tokens + kept) * L
    ach = flops / (ms * 1e-3) / 1e12
    return {"n_decode_queries": n_dec, "queries": "0.5 * per-head key mean + N(0, 1.5^2), synthetic",
            "mean": float(c.mean()), "p10": float(np.percentile(c, 10)), "min": float(c.min()),
            "recent_window_mean": float(cr.mean()), "recent_window_p10": float(np.percentile(cr, 10)),
            "ms_per_call": ms,
            "roofline": {"bound": "tensor", "achieved": ach, "peak": tpeak, "unit": "TFLOP/s",
                         "frac": ach / tpeak, "traffic": None, "peak_kind": tkind,
                         "kernel": "whole mmshift_coverage call (pack, copy of the kept rows, softmax "
                                   "pass over the prompt and over the copied rows, ratio)",
                         "note": "algorithmic flops of the decode queries only; the r * n_dec rows of a "
                                 "KV head are padded to blocks of 256"}}


class PreStep:
    """What runs before the selection when the proxies' statistics do not come
    from the window: --stats prefill (statistics over every prompt query, then
    mmshift_select_with_stats) or --stats hidden (statistics over the prefill
    hidden states, hidden-space proxies projected by W_Q, then mmshift_select
    with them). ``x`` is the per-step input (prompt queries or hidden states)."""

    def __init__(self, kind, wl, shape, params, K, Q, seed, d_model, M):
        import torch
        self.kind, self.wl, self.shape, self.params, self.M = kind, wl, shape, params, M
        dev = K.device
        L, B = wl.n_layers, wl.batch
        if kind == "prefill":
            self.x = prompt_queries_device(wl, K, Q, seed=seed)
            self.ncol = wl.n_q_heads * wl.head_dim
            self.ws_bytes = M.mmshift_prefill_stats_workspace_size(shape)
            self.stages = ["prefill_stats"]
            self.launches = 2
        else:
            self.dm = d_model
            self.x = hidden_states_device(wl, d_model, seed, dev)
            self.W, self.bias = query_projection_device(wl, d_model, seed + 1, dev)
            self.ncol = d_model
            self.ws_bytes = M.mmshift_hidden_stats_workspace_size(shape, d_model)
            self.hp_bytes = M.mmshift_hidden_proxies_workspace_size(shape, d_model, params)
            self.hws = torch.zeros(self.hp_bytes, dtype=torch.uint8, device=dev)
            self.px = torch.empty((L, B, wl.n_q_heads, params.n_proxies, wl.head_dim),
                                  dtype=torch.bfloat16, device=dev)
            self.stages = ["hidden_stats", "hidden_proxies"]
            self.launches = 4
        self.ws = torch.zeros(self.ws_bytes, dtype=torch.uint8, device=dev)
        self.stats = torch.empty((L, B, 2, self.ncol), device=dev)

    def run(self, x, stream, sev=None):
        """Launch the pre-selection steps on ``stream``; sev (nullable) gets
        an event before and after each. Returns the statistics (prefill) or
        the proxies (hidden) the selection takes."""
        M = self.M
        if sev:
            sev[0].record(stream)
        if self.kind == "prefill":
            M.check(M.mmshift_prefill_stats(self.shape, x, 0, self.stats, self.ws, self.ws_bytes,
                                            stream), "mmshift_prefill_stats")
            if sev:
                sev[1].record(stream)
            return self.stats
        M.check(M.mmshift_hidden_stats(self.shape, self.dm, x, 0, self.stats, self.ws, self.ws_bytes,
                                       stream), "mmshift_hidden_stats")
        if sev:
            sev[1].record(stream)
        M.check(M.mmshift_build_hidden_proxies(self.shape, self.dm, self.stats, self.W, 0, self.bias,
                                               None, self.params, self.px, self.hws, self.hp_bytes,
                                               stream), "mmshift_build_hidden_proxies")
        if sev:
            sev[2].record(stream)
        return self.px


def read_peaks():
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as f:
            return json.load(f), "measured"
    except OSError:
        return {"hbm_gbs": 6800.0, "bf16_tflops": 1900.0, "bf16_tflops_sustained": 1700.0,
                "sm_max_mhz": 2070.0}, "fallback"


def tensor_peak(peaks, clk, peak_src):
    """The bf16 dense peak that matches the clocks seen in the timed region:
    the burst figure (a GEMM timed alone, SM clock at its maximum) unless the
    median SM clock under load sat nearer the clock of the sustained,
    power-capped measurement. Returns (TFLOP/s, description)."""
    burst = float(peaks["bf16_tflops"])
    sust = float(peaks.get("bf16_tflops_sustained", burst))
    smax = float(peaks.get("sm_max_mhz", 2070.0))
    s_mhz = float((peaks.get("clocks_under_load") or {}).get("sm_mhz_median") or 0.0)
    med = clk.get("sm_mhz") if clk else None
    if med is not None and s_mhz and abs(med - s_mhz) < abs(med - smax):
        return sust, (f"bf16 dense, sustained ({peak_src}): median SM clock {med:.0f} MHz under "
                      f"load, nearer the sustained run's {s_mhz:.0f} MHz than the maximum {smax:.0f}")
    seen = f"median SM clock {med:.0f} MHz under load" if med is not None else "no clock record"
    return burst, f"bf16 dense, burst ({peak_src}): {seen}, maximum {smax:.0f} MHz"


def score_roofline(wl, hyper, stage_ms, umma, peaks, peak_src, clk, traffic=None):
    """Roofline of the slower scoring pass: tensor (bf16 tensor cores) with
    the MUFU exp2 rate beside it, or fp32 FMA on the CUDA-core path; the
    HBM view of the same kernel (K read once per pass) is added."""
    _, k_read, pass_flops = algorithmic(wl, hyper)
    dom = max(("softmax_pass", "mass_pass"), key=lambda s: stage_ms[s])
    dom_ms = stage_ms[dom]
    achieved = pass_flops / (dom_ms * 1e-3) / 1e12
    med = (clk or {}).get("sm_mhz") or float(peaks.get("sm_max_mhz", 2070.0))
    hbm = {"achieved": k_read / (dom_ms * 1e-3) / 1e9, "peak": peaks["hbm_gbs"], "unit": "GB/s",
           "frac": k_read / (dom_ms * 1e-3) / 1e9 / peaks["hbm_gbs"],
           "bytes_per_launch": k_read, "note": "K read once by the pass"}
    if umma:
        peak, kind = tensor_peak(peaks, clk, peak_src)
        sfu_peak = SFU_EX2_PER_SM_CLK * SM_COUNT * med * 1e6
        exps = pass_flops / (2.0 * wl.head_dim)          # one exp2 per logit
        return {"bound": "tensor", "achieved": achieved, "peak": peak, "unit": "TFLOP/s",
                "frac": achieved / peak, "traffic": traffic, "kernel": dom, "peak_kind": kind,
                "flops_per_launch": pass_flops, "ms_per_launch": dom_ms,
                "sfu": {"achieved": exps / (dom_ms * 1e-3), "peak": sfu_peak, "unit": "exp2/s",
                        "frac": exps / (dom_ms * 1e-3) / sfu_peak,
                        "peak_kind": f"{SFU_EX2_PER_SM_CLK} MUFU.EX2/clk/SM x {SM_COUNT} SMs x "
                                     f"{med:.0f} MHz (median SM clock under load)"},
                "hbm": hbm}
    peak = SM_COUNT * FP32_LANES_PER_SM * 2 * med * 1e6 / 1e12
    return {"bound": "alu", "achieved": achieved, "peak": peak, "unit": "TFLOP/s",
            "frac": achieved / peak, "traffic": None, "kernel": dom,
            "flops_per_launch": pass_flops, "ms_per_launch": dom_ms,
            "peak_kind": f"fp32 FMA: {SM_COUNT} SMs x {FP32_LANES_PER_SM} lanes x 2 flop x "
                         f"{med:.0f} MHz", "hbm": hbm}


class ClockSampler:
    """nvidia-smi clocks and throttle reasons sampled during the timed region."""

    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index: int):
        self.gpu = gpu_index
        self.proc = None

    def start(self):
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", f"--id={self.gpu}", f"--query-gpu={self.FIELDS}",
                 "--format=csv,noheader,nounits", "-lms", "200"],
                stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
        except OSError:
            self.proc = None

    def stop(self):
        if self.proc is None:
            return None
        self.proc.terminate()
        try:
            out, _ = self.proc.communicate(timeout=5)
        except subprocess.TimeoutExpired:
            self.proc.kill()
            out, _ = self.proc.communicate()
        sm, mx, reasons = [], 0.0, set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for line in out.splitlines():
            f = [x.strip() for x in line.split(",")]
            if len(f) < 9:
                continue
            try:
                sm.append(float(f[1]))
                mx = max(mx, float(f[2]))
            except ValueError:
                continue
            for n, v in zip(names, f[5:9]):
                if v.lower() == "active":
                    reasons.add(n)
        if not sm:
            return None
        load = [x for x in sm if x > 0.5 * max(sm)] or sm
        return {"sm_mhz": statistics.median(load), "sm_max_mhz": mx, "reasons": sorted(reasons),
                "samples": len(sm)}


def oracle_sample_rate(wl, K, V, Q, hyper, budget_s: float):
    """Run the oracle on (layer, KV head) units of the workload until about
    ``budget_s`` seconds of CPU work; return (tokens/s/layer, description)."""
    from oracle import mmshift_oracle as O
    r = wl.n_q_heads // wl.n_kv_heads
    cu = wl.cu_seqlens()
    done, spent, units = 0.0, 0.0, 0
    to_f = (lambda a: S.bf16_bits_to_f32(a)) if wl.dtype == S.BF16 else (lambda a: a)
    for layer in range(wl.n_layers):
        for h in range(wl.n_kv_heads):
            for b in range(wl.batch):
                lo, hi = int(cu[b]), int(cu[b + 1])
                k = to_f(K[layer, lo:hi, h:h + 1])
                v = to_f(V[layer, lo:hi, h:h + 1])
                q = to_f(Q[layer, b, :, h * r:(h + 1) * r])
                t0 = time.perf_counter()
                O.select_request(k, v, q, int(wl.budgets[b]), b=b, layer_id=layer, dtype=wl.dtype,
                                 **hyper)
                spent += time.perf_counter() - t0
                done += (hi - lo) / wl.n_kv_heads     # one head = 1/Hkv of a layer
                units += 1
                if spent >= budget_s:
                    return done / spent, f"{units} (layer, KV head, request) units of the workload"
    return done / spent, f"{units} (layer, KV head, request) units (whole workload)"


def blas_threads() -> int:
    try:
        from threadpoolctl import threadpool_info
        n = [i.get("num_threads", 1) for i in threadpool_info() if i.get("user_api") == "blas"]
        if n:
            return int(max(n))
    except Exception:
        pass
    return int(os.environ.get("OMP_NUM_THREADS", os.cpu_count() or 1))


def hyper_for(args, wl):
    if args.proxies == "few":
        n_p = wl.window
        return dict(n_proxies=n_p, n_groups=max(1, n_p // 16), gamma=10.0, tau=float(np.float32(0.95)),
                    lam=1.0, seed=0)
    return dict(n_proxies=512, n_groups=32, gamma=10.0, tau=float(np.float32(0.95)), lam=1.0, seed=0)


def pyramid_budgets(wl):
    """Per-(layer, KV head) budgets [L, B, Hkv] shaped like a pyramid
    allocation: layer l of L gets C * (1.5 - l / (L - 1)) (1.5 C at the
    bottom, C / 2 at the top, C on average), equal across heads."""
    L = wl.n_layers
    hb = np.empty((L, wl.batch, wl.n_kv_heads), dtype=np.int32)
    for l in range(L):
        f = 1.5 - (l / (L - 1) if L > 1 else 0.5)
        for b, c in enumerate(wl.budgets):
            hb[l, b, :] = max(1, int(round(c * f)))
    return hb


def algorithmic(wl, hyper, head_budgets=None):
    """Per step: HBM bytes (K read once + K/V gathered read+write) and the
    logits of one softmax pass (2 d flops per (proxy row, key))."""
    esz = 2 if wl.dtype == S.BF16 else 4
    L, hkv, d = wl.n_layers, wl.n_kv_heads, wl.head_dim
    T = wl.total_tokens
    k_read = L * T * hkv * d * esz
    if head_budgets is None:
        keep = sum(min(c, t) for c, t in zip(wl.budgets, wl.seq_lens))
        gather = 4 * L * keep * hkv * d * esz
    else:
        kept = sum(int(min(head_budgets[l, b, h], t)) for l in range(L)
                   for b, t in enumerate(wl.seq_lens) for h in range(hkv))
        gather = 4 * kept * d * esz
    r = wl.n_q_heads // hkv
    rows = hyper["n_proxies"] * r + r       # proxies of the r query heads + anchor rows
    pass_flops = 2.0 * d * rows * T * hkv * L
    return k_read + gather, k_read, pass_flops


def _source_digest(name):
    import hashlib
    try:
        with open(os.path.join(ROOT, "paper_2607_22586_gb300", "csrc", name), "rb") as f:
            return hashlib.sha256(f.read()).hexdigest()[:16]
    except OSError:
        return None


def stats_traffic(wl):
    """DRAM bytes per launch of the statistics pass from the recorded capture,
    or None if stats.cu or the workload differ from the captured ones."""
    t = STATS_TRAFFIC
    if _source_digest("stats.cu") != t["source_sha256_16"] or wl.name != t["workload"]:
        return None
    return t["bytes"]


def score_traffic(wl, args, kernel):
    """DRAM bytes per launch of a scoring kernel from the recorded capture, or
    None if the kernel source or the workload differ from the captured ones."""
    digest = _source_digest("score_umma.cu")
    t = SCORE_TRAFFIC
    if digest != t["source_sha256_16"] or wl.name != t["workload"] or args.proxies != t["proxies"]:
        return None
    return t.get(kernel)


def measure_select(wl, hyper, K, V, Q, steps, warmup, ranks, M, LB, dev):
    """Device-timed steps of one mmshift_select over every layer of ``wl``,
    inputs resident in HBM: W untimed steps, then K timed ones between CUDA
    events on the launching stream, barriers and synchronisation around them,
    nvidia-smi clocks sampled meanwhile. Returns (ms per step, max over ranks;
    mean stage times; kernel launches; scoring path; clock record)."""
    import torch
    L, T = wl.n_layers, wl.total_tokens
    shape = M.make_shape(wl.n_q_heads, wl.n_kv_heads, wl.head_dim, wl.window,
                         0 if wl.dtype == S.BF16 else 1, wl.cu_seqlens(), wl.budgets, n_layers=L,
                         layer_stride_kv=T * wl.n_kv_heads * wl.head_dim,
                         layer_stride_q=wl.batch * wl.window * wl.n_q_heads * wl.head_dim)
    params = M.default_params(n_proxies=hyper["n_proxies"], n_groups=hyper["n_groups"],
                              gamma=hyper["gamma"], tau=hyper["tau"], lam=hyper["lam"], seed=hyper["seed"])
    rows = M.mmshift_output_rows(shape)
    ws_bytes = M.mmshift_workspace_size(shape, params)
    ws = torch.zeros(ws_bytes, dtype=torch.uint8, device=dev)
    out_idx = torch.empty((L, rows, wl.n_kv_heads), dtype=torch.int32, device=dev)
    out_k = torch.empty((L, rows, wl.n_kv_heads, wl.head_dim), dtype=K.dtype, device=dev)
    out_v = torch.empty_like(out_k)
    stream = torch.cuda.current_stream(dev)

    def step(dbg=None):
        M.check(M.mmshift_select(shape, K, V, Q, None, params, out_idx, out_k, out_v, dbg, ws,
                                 ws_bytes, stream), "mmshift_select")

    for _ in range(warmup):
        step()
    M.check(M.mmshift_poll_status(ws, stream), "warm-up status")
    nst = LB.MMSHIFT_N_STAGES + 1
    stage_ev = [[torch.cuda.Event(enable_timing=True) for _ in range(nst)] for _ in range(steps)]
    for evs in stage_ev:
        for ev in evs:
            ev.record(stream)
    dbgs = [M.make_debug(stage_events=ev) for ev in stage_ev]
    clocks = ClockSampler(torch.cuda.current_device())
    clocks.start()
    time.sleep(0.3)
    torch.cuda.synchronize()
    ranks.barrier()
    # the timed steps record no events between the kernels (so each kernel's
    # launch overlaps the previous one's tail); the same number of steps
    # with stage events follows for the per-stage times
    t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    t0.record(stream)
    for k in range(steps):
        step()
    t1.record(stream)
    torch.cuda.synchronize()
    ranks.barrier()
    for k in range(steps):
        step(dbgs[k])
    torch.cuda.synchronize()
    clk = clocks.stop()
    M.check(M.mmshift_poll_status(ws, stream), "timed status")
    ms = ranks.max(t0.elapsed_time(t1) / steps, dev)
    stage_ms = {name: statistics.mean(ev[i].elapsed_time(ev[i + 1]) for ev in stage_ev)
                for i, name in enumerate(LB.STAGES)}
    return ms, stage_ms, dbgs[0].launches * steps, dbgs[0].score_path, clk


def sub_record(wl, proxies, K, V, Q, steps, warmup, ranks, M, LB, dev, peaks, peak_src, inputs):
    """One more workload / proxy setting timed in the same run (its own
    warm-up, timed steps and clock record), reported beside the headline."""
    hyper = hyper_for(argparse.Namespace(proxies=proxies), wl)
    ms, stage_ms, launches, path, clk = measure_select(wl, hyper, K, V, Q, steps, warmup, ranks, M,
                                                       LB, dev)
    bytes_step, _, _ = algorithmic(wl, hyper)
    return {"workload": wl.name, "proxies": proxies, "n_proxies": hyper["n_proxies"],
            "n_groups": hyper["n_groups"], "layers": wl.n_layers, "prompt_tokens": wl.total_tokens,
            "steps": steps, "warmup": warmup, "ms_per_step": ms,
            "value": job_value(wl.total_tokens * wl.n_layers, ranks.world, ms), "unit": UNIT,
            "hbm_bytes_per_step": bytes_step,
            "hbm_roofline_frac": bytes_step / (ms * 1e-3) / (peaks["hbm_gbs"] * 1e9),
            "stage_ms": stage_ms,
            "roofline": score_roofline(wl, hyper, stage_ms, path == 1, peaks, peak_src, clk),
            "clocks": clk, "gpu_launches": launches, "inputs": inputs}


def run_sub_records(args, wl, K, V, Q, ranks, M, LB, dev, peaks, peak_src):
    """The settings the HBM target is judged on, timed under the same clock
    as the headline: the 32K stack with few proxies (N = W), and the
    72B-class ragged batch (80 layers, eight requests) in both settings."""
    import torch
    recs = []
    if args.proxies == "paper":
        recs.append(sub_record(wl, "few", K, V, Q, args.steps, args.warmup, ranks, M, LB, dev, peaks,
                               peak_src, "the headline's inputs"))
    big = S.WORKLOADS["72b-80l-ragged"]
    t0 = time.perf_counter()
    Kh, Vh, Qh = gen_workload(big, ranks.rank, args.gen_procs)
    gen_s = time.perf_counter() - t0
    as_t = lambda a: torch.from_numpy(a.view(np.int16)).view(torch.bfloat16)
    K4, V4, Q4 = (as_t(a).to(dev) for a in (Kh, Vh, Qh))
    del Kh, Vh, Qh
    note = f"seeded synthetic, all 80 layers drawn on the host in {gen_s:.1f} s, resident in HBM"
    recs.append(sub_record(big, "paper", K4, V4, Q4, max(2, args.steps // 4), args.warmup, ranks, M,
                           LB, dev, peaks, peak_src, note))
    recs.append(sub_record(big, "few", K4, V4, Q4, args.steps, args.warmup, ranks, M, LB, dev, peaks,
                           peak_src, note))
    del K4, V4, Q4
    torch.cuda.empty_cache()
    return recs



class Ranks:
    """One process per GPU, as torchrun starts them (RANK, WORLD_SIZE,
    LOCAL_RANK, MASTER_ADDR / MASTER_PORT from the environment). With more
    than one rank a process group over ``backend`` is opened; every rank runs
    its own replica of the workload (no data-path collective), and only the
    timing uses the group: barriers around the timed region and the maximum of
    the per-rank times."""

    def __init__(self, backend: str):
        self.world = int(os.environ.get("WORLD_SIZE", "1"))
        self.rank = int(os.environ.get("RANK", "0"))
        self.local = int(os.environ.get("LOCAL_RANK", "0"))
        self.dist = None
        if self.world > 1:
            import torch.distributed as dist
            dist.init_process_group(backend)
            self.dist = dist

    def barrier(self):
        if self.dist:
            self.dist.barrier()

    def max(self, x: float, device=None) -> float:
        """Maximum of x over the ranks (x itself with one rank)."""
        if not self.dist:
            return float(x)
        import torch
        t = torch.tensor([float(x)], dtype=torch.float64, device=device)
        self.dist.all_reduce(t, op=self.dist.ReduceOp.MAX)
        return float(t.item())

    def close(self):
        if self.dist:
            self.dist.barrier()
            self.dist.destroy_process_group()
            self.dist = None


def job_value(tokens_per_rank: float, world: int, ms_max: float) -> float:
    """Whole-job throughput: the tokens every rank processed in one step over
    the slowest rank's step time."""
    return tokens_per_rank * world / (ms_max * 1e-3)


def run_reference(args, wl):
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return 0
    hyper = hyper_for(args, wl)
    # one layer of the workload is enough to sample from
    wl1 = wl.replace(n_layers=1)
    K, V, Q = gen_workload(wl1, 0, 1)
    for _ in range(args.warmup):
        oracle_sample_rate(wl1, K, V, Q, hyper, budget_s=0.0)
    rates, t0 = [], time.perf_counter()
    for _ in range(args.steps):
        rate, sample = oracle_sample_rate(wl1, K, V, Q, hyper, budget_s=args.ref_seconds)
        rates.append(rate)
    wall = time.perf_counter() - t0
    value = statistics.mean(rates)
    cores = blas_threads()
    line = {
        "impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": args.gpus,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1e3 * wall / args.steps,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
        "data": "synthetic (seeded, MLLM-shaped)",
        "config": {"workload": wl.name, "proxies": args.proxies, **{k: hyper[k] for k in ("n_proxies", "n_groups")}},
        "cpu_baseline": {"value": value, "unit": UNIT, "cores": cores, "kind": "oracle",
                         "sample": f"per step: {sample}; numpy float64 (BLAS matmul threads={cores}, "
                                   f"elementwise single-threaded)"},
        "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }
    print(json.dumps(line), flush=True)
    return 0


def run_gpu(args, wl):
    import torch
    import paper_2607_22586_gb300 as M
    from paper_2607_22586_gb300 import _lib as LB

    torch.cuda.set_device(int(os.environ.get("LOCAL_RANK", "0")))
    ranks = Ranks("nccl")
    world, rank = ranks.world, ranks.rank
    dev = torch.device("cuda", torch.cuda.current_device())
    hyper = hyper_for(args, wl)
    peaks, peak_src = read_peaks()

    # inputs: seeded on the host (replica r of the workload on rank r)
    t0 = time.perf_counter()
    Kh, Vh, Qh = gen_workload(wl, rank, args.gen_procs)
    gen_s = time.perf_counter() - t0
    tdt = torch.bfloat16 if wl.dtype == S.BF16 else torch.float32
    as_t = (lambda a: torch.from_numpy(a.view(np.int16)).view(torch.bfloat16)) if wl.dtype == S.BF16 \
        else (lambda a: torch.from_numpy(a))
    K_pin, V_pin, Q_pin = (as_t(a).pin_memory() for a in (Kh, Vh, Qh))
    K, V, Q = (t.to(dev) for t in (K_pin, V_pin, Q_pin))

    L = wl.n_layers
    T = wl.total_tokens
    hb_host = pyramid_budgets(wl) if args.head_budgets == "pyramid" else None
    capacity = wl.budgets if hb_host is None else tuple(int(hb_host[:, b].max())
                                                        for b in range(wl.batch))
    shape = M.make_shape(wl.n_q_heads, wl.n_kv_heads, wl.head_dim, wl.window,
                         0 if wl.dtype == S.BF16 else 1, wl.cu_seqlens(), capacity, n_layers=L,
                         layer_stride_kv=T * wl.n_kv_heads * wl.head_dim,
                         layer_stride_q=wl.batch * wl.window * wl.n_q_heads * wl.head_dim)
    params = M.default_params(n_proxies=hyper["n_proxies"], n_groups=hyper["n_groups"],
                              gamma=hyper["gamma"], tau=hyper["tau"], lam=hyper["lam"], seed=hyper["seed"])
    rows = M.mmshift_output_rows(shape)
    ws_bytes = M.mmshift_workspace_size(shape, params)
    ws = torch.zeros(ws_bytes, dtype=torch.uint8, device=dev)
    out_idx = torch.empty((L, rows, wl.n_kv_heads), dtype=torch.int32, device=dev)
    out_k = torch.empty((L, rows, wl.n_kv_heads, wl.head_dim), dtype=tdt, device=dev)
    out_v = torch.empty_like(out_k)
    stream = torch.cuda.current_stream(dev)
    nst = LB.MMSHIFT_N_STAGES + 1
    d_model = args.d_model or wl.n_q_heads * wl.head_dim
    pre = None
    if args.stats != "window":
        pre = PreStep(args.stats, wl, shape, params, K, Q, wl.seed + 7919 * (rank + 1), d_model, M)

    hb_dev = torch.from_numpy(hb_host).to(dev) if hb_host is not None else None

    def select(Kx, Vx, Qx, Xx, dbg=None, sev=None, outs=None):
        oi, ok, ov = outs if outs is not None else (out_idx, out_k, out_v)
        if hb_dev is not None:
            M.check(M.mmshift_select_head_budgets(shape, Kx, Vx, Qx, None, hb_dev, params, oi,
                                                  None, ok, ov, dbg, ws, ws_bytes, stream),
                    "mmshift_select_head_budgets")
        elif pre is None:
            M.check(M.mmshift_select(shape, Kx, Vx, Qx, None, params, oi, ok, ov, dbg,
                                     ws, ws_bytes, stream), "mmshift_select")
        elif pre.kind == "prefill":
            st = pre.run(Xx, stream, sev)
            M.check(M.mmshift_select_with_stats(shape, Kx, Vx, Qx, st, params, oi, ok, ov,
                                                dbg, ws, ws_bytes, stream), "mmshift_select_with_stats")
        else:
            px = pre.run(Xx, stream, sev)
            M.check(M.mmshift_select(shape, Kx, Vx, Qx, px, params, oi, ok, ov, dbg,
                                     ws, ws_bytes, stream), "mmshift_select")

    def step(dbg=None, sev=None):
        select(K, V, Q, pre.x if pre else None, dbg, sev)

    for _ in range(args.warmup):
        step()
    M.check(M.mmshift_poll_status(ws, stream), "warm-up status")

    # device-timed steps: inputs resident in HBM and larger than L2
    stage_ev = [[torch.cuda.Event(enable_timing=True) for _ in range(nst)] for _ in range(args.steps)]
    for evs in stage_ev:          # torch creates the CUDA event on first record
        for ev in evs:
            ev.record(stream)
    dbgs = [M.make_debug(stage_events=ev) for ev in stage_ev]
    stat_ev = [[torch.cuda.Event(enable_timing=True) for _ in range(len(pre.stages) + 1)] if pre else None
               for _ in range(args.steps)]
    clocks = ClockSampler(torch.cuda.current_device())
    clocks.start()
    time.sleep(0.3)
    torch.cuda.synchronize()
    ranks.barrier()
    # the timed steps record no events between the kernels (so each kernel's
    # launch overlaps the previous one's tail); the same number of steps
    # with stage events follows for the per-stage times
    t_start, t_end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    t_start.record(stream)
    for k in range(args.steps):
        step()
    t_end.record(stream)
    torch.cuda.synchronize()
    ranks.barrier()
    for k in range(args.steps):
        step(dbgs[k], stat_ev[k])
    torch.cuda.synchronize()
    clk = clocks.stop()
    M.check(M.mmshift_poll_status(ws, stream), "timed status")
    ms = ranks.max(t_start.elapsed_time(t_end) / args.steps, dev)
    stage_ms = {name: statistics.mean(ev[i].elapsed_time(ev[i + 1]) for ev in stage_ev)
                for i, name in enumerate(LB.STAGES)}
    launches = dbgs[0].launches * args.steps
    if pre:
        stage_ms = {**{name: statistics.mean(e[i].elapsed_time(e[i + 1]) for e in stat_ev)
                       for i, name in enumerate(pre.stages)}, **stage_ms}
        launches += pre.launches * args.steps

    # end to end through the same C ABI call: host buffers in, results out
    idx_h = torch.empty(out_idx.shape, dtype=out_idx.dtype, pin_memory=True)
    ok_h = torch.empty(out_k.shape, dtype=out_k.dtype, pin_memory=True)
    ov_h = torch.empty_like(ok_h, pin_memory=True)
    e_steps = max(1, args.steps)
    # Every step copies its inputs from pinned host memory and reads its
    # results back. K, Qwin (and the prompt queries / hidden states of
    # --stats) are double-buffered on the device, so their copies for step
    # k+1 (on a copy stream) overlap the selection of step k; a buffer is
    # refilled only after the selection that read it. V stays in pinned host
    # memory: the gather reads only the kept rows across the host link. The
    # outputs are double-buffered too and copied back on the copy stream.
    Kb, Qb = [K, torch.empty_like(K)], [Q, torch.empty_like(Q)]
    outs = [(out_idx, out_k, out_v),
            (torch.empty_like(out_idx), torch.empty_like(out_k), torch.empty_like(out_v))]
    if pre:
        X_pin = torch.empty(pre.x.shape, dtype=pre.x.dtype, pin_memory=True)
        X_pin.copy_(pre.x)
        Xb = [pre.x, torch.empty_like(pre.x)]
    cstream = torch.cuda.Stream(dev)
    ready = [torch.cuda.Event() for _ in range(2)]
    free = [torch.cuda.Event() for _ in range(2)]
    done = [torch.cuda.Event() for _ in range(2)]
    drained = [torch.cuda.Event() for _ in range(2)]

    def copy_in(i):
        cstream.wait_event(free[i])
        with torch.cuda.stream(cstream):
            Kb[i].copy_(K_pin, non_blocking=True)
            Qb[i].copy_(Q_pin, non_blocking=True)
            if pre:
                Xb[i].copy_(X_pin, non_blocking=True)
        ready[i].record(cstream)

    def select_out(i):
        stream.wait_event(ready[i])
        stream.wait_event(drained[i])
        select(Kb[i], V_pin, Qb[i], Xb[i] if pre else None, outs=outs[i])
        free[i].record(stream)
        done[i].record(stream)

    def copy_out(i):
        cstream.wait_event(done[i])
        with torch.cuda.stream(cstream):
            idx_h.copy_(outs[i][0], non_blocking=True)
            ok_h.copy_(outs[i][1], non_blocking=True)
            ov_h.copy_(outs[i][2], non_blocking=True)
        drained[i].record(cstream)

    def e2e(nsteps):
        for ev in free + drained:
            ev.record(stream)
        copy_in(0)
        for k in range(nsteps):
            if k + 1 < nsteps:
                copy_in((k + 1) % 2)
            select_out(k % 2)
            copy_out(k % 2)
        stream.wait_stream(cstream)     # the last results are on the host

    e2e(2)                        # untimed warm-up of the pinned host buffers and streams
    torch.cuda.synchronize()
    # three back-to-back trials of e_steps steps each: the host link is shared
    # with the other GPU on the host, so one trial can read far slower than
    # the next; the median is reported, every trial is listed
    e_trials = []
    for _ in range(3):
        ranks.barrier()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        e2e(e_steps)
        e1.record(stream)
        torch.cuda.synchronize()
        e_trials.append(ranks.max(e0.elapsed_time(e1) / e_steps, dev))
    e_ms = statistics.median(e_trials)
    # K, Qwin (and X) copied, plus the kept V rows the gather reads from host memory
    kept_rows = int(out_idx.numel())
    h2d = sum(t.numel() * t.element_size() for t in (K_pin, Q_pin)) + kept_rows * wl.head_dim * \
        V_pin.element_size()
    if pre:
        h2d += X_pin.numel() * X_pin.element_size()
    d2h = sum(t.numel() * t.element_size() for t in (idx_h, ok_h, ov_h))

    bytes_step, k_read, pass_flops = algorithmic(wl, hyper, hb_host)
    extra_roofs = {}
    if pre:
        # algorithmic bytes of the statistics pass: every prompt query (or
        # hidden state) read once, the [L, B, 2, ncol] float32 statistics written
        x_bytes = pre.x.numel() * pre.x.element_size()
        s_bytes = x_bytes + pre.stats.numel() * 4
        bytes_step += x_bytes
        st_ms = stage_ms[pre.stages[0]]
        ach = s_bytes / (st_ms * 1e-3) / 1e9
        extra_roofs[pre.stages[0] + "_roofline"] = {
            "bound": "hbm", "achieved": ach, "peak": peaks["hbm_gbs"], "unit": "GB/s",
            "frac": ach / peaks["hbm_gbs"],
            "traffic": stats_traffic(wl) if pre.kind == "prefill" else None,
            "kernel": "stats_partial_kernel + stats_merge_kernel",
            "bytes_per_launch": s_bytes, "peak_kind": f"HBM copy ({peak_src})"}
        if pre.kind == "hidden":
            # the projection: 2 * N * d_model * Hq*d flops per (layer, request);
            # the stage also holds the sampling kernel
            f_ms = stage_ms["hidden_proxies"]
            flops = 2.0 * hyper["n_proxies"] * d_model * wl.n_q_heads * wl.head_dim * L * wl.batch
            tpeak, tkind = tensor_peak(peaks, clk, peak_src)
            ach = flops / (f_ms * 1e-3) / 1e12
            extra_roofs["hidden_proxies_roofline"] = {
                "bound": "tensor", "achieved": ach, "peak": tpeak, "unit": "TFLOP/s",
                "frac": ach / tpeak, "traffic": None,
                "kernel": "hidden_sample_kernel + hidden_proj_pair_kernel",
                "flops_per_launch": flops, "peak_kind": tkind}
    tokens_layer = T * L * world          # metric unit: tokens per second per layer
    value = job_value(T * L, world, ms)
    hbm_frac = bytes_step / (ms * 1e-3) / (peaks["hbm_gbs"] * 1e9)

    # dominant stage and its roofline
    dom = max(("softmax_pass", "mass_pass"), key=lambda s: stage_ms[s])
    umma = dbgs[0].score_path == 1
    roof = score_roofline(wl, hyper, stage_ms, umma, peaks, peak_src, clk,
                          score_traffic(wl, args, dom) if umma else None)
    tpeak, tkind = tensor_peak(peaks, clk, peak_src)

    coverage = None
    if args.coverage:
        coverage = measure_coverage(args, wl, shape, K, Q, out_idx, stream, wl.seed + 104729 * (rank + 1), M,
                                    tpeak, tkind)

    cpu = None
    if rank == 0 and args.cpu_seconds > 0:
        rate, sample = oracle_sample_rate(wl, Kh, Vh, Qh, hyper, budget_s=args.cpu_seconds)
        cores = blas_threads()
        cpu = {"value": rate, "unit": UNIT, "cores": cores, "kind": "oracle",
               "sample": f"{sample}, about {args.cpu_seconds:.0f} s; numpy float64 "
                         f"(BLAS matmul threads={cores}, elementwise single-threaded)"}

    subs = None
    if args.sub_records == "on" or (args.sub_records == "auto" and args.workload == "qwen7b-28l-32k"
                                    and not args.layers and args.stats == "window"
                                    and args.head_budgets == "uniform" and args.proxies == "paper"):
        subs = run_sub_records(args, wl, K, V, Q, ranks, M, LB, dev, peaks, peak_src)

    line = {
        "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": ms, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "bf16" if wl.dtype == S.BF16 else "f32",
        "data": "synthetic (seeded, MLLM-shaped; stands in for the paper's benchmarks)",
        "config": {"workload": wl.name, "layers": L, "batch": wl.batch, "prompt_tokens": T,
                   "q_heads": wl.n_q_heads, "kv_heads": wl.n_kv_heads, "head_dim": wl.head_dim,
                   "window": wl.window, "budgets": list(wl.budgets), "proxies": args.proxies,
                   "n_proxies": hyper["n_proxies"], "n_groups": hyper["n_groups"],
                   "gamma": hyper["gamma"], "tau": hyper["tau"], "lambda": hyper["lam"],
                   "stats": args.stats, "head_budgets": args.head_budgets,
                   **({"d_model": d_model} if args.stats == "hidden" else {}),
                   "l2": "inputs (K+V %.2f GB) larger than L2; no flush" % (2 * k_read / 1e9),
                   "parallelism": f"replicas x{world}"},
        "hbm_roofline_frac": hbm_frac,
        "hbm_bytes_per_step": bytes_step,
        "stage_ms": stage_ms,
        "roofline": roof,
        **extra_roofs,
        "cpu_baseline": cpu,
        "e2e": {"value": job_value(T * L, world, e_ms), "unit": UNIT, "ms_per_step": e_ms,
                "trials_ms_per_step": e_trials,
                "timing": f"median of 3 back-to-back trials of {e_steps} steps",
                "pipeline": "K and Qwin double-buffered on the device (copies of step k+1 overlap "
                            "the selection of step k); V read in place from pinned host memory, "
                            "only the kept rows, by the gather; outputs double-buffered and "
                            "copied back on the copy stream",
                "h2d_bytes_per_step": h2d, "d2h_bytes_per_step": d2h},
        "clocks": clk,
        "gpu_launches": launches,
        "input_gen_s": gen_s,
        **({"coverage": coverage} if coverage else {}),
        **({"sub_records": subs} if subs else {}),
    }
    if rank == 0:
        print(json.dumps(line), flush=True)
    ranks.close()
    return 0


def main(argv=None):
    ap = argparse.ArgumentParser(description=__doc__.split("\n")[0])
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=10)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", choices=["ours", "reference"], default="ours")
    ap.add_argument("--workload", default="qwen7b-28l-32k", choices=sorted(S.WORKLOADS))
    ap.add_argument("--layers", type=int, default=0,
                    help="use only the first N layers of the workload (profiling runs)")
    ap.add_argument("--proxies", choices=["paper", "few"], default="paper",
                    help="paper: N=512, G=32 (Section 4.1); few: N=W, G=W/16")
    ap.add_argument("--stats", choices=["window", "prefill", "hidden"], default="window",
                    help="proxy statistics: over the W window queries; over every prompt query "
                         "(mmshift_prefill_stats + mmshift_select_with_stats); or over the prefill "
                         "hidden states with proxies projected by W_Q (mmshift_hidden_stats + "
                         "mmshift_build_hidden_proxies + mmshift_select)")
    ap.add_argument("--head-budgets", choices=["uniform", "pyramid"], default="uniform",
                    help="budget per (layer, KV head): uniform C, or pyramid-shaped (1.5 C at the "
                         "first layer to C/2 at the last, C on average) through "
                         "mmshift_select_head_budgets")
    ap.add_argument("--coverage", type=int, default=32,
                    help="decode queries per (layer, request) for the attention-mass coverage of "
                         "the kept set (0 disables)")
    ap.add_argument("--d-model", type=int, default=0,
                    help="hidden size for --stats hidden (0: Hq * d, as in Qwen2.5-VL-7B)")
    ap.add_argument("--cpu-seconds", type=float, default=15.0,
                    help="CPU oracle sample budget for cpu_baseline (0 disables)")
    ap.add_argument("--ref-seconds", type=float, default=8.0,
                    help="per-step oracle sample budget of --impl reference")
    ap.add_argument("--sub-records", choices=["auto", "on", "off"], default="auto",
                    help="also time the 32K stack with few proxies and the 72B-class ragged batch "
                         "(both proxy settings) in the same run; auto: with the default workload")
    ap.add_argument("--gen-procs", type=int, default=min(16, os.cpu_count() or 1))
    args = ap.parse_args(argv)
    if args.warmup < 3:
        ap.error("--warmup must be >= 3")
    wl = S.WORKLOADS[args.workload]
    if args.layers:
        wl = wl.replace(name=f"{wl.name}[:{args.layers} layers]", n_layers=min(args.layers, wl.n_layers))
    if args.impl == "reference":
        return run_reference(args, wl)
    return run_gpu(args, wl)


if __name__ == "__main__":
    sys.exit(main())
