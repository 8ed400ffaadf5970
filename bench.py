#!/usr/bin/env python
"""Benchmark of the partially linear FFN forward (TARDIS, arXiv 2501.10054) on B200.

    python bench.py --gpus N --steps K --warmup W            # the CUDA library
    python bench.py --impl reference --steps K --warmup W    # the fp64 CPU oracle on the host cores

Workload (default): the 7B-class decode configuration - one FFN layer shape d_model = 4096,
d_ff = 16384, bf16, about 10 % of the neurons flagged per token - run as batch-1 decode.  One
"step" is 512 successive tokens, each one call of tardis_ffn_forward (predictor, flagging, folded
product, result fixing).  Calls rotate over `--layers` independently seeded layers so that the
state a call touches (about 80 MB) has left the 126 MB L2 by the time its layer comes round again.
Prints ONE JSON line (metric, value, roofline, cpu_baseline, e2e, clocks and context legs; the keys are
described where they are filled in below).
"""
from __future__ import annotations

import argparse
import ctypes
import json
import os
import sys
import threading
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

METRIC = "tardis_ffn_tokens_per_s"
UNIT = "tokens/s"
L2_BYTES = 126e6


def parse_args():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=40)
    ap.add_argument("--warmup", type=int, default=5)
    ap.add_argument("--impl", default="tardis", choices=["tardis", "reference"])
    ap.add_argument("--workload", default="decode_7b")
    ap.add_argument("--batch", type=int, default=1)
    ap.add_argument("--tokens", type=int, default=512, help="tokens per step")
    ap.add_argument("--layers", type=int, default=8, help="independent layers the calls rotate over (L2-cold)")
    ap.add_argument("--graph", type=int, default=0, help="replay one step as a CUDA graph")
    ap.add_argument("--no-context", action="store_true", help="skip the dense-FFN / batch-64 / oracle context legs")
    ap.add_argument("--cpu-sample-tokens", type=int, default=16)
    ap.add_argument("--mode", default="decode", choices=["decode", "prefill", "studies"],
                    help="prefill: time one prefill chunk of one layer through the batched path (a context run, not the headline)")
    ap.add_argument("--prefill-tokens", type=int, default=8192)
    return ap.parse_args()


def algorithmic_bytes(cfg, batch, union_flagged):
    """Bytes one call must move (bf16): folded matrix + predictor codes + group metadata (4 B per
    neuron and group) + W1 row and W2^T row of every flagged neuron + per-neuron tables + bias + x, y."""
    d, h, G = cfg.d_model, cfg.d_ff, cfg.group
    return (2 * d * d + h * d // 4 + 4 * h * (d // G) + union_flagged * 4 * d + 12 * h + 8 * union_flagged
            + 4 * d + 4 * batch * d)


class ClockSampler:
    """Samples SM clock and throttle reasons through NVML while the timed region runs (read-only)."""

    def __init__(self, index):
        self.samples, self.reasons, self.max_mhz = [], set(), None
        self._stop = threading.Event()
        self._thr = None
        try:
            import pynvml
            pynvml.nvmlInit()
            self.nv = pynvml
            self.dev = pynvml.nvmlDeviceGetHandleByIndex(index)
            self.max_mhz = pynvml.nvmlDeviceGetMaxClockInfo(self.dev, pynvml.NVML_CLOCK_SM)
        except Exception:
            self.nv = None

    def _run(self):
        nv = self.nv
        names = {"hw_slowdown": nv.nvmlClocksEventReasonHwSlowdown if hasattr(nv, "nvmlClocksEventReasonHwSlowdown") else 0x8,
                 "hw_thermal_slowdown": 0x40, "sw_thermal_slowdown": 0x20, "sw_power_cap": 0x4, "hw_power_brake": 0x80}
        while not self._stop.is_set():
            try:
                self.samples.append(nv.nvmlDeviceGetClockInfo(self.dev, nv.NVML_CLOCK_SM))
                r = nv.nvmlDeviceGetCurrentClocksEventReasons(self.dev) if hasattr(nv, "nvmlDeviceGetCurrentClocksEventReasons") \
                    else nv.nvmlDeviceGetCurrentClocksThrottleReasons(self.dev)
                for k, bit in names.items():
                    if r & bit:
                        self.reasons.add(k)
            except Exception:
                pass
            time.sleep(0.02)

    def __enter__(self):
        if self.nv is not None:
            self._thr = threading.Thread(target=self._run, daemon=True)
            self._thr.start()
        return self

    def __exit__(self, *a):
        self._stop.set()
        if self._thr is not None:
            self._thr.join()

    def summary(self):
        s = sorted(self.samples)
        return {"sm_mhz": s[len(s) // 2] if s else None, "sm_max_mhz": self.max_mhz, "reasons": sorted(self.reasons),
                "samples": len(s)}


def oracle_sample(cfg, layer64, x64, reps=1):
    """The oracle as it stands on the host cores: fold once (offline part), then the online part
    (predictor score, flags, folded product, fixing) on the sample tokens.  Returns (tokens/s, fold_s, cores)."""
    from threadpoolctl import threadpool_info
    from oracle import tardis_oracle as O
    s = layer64
    t0 = time.perf_counter()
    folded = O.fold(s["W1"], s["W2"], s["a"], s["c"], s["b1"], s["b2"])
    fold_s = time.perf_counter() - t0
    best = float("inf")
    for _ in range(reps):
        t0 = time.perf_counter()
        O.tardis_ffn(x64, s["W1"], s["W2"], s["a"], s["c"], s["lo"], s["hi"], s["codes"], s["scale"], s["zero"],
                     s["group"], s["b1"], s["b2"], s["act"], s["bits"], folded=folded)
        best = min(best, time.perf_counter() - t0)
    cores = max([p.get("num_threads", 1) for p in threadpool_info()] + [1])
    return x64.shape[0] / best, fold_s, cores


def run_reference(args):
    """--impl reference: the fp64 oracle on the host cores, same metric and workload, bounded sample."""
    import workloads as W
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return
    cfg = W.CONFIGS[args.workload]
    L = W.make_layer(cfg, 0)
    s = L.numpy64()
    n = max(1, min(args.cpu_sample_tokens, 8))
    x64 = W.make_tokens(cfg, n, 0).double().numpy()
    from oracle import tardis_oracle as O
    folded = O.fold(s["W1"], s["W2"], s["a"], s["c"], s["b1"], s["b2"])

    def step():
        O.tardis_ffn(x64, s["W1"], s["W2"], s["a"], s["c"], s["lo"], s["hi"], s["codes"], s["scale"], s["zero"],
                     s["group"], s["b1"], s["b2"], s["act"], s["bits"], folded=folded)

    steps, warm = max(1, min(args.steps, 5)), max(1, min(args.warmup, 2))
    for _ in range(warm):
        step()
    t0 = time.perf_counter()
    for _ in range(steps):
        step()
    dt = (time.perf_counter() - t0) / steps
    from threadpoolctl import threadpool_info
    cores = max([p.get("num_threads", 1) for p in threadpool_info()] + [1])
    val = n / dt
    sample = "%d tokens per step, %d steps, batch-1 semantics (tokens independent), fold excluded (offline)" % (n, steps)
    print(json.dumps({
        "impl": "reference", "metric": METRIC, "value": val, "unit": UNIT, "n_gpus": args.gpus, "steps": steps,
        "warmup": warm, "ms_per_step": dt * 1e3, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
        "dtype": "f64", "data": "synthetic",
        "config": {"workload": "%s batch-%d decode, d_model=%d d_ff=%d" % (cfg.name, args.batch, cfg.d_model, cfg.d_ff)},
        "cpu_baseline": {"value": val, "unit": UNIT, "cores": cores, "kind": "oracle", "sample": sample},
        "e2e": {"value": val, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }))


def main():
    args = parse_args()
    if args.impl == "reference":
        run_reference(args)
        return
    import torch
    import torch.distributed as dist
    import paper_2501_10054_b200 as T
    from paper_2501_10054_b200 import build as tbuild
    import workloads as W

    rank = int(os.environ.get("RANK", "0"))
    world = int(os.environ.get("WORLD_SIZE", "1"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    if not torch.cuda.is_available():
        raise SystemExit("bench.py needs a CUDA device: the library has no CPU fallback")
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    if world > 1:
        dist.init_process_group("nccl", device_id=dev)
    if rank == 0:
        tbuild.build()
    if world > 1:
        dist.barrier()
    lib = T.load_library()

    cfg = W.CONFIGS[args.workload]
    if args.mode == "prefill":
        run_prefill(args, cfg, T, W, torch, dev, rank, world)
        return
    if args.mode == "studies":
        run_studies(args, T, W, torch, dev)
        return
    d, h, B, NT = cfg.d_model, cfg.d_ff, args.batch, args.tokens
    assert NT % B == 0
    # ---- set-up: independent layers (weak scaling: every rank has its own layers and tokens) ----
    handles, dense = [], []
    layer0_64 = None
    for l in range(args.layers):
        L = W.make_layer(cfg, seed=rank * 1000 + l, device=dev)
        handles.append(T.fold_layer(L))
        dense.append((L.W1, L.W2, L.b1, L.b2))
        if l == 0 and rank == 0 and not args.no_context:
            layer0_64 = L.numpy64()
    # every rank takes its contiguous share of one seeded token stream (tokens are independent: no exchange is needed)
    from paper_2501_10054_b200 import sharding
    first, count = sharding.token_shard(NT * world, world, rank)
    x_all = W.make_tokens(cfg, NT * world, seed=0, device=dev)[first:first + count].contiguous()
    y_all = torch.empty_like(x_all)
    torch.cuda.synchronize()
    touched = algorithmic_bytes(cfg, B, int(0.1 * h))
    stream = torch.cuda.current_stream()
    sptr = stream.cuda_stream or None
    esz = x_all.element_size()
    fwd = lib.tardis_ffn_forward

    def make_step(batch, xs, ys):
        calls = [(handles[i % len(handles)], xs.data_ptr() + i * batch * d * esz, ys.data_ptr() + i * batch * d * esz)
                 for i in range(NT // batch)]

        def step():
            for hdl, xp, yp in calls:
                st = fwd(hdl, xp, yp, batch, sptr)
                if st:
                    raise RuntimeError("tardis_ffn_forward status %d" % st)
        return step

    def timed(step, steps, warm, sampler=None, graph=False):
        runner = step
        if graph:
            g = torch.cuda.CUDAGraph()
            side = torch.cuda.Stream()
            side.wait_stream(torch.cuda.current_stream())
            with torch.cuda.stream(side):
                step()
            torch.cuda.current_stream().wait_stream(side)
            with torch.cuda.graph(g):
                step()
            runner = g.replay
        for _ in range(max(3, warm)):
            runner()
        torch.cuda.synchronize()
        if world > 1:
            dist.barrier()
            torch.cuda.synchronize()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        ctx = sampler if sampler is not None else _Null()
        with ctx:
            e0.record()
            for _ in range(steps):
                runner()
            e1.record()
            torch.cuda.synchronize()
        if world > 1:
            dist.barrier()
            torch.cuda.synchronize()
        ms = e0.elapsed_time(e1) / steps
        if world > 1:
            t = torch.tensor([ms], device=dev)
            dist.all_reduce(t, op=dist.ReduceOp.MAX)
            ms = float(t.item())
        return ms

    # ---- device-resident timing (the headline `value`) ----
    st0 = [T.tardis_stats(hd) for hd in handles]
    sampler = ClockSampler(local)
    step = make_step(B, x_all, y_all)
    if args.graph:
        # the graph path captures on torch's capture stream: rebuild the call list inside timed()
        def step_graph():
            s2 = torch.cuda.current_stream().cuda_stream or None
            for i in range(NT // B):
                st = fwd(handles[i % len(handles)], x_all.data_ptr() + i * B * d * esz, y_all.data_ptr() + i * B * d * esz, B, s2)
                if st:
                    raise RuntimeError("tardis_ffn_forward status %d" % st)
        ms = timed(step_graph, args.steps, args.warmup, sampler, graph=True)
    else:
        ms = timed(step, args.steps, args.warmup, sampler)
    st1 = [T.tardis_stats(hd) for hd in handles]
    if any(s["device_error"] for s in st1):
        raise SystemExit("device error word set: %r" % [s["device_error"] for s in st1])
    tokens_done = sum(b["tokens"] - a["tokens"] for a, b in zip(st0, st1))
    flagged = sum(b["flagged_total"] - a["flagged_total"] for a, b in zip(st0, st1)) / max(1, tokens_done)
    launches_per_step = sum(b["launches"] - a["launches"] for a, b in zip(st0, st1)) / (max(3, args.warmup) + args.steps)
    value = world * NT / (ms * 1e-3)

    # ---- end to end: host buffers, H2D of the step's tokens and D2H of its outputs inside the timed region ----
    xh = x_all.cpu().pin_memory()
    yh = torch.empty_like(xh).pin_memory()
    xd = torch.empty_like(x_all)
    yd = torch.empty_like(x_all)
    inner = make_step(B, xd, yd)

    def e2e_step():
        xd.copy_(xh, non_blocking=True)
        inner()
        yh.copy_(yd, non_blocking=True)

    ms_e2e = timed(e2e_step, max(3, args.steps // 4), 3)
    e2e_value = world * NT / (ms_e2e * 1e-3)

    # ---- roofline of the dominant kernel ----
    peaks = {}
    try:
        peaks = json.load(open(os.path.join(ROOT, "MEASURED_PEAKS.json")))
    except Exception:
        pass
    peak = float(peaks.get("hbm_gbs", 6650.0))
    peak_src = "measured" if "hbm_gbs" in peaks else "fallback"
    calls_per_step = NT // B
    union = flagged if B == 1 else h * (1 - (1 - flagged / h) ** B)
    alg = algorithmic_bytes(cfg, B, union)
    dur_s = ms * 1e-3 / calls_per_step
    achieved = alg / dur_s / 1e9
    roofline = {"bound": "hbm", "achieved": achieved, "peak": peak, "unit": "GB/s", "frac": achieved / peak,
                "traffic": None, "peak_source": peak_src, "kernel": "k_fused" if B <= 16 else "k_gemm (batched path)",
                "algorithmic_bytes_per_launch": alg, "avg_launch_us": dur_s * 1e6,
                "frac_of_nominal_8TBs": achieved / 8000.0}
    # DRAM bytes per launch from the committed ncu summary of this kernel (null when there is none)
    prof = os.path.join(ROOT, "profiles", "k_fused_%s.txt" % args.workload)
    if B == 1 and os.path.exists(prof):
        for line in open(prof):
            if line.startswith("dram_bytes_per_launch:"):
                try:
                    roofline["traffic"] = float(line.split(":")[1].split()[0])
                except Exception:
                    pass

    out = {
        "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps, "warmup": max(3, args.warmup),
        "ms_per_step": ms, "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": cfg.dtype,
        "data": "synthetic",
        "config": {"workload": "%s batch-%d decode, d_model=%d d_ff=%d, %d tokens/step" % (cfg.name, B, d, h, NT),
                   "flagged_per_token": flagged, "flagged_frac": flagged / h, "pred_group": cfg.group,
                   "l2": "inputs larger than L2: calls rotate over %d independent layers (%.0f MB touched per call, %.0f MB per round)"
                         % (len(handles), touched / 1e6, touched * len(handles) / 1e6),
                   "cuda_graph": bool(args.graph)},
        "clocks": sampler.summary(),
        "e2e": {"value": e2e_value, "unit": UNIT, "h2d_bytes_per_step": xh.numel() * esz, "d2h_bytes_per_step": yh.numel() * esz,
                "ms_per_step": ms_e2e},
        "gpu_launches": int(round(launches_per_step * args.steps)),
        "roofline": roofline,
    }

    # ---- context legs (rank 0, N = 1 semantics): batch 64, dense FFN, oracle on the host cores ----
    if not args.no_context:
        def decode_leg(cfg_l, hds, xs, ys, batch, steps=6):
            """Batch-`batch` decode calls rotating over the handles `hds`: tokens/s, time per call, fraction of the HBM roofline
            on the algorithmic bytes of a call (union of the flagged neurons measured by the library)."""
            ntok = xs.shape[0] // batch * batch
            esz_l = xs.element_size()
            calls = [(hds[i % len(hds)], xs.data_ptr() + i * batch * cfg_l.d_model * esz_l, ys.data_ptr() + i * batch * cfg_l.d_model * esz_l)
                     for i in range(ntok // batch)]

            def step_l():
                for hdl, xp_, yp_ in calls:
                    st_ = fwd(hdl, xp_, yp_, batch, sptr)
                    if st_:
                        raise RuntimeError("tardis_ffn_forward status %d" % st_)
            s0_ = [T.tardis_stats(hd) for hd in hds]
            ms_l = timed(step_l, steps, 3)
            s1_ = [T.tardis_stats(hd) for hd in hds]
            toks = sum(b_["tokens"] - a_["tokens"] for a_, b_ in zip(s0_, s1_))
            fl = sum(b_["flagged_total"] - a_["flagged_total"] for a_, b_ in zip(s0_, s1_)) / max(1, toks)
            union_l = fl if batch == 1 else cfg_l.d_ff * (1 - (1 - fl / cfg_l.d_ff) ** batch)
            alg_l = algorithmic_bytes(cfg_l, batch, union_l)
            us_call = ms_l * 1e3 / (ntok // batch)
            gbs = alg_l / (us_call * 1e-6) / 1e9
            return {"value": world * ntok / (ms_l * 1e-3), "unit": UNIT, "us_per_call": us_call, "flagged_per_token": fl,
                    "path": s1_[0]["last_path"], "algorithmic_bytes_per_call": alg_l,
                    "roofline": {"bound": "hbm", "achieved": gbs, "peak": peak, "unit": "GB/s", "frac": gbs / peak,
                                 "frac_of_nominal_8TBs": gbs / 8000.0}}

        # the same layers at other batch sizes (one launch of the fused kernel up to 4 tokens, several up to 16, the
        # tensor-core path beyond)
        for bsz in (4, 16, 64):
            if NT % bsz == 0 and B != bsz:
                out["batch%d" % bsz] = decode_leg(cfg, handles, x_all, y_all, bsz, steps=max(3, args.steps // 4))

        # prefill chunk of one layer through the batched path, and its folded GEMM alone against the bf16 peak
        npre = 8192
        xp = W.make_tokens(cfg, npre, seed=rank + 77, device=dev)
        yp = torch.empty_like(xp)

        def prefill_step():
            st = fwd(handles[0], xp.data_ptr(), yp.data_ptr(), npre, sptr)
            if st:
                raise RuntimeError("tardis_ffn_forward status %d" % st)

        msp = timed(prefill_step, 5, 3)
        Wf = torch.empty(d, d, dtype=xp.dtype, device=dev)
        T.tardis_export_folded(handles[0], Wf, None)
        Cout = torch.empty(npre, d, dtype=torch.float32, device=dev)
        msg = timed(lambda: T.tardis_gemm_bf16(xp, Wf, Cout), 10, 3)
        tf = 2.0 * npre * d * d / (msg * 1e-3) / 1e12
        tpeak = float(peaks.get("bf16_tflops", 1590.0))
        out["prefill_context"] = {"tokens": npre, "value": world * npre / (msp * 1e-3), "unit": UNIT, "ms_per_chunk": msp,
                                  "flops_per_token": 6 * d * h + 2 * d * d,   # (scores over one bf16 term: all that these predictors need)
                                  "wf_gemm": {"bound": "tensor", "achieved": tf, "peak": tpeak, "unit": "TFLOP/s", "frac": tf / tpeak,
                                              "ms": msg, "peak_source": "measured burst" if "bf16_tflops" in peaks else "fallback"}}
        del xp, yp, Cout, Wf
        # the offline fold of one layer (tensor-core product + predictor / folded-matrix packing)
        Lf = W.make_layer(cfg, seed=rank * 1000 + 999, device=dev)
        torch.cuda.synchronize()
        ef0, ef1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        ef0.record()
        hf = T.fold_layer(Lf)
        ef1.record()
        torch.cuda.synchronize()
        out["fold_ms_per_layer"] = ef0.elapsed_time(ef1)
        T.tardis_destroy(hf)
        # offline statistics of one layer: pre-activations of 2048 calibration tokens (tensor-core product), then the
        # quantile ranges and least-squares fits of all neurons
        ncal = 2048
        xcal = W.make_tokens(cfg, ncal, rank * 1000 + 998, device=dev, tag="calib")
        zcal = torch.empty(h, ncal, dtype=torch.float32, device=dev)

        def calib_step():
            T.tardis_gemm_bf16(Lf.W1, xcal, zcal)
            T.tardis_calibrate(zcal, Lf.b1, cfg.q_lo, cfg.q_hi, cfg.act)

        msc = timed(calib_step, 5, 3)
        msk = timed(lambda: T.tardis_calibrate(zcal, Lf.b1, cfg.q_lo, cfg.q_hi, cfg.act), 5, 1)
        out["calibrate_context"] = {"ms_per_layer": msc, "ms_ranges_and_fits": msk, "n_cal": ncal,
                                    "what": "z = W1 Xcal^T (tcgen05 GEMM) + quantile ranges + least-squares fits, 16384 neurons"}
        # Algorithm 1's greedy range search (KDE centroid + expansion by the smaller regression error) on the same samples
        T.tardis_range_search(zcal, Lf.b1, 0.85, 0.05, cfg.act)
        msr = timed(lambda: T.tardis_range_search(zcal, Lf.b1, 0.85, 0.05, cfg.act), 2, 1)
        out["range_search_context"] = {"ms_per_layer": msr, "n_cal": ncal, "threshold": 0.85, "step": 0.05,
                                       "what": "Algorithm 1 per neuron on the GPU, %d neurons; the paper reports about 30 minutes per "
                                               "layer for its search (Section 7.3, RTX 4090D)" % h}
        # the predictor by error-compensated quantisation (GPTQ, Section 6): Hessian and its Cholesky factors by torch's
        # routines (the caller's side), the channel-by-channel rounding of all neurons by tardis_build_predictor
        Xd = xcal.double()
        Hm = 2.0 / ncal * Xd.t() @ Xd
        Hm += 0.01 * torch.mean(torch.diagonal(Hm)) * torch.eye(d, dtype=torch.float64, device=dev)
        Um = torch.linalg.cholesky(torch.cholesky_inverse(torch.linalg.cholesky(Hm)), upper=True).contiguous()
        msb = timed(lambda: T.tardis_build_predictor(Lf.W1, Um, cfg.bits, cfg.group), 2, 1)
        out["predictor_build_context"] = {"ms_per_layer": msb, "bits": cfg.bits, "group": cfg.group,
                                          "what": "tardis_build_predictor on %d x %d weights, double precision, scratch allocation "
                                                  "and release included; the Hessian's factor is an input" % (h, d)}
        del Lf, xcal, zcal, Xd, Hm, Um

        # a chain of 32 layers on one residual stream (layer normalisation, forward, addition per layer): the bench's
        # layers four times over, batch 1, once as plain launches and once replayed from a CUDA graph
        chain = (handles * ((32 + len(handles) - 1) // len(handles)))[:32]
        xs1, ys1 = x_all[:1].clone(), torch.empty_like(x_all[:1])
        wk = torch.empty(2, 1, d, dtype=x_all.dtype, device=dev)

        def stack_step():
            T.tardis_stack_forward(chain, xs1, ys1, None, None, 1e-5, True, True, work=wk)
        ms_s = timed(stack_step, max(3, args.steps // 2), 3)
        ms_g = None
        if world == 1:              # (a capture that fails on one rank only would leave the others in a barrier)
            try:
                ms_g = timed(stack_step, max(3, args.steps // 2), 3, graph=True)
            except Exception as e:  # capture refused: reported, not fatal
                out.setdefault("notes", []).append("stack graph capture failed: %s" % str(e)[:120])
        out["stack_context"] = {"layers": 32, "batch": 1, "us_per_layer": ms_s * 1e3 / 32,
                                "us_per_layer_graph": None if ms_g is None else ms_g * 1e3 / 32,
                                "what": "tardis_stack_forward: one launch of the fused kernel per layer, which normalises the stream and adds its "
                                        "output to it, chained by programmatic dependent launch"}

        def dense_step():
            for i in range(NT // B):
                W1, W2, b1, b2 = dense[i % len(dense)]
                xb = x_all[i * B:(i + 1) * B]
                hid = torch.nn.functional.gelu(torch.nn.functional.linear(xb, W1, None if b1 is None else b1.to(W1.dtype)),
                                               approximate="tanh" if cfg.act == 0 else "none")
                torch.nn.functional.linear(hid, W2, None if b2 is None else b2.to(W2.dtype))

        msd = timed(dense_step, max(3, args.steps // 4), 3)
        out["dense_ffn_context"] = {"value": world * NT / (msd * 1e-3), "unit": UNIT, "ms_per_step": msd,
                                    "what": "torch bf16 linear-gelu-linear, same rotation, same GPU",
                                    "bytes_per_call": 4 * d * h}
        # the other decode configurations, batch 1: the Falcon-7B shape at its four quantile pairs, the 8192/32768 layer
        if args.workload == "decode_7b":
            import dataclasses
            for hd in handles:
                T.tardis_destroy(hd)
            handles.clear()
            dense.clear()
            torch.cuda.empty_cache()
            other = {}
            fcfg = W.CONFIGS["falcon_7b"]
            xf = W.make_tokens(fcfg, 96, seed=rank + 5, device=dev)
            yf = torch.empty_like(xf)
            for qi, (qlo, qhi) in enumerate(W.FALCON_QUANTILES):
                c_q = dataclasses.replace(fcfg, q_lo=qlo, q_hi=qhi)
                hq = [T.fold_layer(W.make_layer(c_q, seed=rank * 1000 + 50 + l, device=dev)) for l in range(3)]
                other["falcon_7b_q%d_batch1" % qi] = dict(decode_leg(c_q, hq, xf, yf, 1, steps=4), quantiles=[qlo, qhi])
                if qi == 1:
                    other["falcon_7b_q1_batch4"] = decode_leg(c_q, hq, xf, yf, 4, steps=4)
                for hd in hq:
                    T.tardis_destroy(hd)
                torch.cuda.empty_cache()
            lcfg = W.CONFIGS["large_8k"]
            xl = W.make_tokens(lcfg, 64, seed=rank + 6, device=dev)
            yl = torch.empty_like(xl)
            hl = [T.fold_layer(W.make_layer(lcfg, seed=rank * 1000 + 70 + l, device=dev)) for l in range(2)]
            other["large_8k_batch1"] = decode_leg(lcfg, hl, xl, yl, 1, steps=4)
            for hd in hl:
                T.tardis_destroy(hd)
            torch.cuda.empty_cache()
            out["other_configs"] = other
        out["paper_context"] = {"e2e_speedup_vllm": 1.59, "e2e_speedup_hf": 1.39, "ffn_speedup": 1.86,
                                "hardware": "RTX 4090D, Falcon-7B, 80% FFN compression (paper Section 7.4)"}
        if rank == 0 and layer0_64 is not None:
            n = args.cpu_sample_tokens
            x64 = x_all[:n].double().cpu().numpy()
            v, fold_s, cores = oracle_sample(cfg, layer0_64, x64)
            out["cpu_baseline"] = {"value": v, "unit": UNIT, "cores": cores, "kind": "oracle",
                                   "sample": "online path on %d tokens of layer 0 (fold excluded: offline, %.1f s)" % (n, fold_s),
                                   "fold_s": fold_s}
    if rank == 0:
        print(json.dumps(out))
    for hd in handles:
        T.tardis_destroy(hd)
    if world > 1:
        dist.destroy_process_group()


def run_prefill(args, cfg, T, W, torch, dev, rank, world):
    """One layer, one chunk of --prefill-tokens tokens per step through the batched path (tcgen05 GEMMs)."""
    d, h, n = cfg.d_model, cfg.d_ff, args.prefill_tokens
    L = W.make_layer(cfg, seed=rank * 1000, device=dev)
    hd = T.fold_layer(L)
    x = W.make_tokens(cfg, n, seed=rank + 77, device=dev)
    y = torch.empty_like(x)
    for _ in range(max(3, args.warmup)):
        T.tardis_ffn_forward(hd, x, y)
    torch.cuda.synchronize()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    steps = max(1, args.steps)
    e0.record()
    for _ in range(steps):
        T.tardis_ffn_forward(hd, x, y)
    e1.record()
    torch.cuda.synchronize()
    ms = e0.elapsed_time(e1) / steps
    st = T.tardis_stats(hd)
    peaks = {}
    try:
        peaks = json.load(open(os.path.join(ROOT, "MEASURED_PEAKS.json")))
    except Exception:
        pass
    tpeak = float(peaks.get("bf16_tflops_sustained", 1400.0))
    flops = float(n) * (6 * d * h + 2 * d * d)         # (scores over one bf16 term: all that these predictors need)
    tf = flops / (ms * 1e-3) / 1e12
    if rank == 0:
        print(json.dumps({
            "metric": METRIC, "value": world * n / (ms * 1e-3), "unit": UNIT, "n_gpus": world, "steps": steps,
            "warmup": max(3, args.warmup), "ms_per_step": ms, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
            "dtype": cfg.dtype, "data": "synthetic",
            "config": {"workload": "%s prefill chunk, d_model=%d d_ff=%d, %d tokens/step (one layer)" % (cfg.name, d, h, n),
                       "flagged_frac": st["flagged_total"] / max(1, st["tokens"]) / h, "l2": "inputs larger than L2"},
            "roofline": {"bound": "tensor", "achieved": tf, "peak": tpeak, "unit": "TFLOP/s", "frac": tf / tpeak, "traffic": None,
                         "peak_source": "measured sustained" if "bf16_tflops_sustained" in peaks else "fallback",
                         "kernel": "k_gemm (4 products per chunk: scores, folded, pre-activations, output)",
                         "flops_per_step": flops}}))
    T.tardis_destroy(hd)


def run_studies(args, T, W, torch, dev):
    """Two small studies on synthetic layers, after Sections 7.6 and 7.7 of the paper (context numbers, not the headline):
    (1) predictor size: flag precision and recall of the 2-, 4- and 8-bit predictors against the flags taken on the true
        pre-activations (the exact-range mode), on the 7B-class decode layer;
    (2) precision of the reordered product: error of the folded matrix against the fp64 oracle for three kinds of
        intermediate (leading bf16 term only, exact two-term bf16 split = the default, plain fp32), at two layer sizes."""
    import dataclasses
    import numpy as np
    from oracle import tardis_oracle as O
    from tests import helpers as Hp
    out = {"mode": "studies", "data": "synthetic"}
    base = W.CONFIGS["decode_7b"]
    x = W.make_tokens(base, 64, seed=3, device=dev)
    sweep = {}
    for bits in (2, 3, 4, 8):
        cfg = dataclasses.replace(base, bits=bits)
        L = W.make_layer(cfg, seed=11, device=dev)
        hd = T.fold_layer(L)
        y = torch.empty_like(x)
        flags = {}
        for name, path in (("predictor", 0), ("exact", 4)):
            T.tardis_set_path(hd, path)
            bm = torch.zeros(64, cfg.d_ff // 32, dtype=torch.int32, device=dev)
            T.tardis_set_debug_capture(hd, bm, None)
            for t in range(64):
                T.tardis_set_debug_capture(hd, bm[t:t + 1], None)
                T.tardis_ffn_forward(hd, x[t:t + 1], y[t:t + 1])
            torch.cuda.synchronize()
            T.tardis_set_debug_capture(hd, None, None)
            flags[name] = Hp.unpack_bitmap(bm, cfg.d_ff)
        P, E = flags["predictor"], flags["exact"]
        tp = float((P & E).sum())
        sweep["bits%d" % bits] = {"flagged_frac_predictor": float(P.mean()), "flagged_frac_exact": float(E.mean()),
                                  "precision": tp / max(1.0, float(P.sum())), "recall": tp / max(1.0, float(E.sum())),
                                  "predictor_bytes": cfg.d_ff * cfg.d_model * bits // 8}
        T.tardis_destroy(hd)
        del L
        torch.cuda.empty_cache()
    out["predictor_size"] = {"what": "flags of the quantised predictor against flags from the true pre-activations, 64 tokens, "
                                     "decode_7b shape (ranges tuned for about 10 % flagged with the 2-bit predictor)", **sweep}
    fold = {}
    for name, d, h in (("x1", 2048, 8192), ("x4", 4096, 16384)):
        cfg = W.LayerConfig("fold_" + name, d, h, n_calib=1024, group=128)
        L = W.make_layer(cfg, seed=21, device=dev)
        s = L.numpy64()
        rng = np.random.default_rng(21)
        rows = np.sort(rng.choice(d, size=16, replace=False))
        ref = O.fold_rows(rows, s["W1"], s["W2"], s["a"])
        scale2 = float((ref ** 2).mean())
        res = {}
        for mode, flag in (("bf16_intermediate", 1), ("bf16_two_terms_default", 0), ("fp32_plain", 2)):
            hd = T.fold_layer(L, flags=flag)
            Wf = torch.empty(d, d, dtype=torch.bfloat16, device=dev)
            T.tardis_export_folded(hd, Wf, None)
            torch.cuda.synchronize()
            got = Wf[torch.as_tensor(rows, device=dev)].double().cpu().numpy()
            res[mode] = {"mse": float(((got - ref) ** 2).mean()), "relative_mse": float(((got - ref) ** 2).mean()) / scale2}
            T.tardis_destroy(hd)
        rounded = torch.as_tensor(ref).to(torch.bfloat16).double().numpy()
        res["bf16_rounding_floor"] = {"mse": float(((rounded - ref) ** 2).mean()), "relative_mse": float(((rounded - ref) ** 2).mean()) / scale2}
        fold[name] = dict(res, d_model=d, d_ff=h)
        del L
        torch.cuda.empty_cache()
    out["fold_precision"] = {"what": "mean squared error of 16 sampled rows of W_f (stored in bf16) against the fp64 oracle", **fold}
    print(json.dumps(out))


class _Null:
    def __enter__(self):
        return self

    def __exit__(self, *a):
        return False


if __name__ == "__main__":
    main()
