"""Throughput benchmark of the GB300 CKP periodogram (arXiv:1412.1840).

One step = one best-period search over one synthetic batch through the C ABI
(cp_best_period): per-curve scalars, the pair spectrum and the statistic at
every trial frequency (or the pair sum, where that is cheaper), the pair sum at
the candidates for the best, normalisation, argmax / coarse-then-fine search and
the Table tab:th discriminator.

Default workload (N=1): 4096 lightcurves, N ~ U{300..1000}, seasonal sampling
over 2500 d, grid 0.002-5 1/d step 1e-4 (49,981 frequencies), direct form,
sigma_t from the Bowley-skewness rule.

  value     lightcurves/s with inputs resident in device memory (CUDA events
            around each step; L2 flushed between steps)
  e2e       the same through host (pinned) buffers: H2D of the inputs and D2H
            of the results inside every timed step
  roofline  the pair spectrum's kernels against the measured copy bandwidth (the
            transforms' least traffic); where the pair sum evaluates every frequency,
            that kernel against the SFU ceiling (one ex2 per pair-frequency, 32/clk/SM)
  cpu_baseline  the FP64 oracle timed on the host cores on a bounded sample
  tensor    the tensor-core form on the same batch (FP16 or BF16 operands, per-curve
            harmonics): device-resident rate, its roofline against the measured
            sustained BF16 rate, the other 16-bit type, and its own e2e

Multi-GPU (torchrun): each rank processes its own batch of the same shape
(independent lightcurves; no collective on the data path): weak scaling.
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
sys.path.insert(0, ROOT)

import synth  # noqa: E402

PEAKS_TABLE = os.path.join(ROOT, "paper_1412_1840_gb300", "peaks_gb300.json")
SM_MAX_MHZ = 2070.0


def sfu_ex2_per_clk_sm():
    """MUFU ex2.approx.f32 per clock per SM measured on this GPU by the
    package's instruction-rate probes (paper_1412_1840_gb300.peaks)."""
    with open(PEAKS_TABLE) as f:
        return float(json.load(f)["rates"]["ex2_f32"]["per_clk_per_sm"])
# DRAM bytes per byte of period-independent magnitude-kernel tiles, measured with
# ncu (dram__bytes_read.sum + dram__bytes_write.sum) on 256 curves x 2,048
# frequencies: each tile is read from DRAM once per search, later units of the
# same curve hit L2, so a full launch moves (this ratio) x (its tile bytes).
DRAM_PER_W_BYTE_DIRECT = 1.034
DRAM_PER_W_BYTE_TENSOR = 1.044


def spectrum_bytes(sigma_t, g):
    """Least memory traffic of the pair spectrum of curves with these sigma_t on a uniform grid from a
    multiple of df (csrc/cp_spec.cu): the cells and the data between the two transform passes each
    written and read once, the spectrum written and read once, the values written once."""
    top = int(round(g.f_min / g.df)) + g.n_freq - 1
    total = 0.0
    for st, count in zip(*np.unique(np.round(np.asarray(sigma_t, np.float64), 3), return_counts=True)):
        k = 1.0 / (st * st)                     # a_n = 2 e^-k I_n(k) by the backward recurrence
        n0 = min(130, int(14 + 10 / st))
        a = np.zeros(n0 + 2)
        a[n0] = 1e-200
        for n in range(n0, 0, -1):
            a[n - 1] = a[n + 1] + 2.0 * n / k * a[n]
        a[1:] *= 2.0
        tail = np.cumsum((a / a.sum())[::-1])[::-1]           # tail[n] = a_n + a_{n+1} + ...
        nh = int(np.argmax(tail[1:] <= 2e-8))                 # harmonics kept
        n_out = nh * top + 1
        q = 2.0 ** np.ceil(np.log2(max(1.1 * n_out / 2.0, 256.0)))
        total += count * (4 * 8 * q + 2 * 4 * n_out + 4 * g.n_freq)
    return total


def pair_freq(info, seconds, scale=1.0):
    """Pair-frequencies per second and what the figure stands for: evaluations where the pair sum ran at
    every frequency, else the equivalent (the pairs times the frequencies that a search through the pair
    spectrum covers, which evaluates far fewer)."""
    evaluated = info["w_bytes_direct"] + info["w_bytes_tensor"] > 0
    return {"pair_freq_per_s": scale * info["pair_freq_search"] / seconds,
            "pair_freq_basis": "evaluated" if evaluated else "equivalent (N(N-1)/2 x frequencies covered)"}


def measured_peaks():
    """Measured peaks if present, else the profiling recipe's fallback."""
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    try:
        with open(path) as f:
            d = json.load(f)
        return {"hbm_gbs": d["hbm_gbs"], "bf16_tflops": d["bf16_tflops"],
                "bf16_tflops_sustained": d.get("bf16_tflops_sustained", d["bf16_tflops"]), "source": "measured"}
    except (OSError, KeyError, ValueError):
        return {"hbm_gbs": 6800.0, "bf16_tflops": 1900.0, "bf16_tflops_sustained": 1700.0, "source": "fallback"}


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=3)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--tuning", default=os.path.join(ROOT, "paper_1412_1840_gb300", "tuning_gb300.json"),
                    help="autotuner table (paper_1412_1840_gb300.tune); 'none' for the built-in choices")
    ap.add_argument("--workload", default="ragged", choices=["ragged", "hierarchical", "bands", "single", "small", "throughput"])
    ap.add_argument("--n-curves", type=int, default=None)
    ap.add_argument("--form", default="direct", choices=["direct", "tensor"])
    ap.add_argument("--n-max", type=int, default=0, help="tensor-form harmonics (0: per curve)")
    ap.add_argument("--no-tensor", action="store_true", help="skip the tensor-form measurement")
    ap.add_argument("--dtype", default="fp16", choices=["fp16", "bf16", "bf16split"],
                    help="tensor-form operand type (bf16split: W' and Z both as hi + lo BF16 parts)")
    ap.add_argument("--no-e2e", action="store_true")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-transforms", action="store_true", help="skip timing preprocessing and whitening")
    ap.add_argument("--no-hierarchical", action="store_true",
                    help="skip the coarse-then-fine search on the same batch (both forms)")
    ap.add_argument("--no-throughput", action="store_true",
                    help="skip the 200,000-curve two-band throughput run (both forms, one timed step each)")
    ap.add_argument("--seed", type=int, default=1)
    ap.add_argument("--shard", action="store_true",
                    help="under torchrun: split ONE batch across the ranks by pair-sum cost (strong scaling) "
                         "instead of giving every rank its own batch (weak scaling)")
    return ap.parse_args()


def make_workload(args, rank):
    seed = args.seed + 1000 * rank
    if args.workload == "single":
        b, g = synth.workload_single()
        name = "single curve N=150, 9,991 freqs (0.002-2.0 step 2e-4)"
    elif args.workload == "small":
        n = args.n_curves or 256
        b, g = synth.workload_ragged(n, seed)
        g = synth.Grid(g.f_min, g.df, 2048)
        name = "%d curves N~U[300,1000], 2,048 freqs (profiling case)" % n
    elif args.workload == "throughput":
        ns = (args.n_curves or 200000) // 2
        b, g = synth.workload_throughput(ns, seed)
        name = ("%d two-band sources (%d curves) N~U[200,1000] per band, SNR 0.2-10; coarse 0.002-5 step 1e-3, "
                "top-10 refined at 1e-5 over +-2e-3" % (ns, 2 * ns))
    elif args.workload == "bands":
        n = args.n_curves or 4096
        b, g = synth.workload_bands(n, seed)
        name = ("%d curves N~U[300,1000] seasonal 2500 d; bands method N_b=3, N_t=150 on 0.00125-3 step 1e-4 "
                "(29,988 window freqs, 450 trial freqs per curve)" % n)
    elif args.workload == "hierarchical":
        n = args.n_curves or 4096
        b, g = synth.workload_hierarchical(n, seed)
        name = ("%d curves N~U[300,1000] seasonal 2500 d; coarse 0.002-5 step 1e-3, top-10 refined "
                "at 1e-5 over +-2e-3" % n)
    else:
        n = args.n_curves or 4096
        b, g = synth.workload_ragged(n, seed)
        name = "%d curves N~U[300,1000] seasonal 2500 d; grid 0.002-5 step 1e-4 (49,981 freqs)" % n
    return b, g, name


class ClockSampler:
    """nvidia-smi SM clock / throttle sampling during the timed region."""

    def __init__(self, index: int):
        self.index = index
        self.rows = []
        self.proc = None

    def __enter__(self):
        q = ("clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.hw_slowdown,"
             "clocks_event_reasons.hw_thermal_slowdown,clocks_event_reasons.sw_thermal_slowdown,"
             "clocks_event_reasons.sw_power_cap")
        try:
            self.proc = subprocess.Popen(["nvidia-smi", "-i", str(self.index), "--query-gpu=" + q,
                                          "--format=csv,noheader,nounits", "-lms", "200"],
                                         stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.thread = threading.Thread(target=self._read, daemon=True)
            self.thread.start()
        except (OSError, FileNotFoundError):
            self.proc = None
        return self

    def _read(self):
        for line in self.proc.stdout:
            parts = [x.strip() for x in line.split(",")]
            if len(parts) >= 7:
                self.rows.append(parts)

    def __exit__(self, *exc):
        if self.proc:
            self.proc.terminate()
            try:
                self.proc.wait(timeout=5)
            except subprocess.TimeoutExpired:
                self.proc.kill()

    def summary(self):
        if not self.rows:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["unsampled"]}
        sm = [float(r[0]) for r in self.rows if r[0].replace(".", "").isdigit()]
        mx = [float(r[1]) for r in self.rows if r[1].replace(".", "").isdigit()]
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        reasons = sorted({names[k] for r in self.rows for k in range(4) if r[3 + k].lower() == "active"})
        return {"sm_mhz": float(np.median(sm)) if sm else None, "sm_max_mhz": max(mx) if mx else None,
                "reasons": reasons, "samples": len(self.rows)}


def cpu_baseline(b, g, target_s=15.0, max_curves=8):
    """The FP64 oracle, as it stands, on a bounded sample of the workload:
    the first curves of the batch at a strided subset of the grid; the
    per-(N^2 K) cost is scaled to the whole batch's grid."""
    import oracle
    oracle.build()
    freqs = g.freqs()
    cores = oracle.max_threads()        # the threads its OpenMP loops actually run on
    nc = min(max_curves, b.n_curves)
    sub = b.subset(range(nc))
    k_sample = 256
    st = np.full(nc, 0.3)
    # calibrate on a small slice, then size the sample to about target_s
    t0 = time.perf_counter()
    oracle.batch_nckp(sub, st, freqs[:: max(1, len(freqs) // 32)][:32])
    dt = time.perf_counter() - t0
    k_sample = int(np.clip(32 * target_s / max(dt, 1e-3), 16, len(freqs)))
    fs = freqs[np.linspace(0, len(freqs) - 1, k_sample).astype(np.int64)]
    t0 = time.perf_counter()
    oracle.batch_nckp(sub, st, fs)
    dt = time.perf_counter() - t0
    n2k_sample = float(np.sum(sub.sizes.astype(np.float64) ** 2)) * k_sample
    if getattr(g, "bands", False):
        # the whole bands search (windows + nCKP at the trials) on the sampled curves, per curve
        t0 = time.perf_counter()
        oracle.batch_best(sub, g, sigma_t_mode=2)
        dt = time.perf_counter() - t0
        return {"value": nc / dt, "unit": "lightcurves/s", "cores": min(cores, nc), "kind": "oracle",
                "sample": "%d curves, whole bands search (FP64 spectral windows and N^2 double loop at the "
                          "trials, OpenMP over curves), %.1f s" % (nc, dt), "seconds": dt}
    if g.hierarchical:
        kc = int(np.floor((g.f_max - g.f_min) / g.coarse_df + 0.5)) + 1
        k_full = kc + g.top_k * (2 * int(round(g.fine_halfwidth / g.fine_df)) + 1)
    else:
        k_full = g.n_freq
    n2k_full = float(np.sum(b.sizes.astype(np.float64) ** 2)) * k_full
    lc_s = b.n_curves / (dt * n2k_full / n2k_sample)
    return {"value": lc_s, "unit": "lightcurves/s", "cores": cores, "kind": "oracle",
            "sample": "%d curves x %d of %d frequencies (FP64 N^2 double loop, OpenMP over curve-frequency), "
                      "%.1f s; scaled by sum N^2 K to the whole batch" % (nc, k_sample, k_full, dt),
            "seconds": dt}


def run_reference(args):
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return
    # rank 0 runs alone: give the oracle every host core (torchrun sets OMP_NUM_THREADS=1
    # per rank; the variable is read when the oracle library is loaded, below)
    if int(os.environ.get("WORLD_SIZE", "1")) > 1:
        os.environ["OMP_NUM_THREADS"] = str(os.cpu_count() or 1)
    b, g, name = make_workload(args, 0)
    per_step = []
    for _ in range(args.warmup + args.steps):
        per_step.append(cpu_baseline(b, g, target_s=8.0))
    timed = per_step[args.warmup:]
    v = float(np.mean([r["value"] for r in timed]))
    cb = dict(timed[-1])
    cb["value"] = v
    line = {"impl": "reference", "metric": "lightcurves/s", "value": v, "unit": "lightcurves/s",
            "n_gpus": args.gpus, "steps": args.steps, "warmup": args.warmup,
            "ms_per_step": float(np.mean([r["seconds"] for r in timed]) * 1e3), "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": {"workload": name, "form": "oracle", "l2": "n/a (host)"},
            "cpu_baseline": cb,
            "e2e": {"value": v, "unit": "lightcurves/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)


def main():
    args = parse()
    if args.impl == "reference":
        run_reference(args)
        return
    import torch
    import paper_1412_1840_gb300 as cp
    from paper_1412_1840_gb300.shard import curve_ranges, gather_results, local_csr, max_over_ranks
    DTYPES = {"fp16": cp.CP_DTYPE_FP16, "bf16": cp.CP_DTYPE_BF16, "bf16split": cp.CP_DTYPE_BF16_SPLIT}

    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    dist = None
    if world > 1:
        import torch.distributed as dist
        torch.cuda.set_device(local)
        dist.init_process_group("nccl")
    dev = torch.device("cuda", local)
    torch.cuda.set_device(dev)
    shard = None
    if args.shard:
        # one global batch (every rank draws the same one), a contiguous curve range per rank
        full, g, name = make_workload(args, 0)
        shard = curve_ranges(full.offsets, world)
        a0, a1 = shard[rank]
        t_, m_, e_, off_ = local_csr(full.times, full.mags, full.errs, full.offsets, (a0, a1))
        b = synth.Batch(t_, m_, e_, off_, full.period[a0:a1], full.periodic[a0:a1], full.kind[a0:a1])
        n_job = full.n_curves
        del full
    else:
        b, g, name = make_workload(args, rank)
        n_job = world * b.n_curves              # every rank its own batch of the same shape
    form = cp.CP_FORM_TENSOR if args.form == "tensor" else cp.CP_FORM_DIRECT
    grid = cp.grid_from(g)
    stream = torch.cuda.current_stream(dev)
    flush = torch.empty(256 << 20, dtype=torch.uint8, device=dev)   # > 129 MB L2

    def barrier():
        if dist is not None:
            dist.barrier()
        torch.cuda.synchronize(dev)

    # ---- device-resident inputs ------------------------------------------
    td = torch.from_numpy(b.times).to(dev)
    md = torch.from_numpy(b.mags).to(dev)
    ed = torch.from_numpy(b.errs).to(dev)
    tuning = None
    if args.tuning != "none" and os.path.exists(args.tuning):
        tuning = cp.tuning_from(args.tuning)
    tkw = dict(n_max=args.n_max, dtype=DTYPES[args.dtype], tuning=tuning)
    plan = cp.Plan(td, md, ed, b.offsets, grid, sigma_t_mode=cp.CP_SIGMA_T_RULE, form=form,
                   device=local, stream=stream.cuda_stream, **tkw)
    n = b.n_curves
    idx = np.empty(n, np.int64); bf = np.empty(n, np.float64); bs = np.empty(n, np.float32)
    per = np.empty(n, np.uint8); ps = np.empty(n, np.float32)
    for _ in range(args.warmup):
        plan.best_period_into(idx, bf, bs, per, ps)
    ev0 = [torch.cuda.Event(enable_timing=True) for _ in range(args.steps)]
    ev1 = [torch.cuda.Event(enable_timing=True) for _ in range(args.steps)]
    pair_ms = []
    barrier()
    with ClockSampler(local) as clk:
        for k in range(args.steps):
            flush.fill_(k & 0xff)
            ev0[k].record(stream)
            plan.best_period_into(idx, bf, bs, per, ps)
            ev1[k].record(stream)
            pair_ms.append(plan.info()["last_pair_kernel_ms"])
        barrier()
    step_ms = [ev0[k].elapsed_time(ev1[k]) for k in range(args.steps)]
    info = plan.info()
    sigma_t = plan.curve_stats()["sigma_t"]
    total_s = max_over_ranks(sum(step_ms) / 1e3, device=dev)
    value = n_job * args.steps / total_s
    plan.close()

    # ---- per-curve transforms around the search (Sections 5.2 and 7.1) ----
    transforms = None
    if not args.no_transforms:
        def timed_ms(fn, reps=3):
            fn()
            ts = []
            for _ in range(reps):
                e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                e0.record(stream)
                fn()
                e1.record(stream)
                torch.cuda.synchronize(dev)
                ts.append(e0.elapsed_time(e1))
            return float(np.median(ts))
        p0 = np.where(bf > 0, 1.0 / np.where(bf > 0, bf, 1.0), 0.0)
        wout = torch.empty_like(md)
        prep_ms = timed_ms(lambda: cp.cp_preprocess(td, md, ed, b.offsets, stream=stream.cuda_stream))
        whiten_ms = timed_ms(lambda: cp.cp_whiten(td, md, b.offsets, p0, out=wout, stream=stream.cuda_stream))
        transforms = {"preprocess": {"value": n / (prep_ms * 1e-3), "unit": "lightcurves/s", "ms": prep_ms,
                                     "includes": "offsets H2D, per-curve summaries D2H (synchronous call)"},
                      "whiten": {"value": n / (whiten_ms * 1e-3), "unit": "lightcurves/s", "ms": whiten_ms,
                                 "p0": "best periods of the timed search"}}

    # ---- end to end through host buffers ---------------------------------
    e2e = None
    if not args.no_e2e:
        tp = torch.from_numpy(b.times).pin_memory()
        mp = torch.from_numpy(b.mags).pin_memory()
        ep = torch.from_numpy(b.errs).pin_memory()
        hplan = cp.Plan(tp, mp, ep, b.offsets, grid, sigma_t_mode=cp.CP_SIGMA_T_RULE, form=form,
                        device=local, stream=stream.cuda_stream, **tkw)
        hplan.best_period_into(idx, bf, bs, per, ps)
        e_steps = max(1, min(args.steps, 2))
        barrier()
        t0 = time.perf_counter()
        for _ in range(e_steps):
            hplan.best_period_into(idx, bf, bs, per, ps)
        barrier()
        e_s = max_over_ranks(time.perf_counter() - t0, device=dev)
        hplan.close()
        h2d = b.times.nbytes + b.mags.nbytes + b.errs.nbytes
        d2h = idx.nbytes + bf.nbytes + bs.nbytes + per.nbytes + ps.nbytes + 8
        e2e = {"value": n_job * e_steps / e_s, "unit": "lightcurves/s", "h2d_bytes_per_step": int(h2d),
               "d2h_bytes_per_step": int(d2h), "steps": e_steps}

    # ---- tensor-core form on the same resident batch ---------------------
    tensor = None
    if not args.no_tensor and args.form == "direct":
        tkw2 = dict(n_max=args.n_max, dtype=DTYPES[args.dtype], tuning=tuning)
        tplan = cp.Plan(td, md, ed, b.offsets, grid, sigma_t_mode=cp.CP_SIGMA_T_RULE, form=cp.CP_FORM_TENSOR,
                        device=local, stream=stream.cuda_stream, **tkw2)
        tidx = np.empty(n, np.int64); tbf = np.empty(n, np.float64); tbs = np.empty(n, np.float32)
        tper = np.empty(n, np.uint8); tps = np.empty(n, np.float32)
        for _ in range(max(1, min(args.warmup, 3))):
            tplan.best_period_into(tidx, tbf, tbs, tper, tps)
        t_steps = args.steps                   # the same timed steps as the direct form
        te0 = [torch.cuda.Event(enable_timing=True) for _ in range(t_steps)]
        te1 = [torch.cuda.Event(enable_timing=True) for _ in range(t_steps)]
        tk_ms = []
        barrier()
        with ClockSampler(local) as tclk:
            for k in range(t_steps):
                flush.fill_(k & 0xff)
                te0[k].record(stream)
                tplan.best_period_into(tidx, tbf, tbs, tper, tps)
                te1[k].record(stream)
                ti = tplan.info()
                tk_ms.append(ti["last_tensor_kernel_ms"])
            barrier()
        t_total = max_over_ranks(sum(te0[k].elapsed_time(te1[k]) for k in range(t_steps)) / 1e3, device=dev)
        tplan.close()
        peaks = measured_peaks()
        tflops = ti["tensor_flops_search"] / (np.mean(tk_ms) / 1e3) / 1e12
        rel = np.abs(tbs.astype(np.float64) - bs) / np.maximum(np.abs(bs.astype(np.float64)), 1e-30)
        tensor = {
            "value": n_job * t_steps / t_total, "unit": "lightcurves/s",
            "ms_per_step": t_total * 1e3 / t_steps, "steps": t_steps,
            "dtype": args.dtype, "n_max": "per curve (8/12/16/32/48 by truncation tail <= 1e-4)" if args.n_max == 0
            else args.n_max,
            "class_curves": dict(zip(["direct", "n4", "n8", "n12", "n16", "n32", "n48"], ti["class_curves"])),
            "best_idx_agreement_vs_direct": float(np.mean(tidx == idx)),
            "best_stat_max_rel_diff_vs_direct": float(rel.max()),
            "within_1e-3_of_direct": bool(rel.max() <= 1e-3),
            "clocks": tclk.summary(),
            "roofline": {"bound": "tensor", "achieved": tflops,
                         "peak": peaks["bf16_tflops_sustained"], "unit": "TFLOP/s",
                         "frac": tflops / peaks["bf16_tflops_sustained"],
                         "traffic": DRAM_PER_W_BYTE_TENSOR * ti["w_bytes_tensor"],
                         "kernel": "k_pair_tensor", "flops_basis": "2 N^2 n_max per curve-frequency (upper block "
                         "triangle of the 4 N^2 n_max dense GEMM)",
                         "peak_basis": "bf16 dense sustained, %s (fp16 has the same nominal rate)" % peaks["source"],
                         "avg_launch_ms": float(np.mean(tk_ms))},
        }
        # the tensor form end to end through the same pinned host buffers
        if e2e is not None:
            thplan = cp.Plan(tp, mp, ep, b.offsets, grid, sigma_t_mode=cp.CP_SIGMA_T_RULE, form=cp.CP_FORM_TENSOR,
                             device=local, stream=stream.cuda_stream, **tkw2)
            thplan.best_period_into(tidx, tbf, tbs, tper, tps)
            barrier()
            t0 = time.perf_counter()
            te_steps = max(1, min(args.steps, 3))
            for _ in range(te_steps):
                thplan.best_period_into(tidx, tbf, tbs, tper, tps)
            barrier()
            te_s = max_over_ranks(time.perf_counter() - t0, device=dev)
            thplan.close()
            tensor["e2e"] = {"value": n_job * te_steps / te_s, "unit": "lightcurves/s",
                             "h2d_bytes_per_step": int(h2d), "d2h_bytes_per_step": int(d2h), "steps": te_steps}
        # the other 16-bit operand types on the same batch (same plan shape, a few timed steps)
        operands = {"fp16": "FP16",
                    "bf16": "W' as hi + lo BF16 parts (two MMAs per K slice), Z one BF16 part",
                    "bf16split": "W' and Z both as hi + lo BF16 parts (Z's lo part in the upper half of the MMA "
                                 "columns: two MMAs per K slice over half the frequencies per unit)"}
        tensor["other_dtypes"] = []
        for oname in [d for d in ("fp16", "bf16", "bf16split") if d != args.dtype]:
            oplan = cp.Plan(td, md, ed, b.offsets, grid, sigma_t_mode=cp.CP_SIGMA_T_RULE, form=cp.CP_FORM_TENSOR,
                            device=local, stream=stream.cuda_stream, n_max=args.n_max, dtype=DTYPES[oname],
                            tuning=tuning)
            oplan.best_period_into(tidx, tbf, tbs, tper, tps)
            o_steps = max(1, min(args.steps, 3))
            barrier()
            o_ms = []
            for k in range(o_steps):
                oe0, oe1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                flush.fill_(7 + k)
                oe0.record(stream)
                oplan.best_period_into(tidx, tbf, tbs, tper, tps)
                oe1.record(stream)
                barrier()
                o_ms.append(oe0.elapsed_time(oe1))
            oi = oplan.info()
            o_s = max_over_ranks(sum(o_ms) / 1e3, device=dev)
            oplan.close()
            orel = np.abs(tbs.astype(np.float64) - bs) / np.maximum(np.abs(bs.astype(np.float64)), 1e-30)
            otf = oi["tensor_flops_search"] / (oi["last_tensor_kernel_ms"] / 1e3) / 1e12
            tensor["other_dtypes"].append({
                "dtype": oname, "value": n_job * o_steps / o_s, "unit": "lightcurves/s",
                "ms_per_step": o_s * 1e3 / o_steps, "steps": o_steps,
                "class_curves": dict(zip(["direct", "n4", "n8", "n12", "n16", "n32", "n48"], oi["class_curves"])),
                "best_idx_agreement_vs_direct": float(np.mean(tidx == idx)),
                "best_stat_max_rel_diff_vs_direct": float(orel.max()),
                "within_1e-3_of_direct": bool(orel.max() <= 1e-3),
                "operands": operands[oname], "tensor_tflops_algorithmic": otf})

    # ---- coarse-then-fine search on the same batch (both forms) -------------
    hier = None
    if not args.no_hierarchical and args.workload == "ragged" and shard is None:
        hb, hg = synth.workload_hierarchical(n, args.seed + 1000 * rank)
        assert np.array_equal(hb.offsets, b.offsets) and np.array_equal(hb.mags, b.mags)   # the same batch
        hgrid = cp.grid_from(hg)
        hidx = np.empty(n, np.int64); hbf = np.empty(n, np.float64); hbs = np.empty(n, np.float32)
        hper = np.empty(n, np.uint8); hps = np.empty(n, np.float32)
        hier = {"workload": "%d curves N~U[300,1000] seasonal 2500 d; coarse 0.002-5 step 1e-3 (4,999), top-10 "
                            "refined at 1e-5 over +-2e-3 (401 each)" % n}
        for fname, fkw in (("direct", dict(form=cp.CP_FORM_DIRECT)),
                           ("tensor", dict(form=cp.CP_FORM_TENSOR, n_max=args.n_max, dtype=cp.CP_DTYPE_FP16))):
            hp = cp.Plan(td, md, ed, hb.offsets, hgrid, sigma_t_mode=cp.CP_SIGMA_T_RULE, device=local,
                         stream=stream.cuda_stream, tuning=tuning, **fkw)
            hp.best_period_into(hidx, hbf, hbs, hper, hps)
            h_steps = max(1, min(args.steps, 5))
            ms, km = [], []
            barrier()
            for k in range(h_steps):
                e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                flush.fill_(k & 0xff)
                e0.record(stream)
                hp.best_period_into(hidx, hbf, hbs, hper, hps)
                e1.record(stream)
                barrier()
                ms.append(e0.elapsed_time(e1))
                hi_ = hp.info()
                km.append(hi_["last_tensor_kernel_ms"] if fname == "tensor" else hi_["last_pair_kernel_ms"])
            hp.close()
            h_s = max_over_ranks(sum(ms) / 1e3, device=dev)
            ent = {"value": n * h_steps / h_s, "unit": "lightcurves/s", "steps": h_steps,
                   "ms_per_step": h_s * 1e3 / h_steps, "launches_per_search": int(hi_["launches_per_search"]),
                   **pair_freq(hi_, h_s / h_steps)}
            if fname == "tensor":
                ent["roofline_frac"] = hi_["tensor_flops_search"] / (np.mean(km) / 1e3) / 1e12 / \
                    measured_peaks()["bf16_tflops_sustained"]
                ent["dtype"] = "fp16"
            elif hi_["w_bytes_direct"]:        # every frequency by the pair sum
                ent["roofline_frac"] = hi_["pair_freq_search"] / (np.mean(km) / 1e3) / \
                    (sfu_ex2_per_clk_sm() * hi_["n_sm"] * SM_MAX_MHZ * 1e6)
            hier[fname] = ent

    # ---- the 200,000-curve two-band throughput run (both forms) -----------
    thr = None
    if not args.no_throughput and args.workload == "ragged" and shard is None and world == 1:
        del td, md, ed
        torch.cuda.empty_cache()
        t_gen = time.perf_counter()
        tb, tg = synth.workload_throughput(100000, 5)
        t_gen = time.perf_counter() - t_gen
        ttd = torch.from_numpy(tb.times).to(dev)
        tmd = torch.from_numpy(tb.mags).to(dev)
        ted = torch.from_numpy(tb.errs).to(dev)
        tn = tb.n_curves
        ti_ = np.empty(tn, np.int64); tf_ = np.empty(tn, np.float64); ts_ = np.empty(tn, np.float32)
        tp_ = np.empty(tn, np.uint8); tq_ = np.empty(tn, np.float32)
        thr = {"workload": "100,000 two-band sources (200,000 curves) N~U[200,1000] per band, SNR 0.2-10, seed 5; "
                           "coarse 0.002-5 step 1e-3, top-10 refined at 1e-5 over +-2e-3",
               "generator_s": t_gen}
        res = {}
        for fname, fkw, warm in (("tensor", dict(form=cp.CP_FORM_TENSOR, n_max=args.n_max, dtype=cp.CP_DTYPE_FP16), 1),
                                 ("direct", dict(form=cp.CP_FORM_DIRECT), 0)):
            tpl = cp.Plan(ttd, tmd, ted, tb.offsets, cp.grid_from(tg), sigma_t_mode=cp.CP_SIGMA_T_RULE,
                          device=local, stream=stream.cuda_stream, tuning=tuning, **fkw)
            for _ in range(warm):
                tpl.best_period_into(ti_, tf_, ts_, tp_, tq_)
            barrier()
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record(stream)
            tpl.best_period_into(ti_, tf_, ts_, tp_, tq_)
            e1.record(stream)
            barrier()
            t_ms = e0.elapsed_time(e1)
            tinfo = tpl.info()
            tpl.close()
            res[fname] = ts_.copy()
            ent = {"value": tn / (t_ms / 1e3), "unit": "lightcurves/s", "steps": 1, "warmup": warm,
                   "ms_per_step": t_ms, **pair_freq(tinfo, t_ms / 1e3)}
            if fname == "tensor":
                ent["dtype"] = "fp16"
                ent["roofline_frac"] = tinfo["tensor_flops_search"] / (tinfo["last_tensor_kernel_ms"] / 1e3) / 1e12 / \
                    measured_peaks()["bf16_tflops_sustained"]
            else:
                ent["note"] = "no warm-up step (kernels already loaded by the runs above; the first call " \
                              "instantiates its CUDA graph inside the timed step)"
                if tinfo["w_bytes_direct"]:
                    ent["roofline_frac"] = tinfo["pair_freq_search"] / (tinfo["last_pair_kernel_ms"] / 1e3) / \
                        (sfu_ex2_per_clk_sm() * tinfo["n_sm"] * SM_MAX_MHZ * 1e6)
            thr[fname] = ent
        rel = np.abs(res["tensor"].astype(np.float64) - res["direct"]) / \
            np.maximum(np.abs(res["direct"].astype(np.float64)), 1e-30)
        thr["tensor_best_stat_max_rel_diff_vs_direct"] = float(rel.max())
        # the coarse top-10 cutoff can rank near-tied peaks differently within 1e-3, and then the two
        # forms refine different peaks: per-curve agreement is the fraction, the oracle test the bar
        thr["tensor_best_stat_within_1e-3_of_direct_frac"] = float(np.mean(rel <= 1e-3))
        thr["agreement_with_oracle"] = "tests/test_gpu_agreement.py: fixed 1,000-curve sample of this generator"
        del ttd, tmd, ted

    gathered = None
    if shard is not None:
        # every rank's best periods, in global curve order (host-side, after the timed region)
        gathered = int(gather_results({"best_idx": idx}, world)["best_idx"].shape[0])
        pf_job = float(np.sum(gather_results({"pf": np.array([info["pair_freq_search"]])}, world)["pf"]))
    if rank != 0:
        if dist is not None:
            dist.destroy_process_group()
        return
    clocks = clk.summary()
    pf = info["pair_freq_search"]
    pair_s = np.mean(pair_ms) / 1e3
    achieved = pf / pair_s / 1e9                       # Gex2/s: one ex2 per pair-frequency evaluation
    ex2_clk = sfu_ex2_per_clk_sm()
    peak = ex2_clk * info["n_sm"] * SM_MAX_MHZ * 1e6 / 1e9
    line = {
        "metric": "lightcurves/s", "value": value, "unit": "lightcurves/s", "n_gpus": world,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": float(np.mean(step_ms)),
        "higher_is_better": True, "scaling": "strong" if shard is not None else "weak", "vs_baseline": None,
        "dtype": "f32" if args.form == "direct" else args.dtype,
        "data": "synthetic",
        "config": {"workload": name, "form": args.form, "sigma_t": "Bowley-skewness rule",
                   "curves_per_gpu": n, "l2": "flushed between steps (256 MB write)",
                   "tuning": os.path.basename(args.tuning) if tuning is not None else "built-in",
                   "parallelism": ("one batch split by pair-sum cost across %d GPUs (curve ranges %s)"
                                   % (world, shard)) if shard is not None else "independent curve batches per GPU"},
        **pair_freq(info, total_s / args.steps, world if shard is None else pf_job / pf),
        "gpu_launches": int(info["launches_per_search"]) * args.steps,
        "e2e": e2e,
        "roofline": {"bound": "alu", "achieved": achieved, "peak": peak, "unit": "Gex2/s",
                     "frac": achieved / peak, "traffic": DRAM_PER_W_BYTE_DIRECT * info["w_bytes_direct"],
                     "kernel": "k_pair_direct",
                     "peak_basis": "%.2f MUFU ex2/clk/SM (measured by paper_1412_1840_gb300.peaks on GB300) x %d SMs "
                                   "x %.0f MHz (max SM clock)" % (ex2_clk, info["n_sm"], SM_MAX_MHZ),
                     "avg_launch_ms": float(np.mean(pair_ms))},
        "clocks": clocks,
    }
    if args.form == "direct" and not info["w_bytes_direct"]:      # through the pair spectrum
        peaks = measured_peaks()
        line["roofline"] = {"bound": "hbm", "peak": peaks["hbm_gbs"], "unit": "GB/s", "kernel": "k_spec_*",
                            "peak_basis": "copy bandwidth, " + peaks["source"], "avg_launch_ms": float(np.mean(pair_ms))}
        if not (g.hierarchical or getattr(g, "bands", False)):
            least = spectrum_bytes(sigma_t, g)
            line["roofline"].update(achieved=least / pair_s / 1e9, frac=least / pair_s / 1e9 / peaks["hbm_gbs"],
                                    traffic=least, traffic_basis="least traffic of the transforms (not measured)")
    if args.form == "tensor":
        peaks = measured_peaks()
        tflops = info["tensor_flops_search"] / (info["last_tensor_kernel_ms"] / 1e3) / 1e12
        line["roofline"] = {"bound": "tensor", "achieved": tflops, "peak": peaks["bf16_tflops_sustained"],
                            "unit": "TFLOP/s", "frac": tflops / peaks["bf16_tflops_sustained"],
                            "traffic": DRAM_PER_W_BYTE_TENSOR * info["w_bytes_tensor"],
                            "kernel": "k_pair_tensor", "peak_basis": "bf16 dense sustained, " + peaks["source"],
                            "avg_launch_ms": float(info["last_tensor_kernel_ms"])}
    if shard is not None:
        line["shard"] = {"ranges": shard, "gathered_curves": gathered}
    if tensor is not None:
        line["tensor"] = tensor
    if hier is not None:
        line["hierarchical"] = hier
    if thr is not None:
        line["throughput"] = thr
    if transforms is not None:
        line["transforms"] = transforms
    if getattr(g, "bands", False):
        line["bands"] = {"kernels": "k_bands + k_window + k_window_refine", "ms_per_step": float(info["last_bands_kernel_ms"]),
                         "window_terms_per_s": info["window_terms_search"] / (info["last_bands_kernel_ms"] / 1e3),
                         "trials_per_curve": int(g.n_bands * g.trials_per_band)}
    if not args.no_cpu_baseline and world == 1:
        line["cpu_baseline"] = cpu_baseline(b, g)
        line["cpu_baseline"].pop("seconds", None)
    print(json.dumps(line), flush=True)
    if dist is not None:
        dist.destroy_process_group()


if __name__ == "__main__":
    main()
