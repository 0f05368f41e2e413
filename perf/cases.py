"""Performance cases of the correntropy kernelized periodogram.

Each case is one call that a period search makes through the public entry
points: the periodogram and the best-period search of a batch of lightcurves
(direct FP32 form and the 16-bit tensor form), the coarse-then-fine and the
bands search, the call that allocates nothing, and the per-curve transforms
before and after a search (cleaning and whitening).  Sizes are those of the
repository's workloads (150 samples on 9,991 frequencies; 300 to 1000 samples
on 0.002-5 1/day in steps of 1e-4; coarse 1e-3 with ten windows at 1e-5; the
bands method with 3 bands and 150 trials) on batches that keep a pass below a
second, and the smallest and longest curves that the entry points take.
"""
import math

import numpy as np
import torch

import paper_1412_1840_gb300 as cp

YEAR, SEASON = 365.25, 243.5      # seasonal sampling: eight months of each year

DTYPES = {"fp16": cp.CP_DTYPE_FP16, "bf16": cp.CP_DTYPE_BF16}


def _case(kind, curves, n_lo, n_hi, f_min=0.002, df=1e-4, n_freq=49981, sigma_t=0.0, span=2500.0, memory="device",
          form="direct", **more):
    """sigma_t = 0 is the skewness rule (a value for every curve from its magnitudes)."""
    return dict(kind=kind, curves=curves, n_lo=n_lo, n_hi=n_hi, span=span, f_min=f_min, df=df, n_freq=n_freq,
                sigma_t=sigma_t, memory=memory, form=form, **more)


def listed():
    hier = dict(coarse_df=1e-3, top_k=10, fine_df=1e-5, fine_halfwidth=2e-3)
    return [
        # one star looked at interactively: launches and latency
        dict(_case("search", 1, 150, 150, 0.002, 2e-4, 9991, 0.3, 1000.0), name="single_search"),
        # a small request from numpy arrays: short curves, a short grid, copies included
        dict(_case("search", 64, 40, 200, 0.01, 1e-3, 2000, 0.0, 1500.0, "host"), name="small_batch_host"),
        # a handful of stars whose whole periodogram is wanted (plots, later statistics)
        dict(_case("periodogram", 12, 300, 1000), name="ragged_periodogram"),
        # the survey's work: the best period of every curve on the full grid
        dict(_case("search", 384, 300, 1000), name="ragged_search"),
        # well observed fields, long periods: few, long curves up to the largest size
        dict(_case("periodogram", 3, 2000, 4096, 0.002, 1e-4, 4981, 0.45), name="long_periodogram"),
        # the throughput search: coarse grid, then windows around its peaks
        dict(_case("coarse_fine", 256, 200, 1000, **hier), name="coarse_fine_search"),
        # the paper's trial-period extraction, then the statistic at its trials
        dict(_case("bands", 256, 300, 1000, 0.00125, 1e-4, 29988, n_bands=3, n_trials=150), name="bands_search"),
        # the 16-bit tensor form, both operand types
        dict(_case("periodogram", 16, 300, 1000, n_freq=19981, form="fp16"), name="tensor_fp16_periodogram"),
        dict(_case("periodogram", 24, 200, 800, n_freq=9981, form="bf16"), name="tensor_bf16_periodogram"),
        # a host that cannot allocate at call time
        dict(_case("noalloc", 8, 40, 420, 0.01, 1e-3, 900, 0.3), name="noalloc_search"),
        # cleaning a field before its search, and removing the first mode after it
        dict(_case("preprocess", 2048, 60, 1000), name="preprocess_field"),
        dict(_case("whiten", 2048, 200, 1000), name="whiten_field"),
    ]


def draw(rng):
    def log(lo, hi):
        return math.exp(rng.uniform(math.log(lo), math.log(hi)))

    kind = rng.choice(["search", "search", "periodogram", "periodogram", "coarse_fine", "bands", "tensor", "noalloc",
                       "transform"])
    n_hi = int(log(60, 4096)) if kind in ("search", "periodogram") else int(log(100, 1500))
    n_lo = max(40, int(n_hi * rng.uniform(0.2, 1.0)))
    n_hi = max(n_lo, n_hi)
    span = rng.choice([700.0, 1000.0, 1500.0, 2500.0, 3652.5])
    # steps as they are chosen: a round number, or a fraction of the resolution 1 / span
    df = rng.choice([1e-4, 2e-4, 5e-4, 1.0 / (5.0 * span)])
    # the lowest frequency: a round number, half a step, or one cycle in the span
    f_min = rng.choice([round(log(0.001, 0.1), 4), 0.5 * df, 1.0 / span])
    f_max = rng.choice([1.0, 2.0, 3.0, 5.0])
    n_freq = max(200, int((f_max - f_min) / df * rng.uniform(0.5, 1.0)))
    sigma_t = rng.choice([0.0, 0.0, 0.3, round(log(0.1, 0.6), 3)])
    memory = rng.choice(["device", "device", "host"])
    size = 0.4 * n_hi * n_hi * n_freq          # pair terms of one curve, about
    curves = int(min(log(1, 400), max(1.0, 1e12 / size)))
    if kind == "coarse_fine":
        return _case(kind, int(log(1, 256)), n_lo, n_hi, f_min, 1e-4, int((f_max - f_min) / 1e-4), sigma_t, span, memory,
                     coarse_df=rng.choice([5e-4, 1e-3, 2e-3]), top_k=rng.choice([3, 5, 10]), fine_df=1e-5,
                     fine_halfwidth=rng.choice([1e-3, 2e-3]))
    if kind == "bands":
        return _case(kind, int(log(1, 256)), n_lo, n_hi, 0.00125, 1e-4, int(log(3000, 29988)), sigma_t, span, memory,
                     n_bands=rng.randint(1, 4), n_trials=rng.choice([20, 100, 150]))
    if kind == "tensor":
        n_freq = min(n_freq, 20000)
        return _case("periodogram", int(log(2, 48)), n_lo, n_hi, f_min, df, n_freq, 0.0, span, "device",
                     rng.choice(["fp16", "bf16"]))
    if kind == "noalloc":
        return _case(kind, rng.randint(1, 16), n_lo, min(n_hi, 600) if n_lo < 600 else n_lo, 0.01, 1e-3,
                     int(log(200, 3000)), rng.choice([0.25, 0.3, 0.45]), span)
    if kind == "transform":
        return _case(rng.choice(["preprocess", "whiten"]), int(log(4, 4096)), n_lo, n_hi, span=span)
    return _case(kind, curves, n_lo, n_hi, f_min, df, n_freq, sigma_t, span, memory)


# ---- inputs ------------------------------------------------------------------

def _lightcurves(case, seed):
    """Seasonally sampled curves: half of them periodic (sinusoid with
    harmonics, sawtooth or eclipses, periods 0.2 to 500 days), half noise or a
    slow drift; error bars of 0.02 to 0.3 mag."""
    sizes = np.random.default_rng([case["curves"], case["n_lo"], case["n_hi"]]).integers(
        case["n_lo"], case["n_hi"] + 1, case["curves"])      # the case's, so that outputs keep their shapes
    rng = np.random.default_rng([int(seed), 77])
    starts = np.arange(0.0, case["span"], YEAR)
    lens = np.minimum(SEASON, case["span"] - starts)
    edges = np.concatenate([[0.0], np.cumsum(lens)])
    ts, ms, es, periods = [], [], [], []
    for n in sizes:
        u = np.sort(rng.uniform(0.0, edges[-1], n))
        w = np.clip(np.searchsorted(edges, u, side="right") - 1, 0, len(lens) - 1)
        t = starts[w] + (u - edges[w])
        period = float(np.exp(rng.uniform(np.log(0.2), np.log(500.0))))
        phase = np.mod(t / period + rng.uniform(), 1.0)
        shape = int(rng.integers(0, 6))
        if shape == 0:
            y = np.sin(2 * np.pi * phase) + rng.uniform(0, 0.6) * np.sin(4 * np.pi * phase + 1.0)
        elif shape == 1:
            y = 2.0 * phase - 1.0
        elif shape == 2:
            y = np.where(phase < rng.uniform(0.03, 0.15), 1.0, np.where(np.abs(phase - 0.5) < 0.03, 0.4, 0.0))
        elif shape == 3:
            y = np.sin(2 * np.pi * t / 2000.0 + 6.0 * rng.uniform()) + 0.3 * rng.standard_normal(n)
        else:
            y = rng.standard_normal(n)
        e0 = np.exp(rng.uniform(np.log(0.02), np.log(0.3)))
        e = np.maximum(e0 * (1.0 + 0.1 * rng.standard_normal(n)), 0.5 * e0)
        if case["kind"] == "preprocess":          # bad error bars and a trend, as raw photometry has
            e[rng.permutation(n)[:max(1, n // 100)]] *= 8.0
            y = y + (2e-3 * t if rng.uniform() < 0.3 else 0.0)
        ts.append(t)
        ms.append(rng.uniform(15.0, 20.0) + rng.uniform(0.05, 1.0) * y + e * rng.standard_normal(n))
        es.append(e)
        periods.append(period)
    offsets = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    return (np.concatenate(ts), np.concatenate(ms).astype(np.float32), np.concatenate(es).astype(np.float32), offsets,
            np.array(periods))


def _grid(case):
    more = {}
    if case["kind"] == "coarse_fine":
        more = dict(hierarchical=True, coarse_df=case["coarse_df"], top_k=case["top_k"], fine_df=case["fine_df"],
                    fine_halfwidth=case["fine_halfwidth"])
    if case["kind"] == "bands":
        more = dict(bands=True, n_bands=case["n_bands"], trials_per_band=case["n_trials"])
    return cp.make_grid(case["f_min"], case["df"], case["n_freq"], **more)


def prepare(case, seed):
    t, m, e, offsets, periods = _lightcurves(case, seed)
    if case["memory"] == "device":
        t, m, e = (torch.from_numpy(a).cuda() for a in (t, m, e))
    state = dict(case=case, t=t, m=m, e=e, offsets=offsets, periods=periods)
    n = case["curves"]
    if case["kind"] == "noalloc":
        state["grid"] = _grid(case)
        state["out"] = (torch.zeros(n, dtype=torch.int64, device="cuda"), torch.zeros(n, dtype=torch.float64, device="cuda"),
                        torch.zeros(n, dtype=torch.float32, device="cuda"), torch.zeros(n, dtype=torch.uint8, device="cuda"))
    elif case["kind"] not in ("preprocess", "whiten"):
        opt = dict(sigma_t=case["sigma_t"]) if case["sigma_t"] else dict(sigma_t_mode=cp.CP_SIGMA_T_RULE)
        if case["form"] != "direct":
            opt.update(form=cp.CP_FORM_TENSOR, dtype=DTYPES[case["form"]])
        state["plan"] = cp.cp_plan(t, m, e, offsets, _grid(case), **opt)
        if case["kind"] == "periodogram":
            state["out"] = torch.zeros((n, case["n_freq"]), dtype=torch.float32, device="cuda")
    return state


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "periodogram":
        return cp.cp_periodogram(state["plan"], state["out"])
    if kind == "preprocess":
        return cp.cp_preprocess(state["t"], state["m"], state["e"], state["offsets"])
    if kind == "whiten":
        return cp.cp_whiten(state["t"], state["m"], state["offsets"], state["periods"])
    if kind == "noalloc":
        cp.cp_best_period_noalloc(state["t"], state["m"], state["e"], state["offsets"], state["grid"], case["sigma_t"],
                                  *state["out"])
        return state["out"]
    best = cp.cp_best_period(state["plan"])
    if kind == "bands":
        return dict(best, **cp.cp_trial_frequencies(state["plan"]))
    return best


# ---- the least work ------------------------------------------------------------

def work(case):
    """Every sample is read once and every result written once.  Operations:
    the magnitude kernel of every pair of samples (about 4 each), and at every
    trial frequency the eight or more harmonics of the periodic kernel (2 each):
    how often the pairs are gone through for the frequencies is the method's
    choice, not the statistic's."""
    n = 0.5 * (case["n_lo"] + case["n_hi"])
    pairs = 0.5 * (case["n_lo"] ** 2 + case["n_lo"] * case["n_hi"] + case["n_hi"] ** 2) / 3.0
    c, kind = case["curves"], case["kind"]
    if kind == "preprocess":
        return {"bytes": 32.0 * n * c, "flops": 30.0 * n * c}
    if kind == "whiten":
        return {"bytes": 16.0 * n * c, "flops": n * c * (math.log2(n) + 6.0)}
    freqs = float(case["n_freq"])
    extra = 0.0
    if kind == "coarse_fine":
        freqs = freqs * case["df"] / case["coarse_df"] + case["top_k"] * (
            2.0 * round(case["fine_halfwidth"] / case["fine_df"]) + 1.0)
    if kind == "bands":      # the spectral window of each kept band: a tenth of the samples at every grid frequency
        extra = 8.0 * case["n_bands"] * freqs
        freqs = float(case["n_bands"] * case["n_trials"])
    out = 4.0 * freqs if kind == "periodogram" else 25.0 + (8.0 * freqs if kind == "bands" else 0.0)
    return {"bytes": c * (16.0 * n + out), "flops": c * (4.0 * pairs + 16.0 * freqs + extra)}


# ---- what the outputs are in 64 bits -------------------------------------------

def _sigma_t(y):
    s = np.sort(y)
    h = len(s) // 2
    q1, q2, q3 = np.median(s[:h]), np.median(s), np.median(s[len(s) - h:])
    skew = 0.0 if q3 == q1 else (q3 + q1 - 2.0 * q2) / (q3 - q1)
    return 0.1 + 0.5 * math.exp(-12.0 * skew * skew)


def _statistic(case, t, y, e, freqs):
    """nCKP of one curve at the given frequencies: the double sum over all pairs."""
    y = y.astype(np.float64)
    sy = float(np.median(e.astype(np.float64)))
    st = case["sigma_t"] or _sigma_t(y)
    n = len(t)
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    i, j = (torch.from_numpy(k).to(dev) for k in np.triu_indices(n, 1))
    tt, yy = (torch.from_numpy(np.ascontiguousarray(a)).to(dev) for a in (t - t.min(), y))
    g = torch.exp(-(yy[i] - yy[j]) ** 2 / (2.0 * sy * sy))
    ip = float((n + 2.0 * g.sum()) / (n * n))
    w = g - ip
    f = torch.from_numpy(freqs).to(dev)
    out = torch.empty(len(freqs), dtype=torch.float64, device=dev)
    step = max(1, (1 << 26) // len(i))
    for k in range(0, len(freqs), step):
        ph = torch.remainder(f[k:k + step, None] * tt[None, :], 1.0) * (2.0 * math.pi)
        c, s = torch.cos(ph), torch.sin(ph)
        x = c[:, i]
        x *= c[:, j]
        x.addcmul_(s[:, i], s[:, j])
        x -= 1.0
        x *= 1.0 / (st * st)
        out[k:k + step] = x.exp_() @ w
    total = n * (1.0 - ip) + 2.0 * out
    return (total * math.sqrt(n * st) / (n * n * ip * math.sqrt(2.0 * math.pi) * st)).cpu().numpy()


def _psnr(y, e):
    q = np.percentile(y.astype(np.float64), [25, 75])
    return 0.7413 * (q[1] - q[0]) / float(np.median(e.astype(np.float64)))


def exact(case, seed):
    t, m, e, offsets, periods = _lightcurves(case, seed)
    curves = [(t[a:b], m[a:b], e[a:b]) for a, b in zip(offsets[:-1], offsets[1:])]
    kind = case["kind"]
    if kind == "preprocess":
        outs = {"times": [], "mags": [], "errs": []}
        for tc, mc, ec in curves:
            e64 = ec.astype(np.float64)
            keep = e64 < e64.mean() + 3.0 * e64.std()
            if keep.sum() < 50:
                continue
            x, w, tk = mc[keep].astype(np.float64), 1.0 / e64[keep] ** 2, tc[keep]
            tm, xm = (w * tk).sum() / w.sum(), (w * x).sum() / w.sum()
            slope = (w * (tk - tm) * (x - xm)).sum() / (w * (tk - tm) ** 2).sum()
            fit = xm + slope * (tk - tm)
            r = np.corrcoef(x, fit)[0, 1]
            outs["times"].append(tk)
            outs["mags"].append(x - fit if r > 0.5 else x)
            outs["errs"].append(e64[keep])
        full = {k: np.concatenate(v + [np.zeros(0)]) for k, v in outs.items()}
        return dict(full, offsets=None, offsets_all=None, curve=None, flags=None, fit=None)
    if kind == "whiten":
        got = []
        for (tc, mc, _), p in zip(curves, periods):
            x = mc.astype(np.float64)
            order = np.argsort(np.mod(tc / p, 1.0), kind="stable")
            n, w = len(x), min(30, len(x))
            at = (np.arange(n)[:, None] - w // 2 + np.arange(w)[None, :]) % n
            y = np.empty(n)
            y[order] = x[order] - x[order][at].mean(axis=1)
            got.append(y)
        return np.concatenate(got)
    pairs = sum(0.5 * len(c[0]) ** 2 for c in curves)
    freqs = case["f_min"] + case["df"] * np.arange(case["n_freq"])
    whole = pairs * len(freqs) < 1.8e11 and kind in ("periodogram", "search", "noalloc")
    rows = [_statistic(case, *c, freqs) for c in curves] if whole else None
    if kind == "periodogram":
        return None if rows is None else np.stack(rows)
    stat = None if rows is None else np.array([r.max() for r in rows])
    if kind == "noalloc":
        return [None, None, stat, None]
    psnr = np.array([_psnr(c[1], c[2]) for c in curves])
    known = {"best_idx": None, "best_freq": None, "best_stat": stat, "is_periodic": None, "psnr": psnr}
    if kind == "bands":
        known.update(trial_idx=None, trial_stat=None)
    return known
