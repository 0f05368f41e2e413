"""Searches through the pair spectrum (csrc/cp_spec.cu) at the edges of its
paths, against the pair sum at every frequency and the FP64 oracle."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1412_1840_gb300 as cp  # noqa: E402

TOL = 1e-5     # of the curve's peak, the direct form's bar


@pytest.fixture(scope="module", autouse=True)
def _need_gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def search(b, g, rows=False, **kw):
    """Results of one search (and of a periodogram), and the plan's information."""
    dev = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (b.times, b.mags, b.errs)]
    with cp.Plan(*dev, b.offsets, cp.grid_from(g), **kw) as p:
        got = p.best_period()
        if g.bands:
            got = dict(got, **p.trials())
        if rows:
            out = torch.zeros((b.n_curves, g.n_freq), dtype=torch.float32, device="cuda")
            p.periodogram(out)
            p.sync()
            got["rows"] = out.cpu().numpy()
        return got, p.info()


def by_the_pair_sum(monkeypatch, b, g, **kw):
    """The same search on a plan that has room for the magnitude-kernel tiles, not for a spectrum."""
    nb = (np.diff(b.offsets) + 31) // 32
    tiles = int(np.sum(nb * (nb + 1) // 2)) * 4096
    room = tiles + 60 * int(b.offsets[-1]) + (768 << 10)
    if g.hierarchical:
        room += 8 * b.n_curves * int((g.n_freq - 1) * g.df / g.coarse_df + 2)
    with monkeypatch.context() as m:
        m.setenv("CP_FAIL_ALLOC_ABOVE_KB", str(room >> 10))
        got, info = search(b, g, **kw)
    assert info["w_bytes_direct"] == tiles
    return got


def same_search(got, want):
    for key in ("best_idx", "best_freq", "best_stat", "is_periodic"):
        np.testing.assert_array_equal(got[key], want[key], err_msg=key)


def strong_batch(n_curves, n, span, seed, integer):
    """Clean square waves of one period on curves of n samples; integer times tie f, 1 - f, 1 + f, ..."""
    rng = np.random.default_rng(seed)
    t = np.sort(rng.uniform(0.0, span, (n_curves, n)), axis=1)
    if integer:
        t = np.floor(t)
    y = 17.0 + (np.mod(t / 3.7 + rng.uniform(0, 1, (n_curves, 1)), 1.0) < 0.5) + 0.02 * rng.standard_normal(t.shape)
    off = np.arange(n_curves + 1, dtype=np.int64) * n
    return synth.Batch(t.ravel(), y.ravel().astype(np.float32), np.full(t.size, 0.1, np.float32), off,
                       np.full(n_curves, 3.7), np.ones(n_curves, bool), np.zeros(n_curves, np.int8))


@pytest.mark.parametrize("n,n_curves", [(400, 24), (4000, 6)])
@pytest.mark.parametrize("integer", [False, True])
@pytest.mark.parametrize("kw", [dict(), dict(hierarchical=True, coarse_df=5e-4, top_k=5, fine_df=2e-5, fine_halfwidth=1e-3),
                                dict(bands=True, n_bands=3, trials_per_band=150)])
def test_best_beside_excluded_peaks_is_the_pair_sums(monkeypatch, n, n_curves, integer, kw):
    """Windows over every frequency above a tenth of the peak: what is left to
    choose from is below the largest values of the row, whose rounding it
    carries; the best is the pair sum's, bit for bit."""
    b = strong_batch(n_curves, n, 1500.0, 91, integer)
    g0 = synth.Grid(0.2, 2e-4, 1500)
    got, info = search(b, g0, rows=True, sigma_t=0.3)
    assert info["w_bytes_direct"] == 0
    rows = got["rows"]
    high = np.flatnonzero((rows > 0.1 * rows.max(axis=1, keepdims=True)).any(axis=0))
    f, ex = g0.freqs(), []
    for k in high:                        # windows of neighbours, joined across gaps
        if ex and f[k] - ex[-1][1] < 0.0025:
            ex[-1][1] = f[k] + 0.001
        else:
            ex.append([f[k] - 0.001, f[k] + 0.001])
    assert 0 < len(ex) <= 64
    g = synth.Grid(g0.f_min, g0.df, g0.n_freq, exclude=tuple(map(tuple, ex)), **kw)
    best, info = search(b, g, sigma_t=0.3)
    assert info["w_bytes_direct"] == 0
    assert np.all(best["best_idx"] >= 0)
    same_search(best, by_the_pair_sum(monkeypatch, b, g, sigma_t=0.3))


@pytest.mark.parametrize("n", [700, 2000])
@pytest.mark.parametrize("seed", range(12))
def test_ties_far_below_an_excluded_peak(monkeypatch, n, seed):
    """Only the aliases +-f (mod 1) of one frequency are left to choose from, one
    whose value is near zero: on integer times they tie exactly, so the pair sum's
    last bits decide, and the spectrum's values carry the rounding of a peak
    hundreds of times as high."""
    b = strong_batch(1, n, 1500.0, 300 + seed, True)
    g0 = synth.Grid(0.2, 2e-4, 13001)                 # 0.2 .. 2.8
    got, info = search(b, g0, rows=True, sigma_t=0.3)
    assert info["w_bytes_direct"] == 0
    v, cells = got["rows"][0], 1000 + np.arange(g0.n_freq)     # frequencies in steps of 2e-4
    k = 250 + int(np.argmin(np.abs(v[250:1250])))              # 0.25 .. 0.45
    assert abs(v[k]) < 0.01 * v.max()
    left = np.flatnonzero((cells % 5000 == cells[k]) | (-cells % 5000 == cells[k]))
    f = g0.freqs()
    edges = np.r_[0.0, np.repeat(f[left], 2) + np.tile([-1e-4, 1e-4], len(left)), 3.0].reshape(-1, 2)
    g = synth.Grid(g0.f_min, g0.df, g0.n_freq, exclude=tuple(map(tuple, edges)))
    best, info = search(b, g, sigma_t=0.3)
    assert info["w_bytes_direct"] == 0 and int(best["best_idx"][0]) in left and len(left) >= 5
    same_search(best, by_the_pair_sum(monkeypatch, b, g, sigma_t=0.3))


def harmonics_of(sigma_t, tail=2e-8):
    """Harmonics kept: a_n = 2 e^-k I_n(k), k = 1 / sigma_t^2, by the backward recurrence,
    up to the first n whose remaining sum is at most `tail` of the kernel's peak."""
    k = 1.0 / (sigma_t * sigma_t)
    a = np.zeros(160)
    a[140] = 1e-200
    for n in range(140, 0, -1):
        a[n - 1] = a[n + 1] + 2.0 * n / k * a[n]
    a[1:] *= 2.0
    rest = np.cumsum((a / a.sum())[::-1])[::-1]
    return int(np.argmax(rest[1:] <= tail))


def transform_log2(n_out):
    """log2 of the complex transform for n_out entries: 1.1 times as many cells at least, two a point."""
    lq = 8
    while (2 << lq) < 1.1 * n_out:
        lq += 1
    return lq


# transform length, sigma_t, f_min, df, steps of the spectrum per df, K, curves, N.
# Up to 2^13 points one block transforms a curve; 2^22 is the longest.
LENGTHS = [(8, 1.5, 0.0, 1e-3, 1, 78, 64, 2000), (9, 1.5, 0.0, 1e-3, 1, 155, 64, 1200), (10, 1.5, 0.0, 1e-3, 1, 311, 64, 700),
           (11, 1.5, 0.0, 1e-3, 1, 621, 64, 500), (12, 1.5, 0.0, 1e-3, 1, 1241, 48, 400), (13, 1.5, 0.0, 1e-3, 1, 2482, 24, 400),
           (14, 1.5, 0.0, 1e-3, 1, 2500, 24, 400), (21, 0.1, 0.0, 1e-4, 1, 49981, 2, 400), (22, 0.1, 5e-5, 1e-4, 2, 49981, 2, 400)]


@pytest.mark.parametrize("case", LENGTHS, ids=["2^%d" % c[0] for c in LENGTHS])
def test_every_transform_length(monkeypatch, case):
    """Against the oracle: within 1e-5 of the curve's peak or, where the pair sum at every frequency
    does not meet that (noise curves on a few frequencies: 1.8e-5 at sigma_t 1.5, N 2,000), within the
    pair sum's own error."""
    logq, st, f_min, df, q, K, n_curves, n = case
    top = int(round(f_min / df * q)) + q * (K - 1)
    assert transform_log2(harmonics_of(st) * top + 1) == logq
    b = synth.ragged_batch(n_curves, seed=93, n_lo=n - 30, n_hi=n, span=900.0)
    g = synth.Grid(f_min, df, K)
    got, info = search(b, g, rows=True, sigma_t=st)
    assert info["w_bytes_direct"] == 0
    rows = got["rows"]
    np.testing.assert_array_equal(got["best_idx"], rows.argmax(axis=1))
    np.testing.assert_array_equal(got["best_stat"], rows.max(axis=1))
    some = list(range(min(n_curves, 6)))
    ks = np.unique(np.r_[0, 1, K - 1, np.random.default_rng(4).choice(K, 60, replace=False), got["best_idx"][some]])
    ref = oracle.batch_nckp(b.subset(some), np.full(len(some), float(np.float32(st))), g.freqs()[ks])
    peak = np.maximum(np.abs(ref).max(axis=1), np.abs(rows[some]).max(axis=1))
    err = np.abs(rows[some][:, ks] - ref).max(axis=1) / peak
    pair = by_the_pair_sum(monkeypatch, b, g, rows=True, sigma_t=st)
    perr = np.abs(pair["rows"][some][:, ks] - ref).max(axis=1) / peak
    print("max error %.2e of the peak, of the pair sum %.2e" % (err.max(), perr.max()))
    assert np.all(err <= np.maximum(TOL, perr)), (err, perr)
    same_search(got, pair)


def mixed_batch(n_curves, n_lo, n_hi, seed):
    """A batch with a constant curve (every value ties at zero) and two whose sigma_t needs more
    harmonics than the spectrum keeps."""
    b = synth.ragged_batch(n_curves, seed=seed, n_lo=n_lo, n_hi=n_hi, span=1500.0)
    b.mags[b.offsets[4]:b.offsets[5]] = 17.25
    st = np.full(n_curves, 0.3, np.float32)
    st[[1, 7]] = 0.05
    return b, st


@pytest.mark.parametrize("coarse_df,top_k", [(1e-3, 10), (3e-3, 1)])
def test_coarse_fine_curves_that_the_pair_sum_evaluates_whole(monkeypatch, coarse_df, top_k):
    b, st = mixed_batch(64, 200, 300, 94)
    g = synth.Grid(0.0041, 1e-4, 14501, hierarchical=True, coarse_df=coarse_df, top_k=top_k, fine_df=1.3e-5,
                   fine_halfwidth=2e-3)
    got, info = search(b, g, sigma_t_per_curve=st)
    assert info["w_bytes_direct"] == 0
    same_search(got, by_the_pair_sum(monkeypatch, b, g, sigma_t_per_curve=st))


def test_coarse_rows_longer_than_shared_memory(monkeypatch):
    """Coarse rows of 30,001 points (above 24,576 they are read from global memory)."""
    b, st = mixed_batch(24, 150, 200, 95)
    g = synth.Grid(0.01, 1e-4, 30001, hierarchical=True, coarse_df=1e-4, top_k=10, fine_df=1e-5, fine_halfwidth=1e-4)
    got, info = search(b, g, sigma_t_per_curve=st)
    assert info["w_bytes_direct"] == 0
    same_search(got, by_the_pair_sum(monkeypatch, b, g, sigma_t_per_curve=st))


def test_trial_lists_that_the_pair_sum_evaluates_whole(monkeypatch):
    """Bands search: the constant curve's 450 trials all tie, two curves have no spectrum; their
    trial values are the pair sum's own, the others' within the direct form's bar."""
    b, st = mixed_batch(64, 500, 600, 96)
    g = synth.Grid(0.00125, 1e-4, 20000, bands=True, n_bands=3, trials_per_band=150)
    got, info = search(b, g, sigma_t_per_curve=st)
    assert info["w_bytes_direct"] == 0
    want = by_the_pair_sum(monkeypatch, b, g, sigma_t_per_curve=st)
    same_search(got, want)
    np.testing.assert_array_equal(got["trial_idx"], want["trial_idx"])
    for c in range(b.n_curves):
        if c in (1, 4, 7):
            np.testing.assert_array_equal(got["trial_stat"][c], want["trial_stat"][c])
        else:
            np.testing.assert_allclose(got["trial_stat"][c], want["trial_stat"][c], rtol=0,
                                       atol=TOL * np.nanmax(np.abs(want["trial_stat"][c])))


SEARCHES = [dict(), dict(hierarchical=True, coarse_df=1e-3, top_k=5, fine_df=2e-5, fine_halfwidth=1e-3),
            dict(bands=True, n_bands=3, trials_per_band=100)]


def short_and_long(seed=98):
    """Curves of 2 to 100 samples (one of a single time) beside 60 of 600."""
    rng = np.random.default_rng(seed)
    sizes = np.array([2, 2, 3, 4, 5, 7, 9, 10, 16, 31, 32, 33, 63, 64, 65, 100] + [600] * 60)
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    t = rng.uniform(0.0, 1500.0, off[-1])
    t[off[1]:off[2]] = 40.0
    y = 17.0 + 0.3 * np.sin(2 * np.pi * t / 2.3) + rng.normal(0, 0.1, t.shape[0])
    z = np.zeros(len(sizes))
    return synth.Batch(t, y.astype(np.float32), np.full(t.shape[0], 0.1, np.float32), off, z, z.astype(bool), z.astype(np.int8))


@pytest.mark.parametrize("kw", SEARCHES)
def test_short_curves_beside_long_ones(monkeypatch, kw):
    b = short_and_long()
    g = synth.Grid(0.01, 1e-4, 20000, **kw)
    got, info = search(b, g, rows=not kw, sigma_t=0.3)
    assert info["w_bytes_direct"] == 0
    same_search(got, by_the_pair_sum(monkeypatch, b, g, sigma_t=0.3))
    if not kw:
        some = list(range(17))
        ks = np.arange(0, g.n_freq, 97)
        ref = oracle.batch_nckp(b.subset(some), np.full(len(some), float(np.float32(0.3))), g.freqs()[ks])
        err = np.abs(got["rows"][some][:, ks] - ref).max(axis=1)
        peak = np.abs(got["rows"][some]).max(axis=1)
        peak[1] = peak[0]                  # a single time: zero at every frequency
        print("max error %.2e of the peak" % np.max(err / peak))
        assert np.all(err <= TOL * peak), err / peak


@pytest.mark.parametrize("kw", SEARCHES)
def test_waves_of_a_small_tile_budget(monkeypatch, kw):
    """Several waves of curves (each with its chunks and its curves left to the pair sum): the results
    of one wave."""
    b, st = mixed_batch(64, 500, 600, 99)
    g = synth.Grid(0.01, 1e-4, 20000, **kw)
    got, info = search(b, g, rows=True, sigma_t_per_curve=st)
    monkeypatch.setenv("CP_W_BUDGET_KB", str(10 * 190 * 4))
    waves, info2 = search(b, g, rows=True, sigma_t_per_curve=st)
    assert info["w_bytes_direct"] == info2["w_bytes_direct"] == 0
    assert info2["launches_per_search"] > info["launches_per_search"]
    for key in got:
        np.testing.assert_array_equal(waves[key], got[key], err_msg=key)


@pytest.mark.parametrize("n", [40, 300, 448])
def test_cos_form_pair_sum_is_the_same_on_either_block_size(monkeypatch, n):
    """The pair sum's cos form (sigma_t 0.3 and above) on 16 warps and, with four units for every SM,
    on blocks of 4: the same bits (the lanes are added in the same order)."""
    b = synth.ragged_batch(1, seed=11, n_lo=n, n_hi=n, span=900.0)
    ks = (2000, 6400, 16 * 4 * 160)         # units of 16 frequencies: fewer than 2 per SM, than 4 per SM, more
    rows = [by_the_pair_sum(monkeypatch, b, synth.Grid(0.01, 1e-4, k), rows=True, sigma_t=0.4)["rows"][0] for k in ks]
    for k, row in zip(ks, rows):
        np.testing.assert_array_equal(row, rows[-1][:k])


@pytest.mark.parametrize("seed", range(4))
@pytest.mark.parametrize("kw,K", [(dict(), 195), (dict(), 2500), (dict(hierarchical=True, coarse_df=1e-3, top_k=3, fine_df=1e-4,
                                                                      fine_halfwidth=2e-3), 2500)])
def test_curves_that_cover_little_of_a_cycle(monkeypatch, kw, K, seed):
    """Half a day of observations on frequencies of 0 to 0.25 1/day: every value lies far below the scale
    of a noise curve, and the rounding of both ways decides the best; it is the pair sum's."""
    b = synth.ragged_batch(180, seed=120 + seed, n_lo=200, n_hi=480, span=0.5)
    st = np.random.default_rng(seed).choice([0.25, 0.3, 0.5, 0.9], b.n_curves).astype(np.float32)
    g = synth.Grid(0.0, 1e-4, K, **kw)
    got, info = search(b, g, sigma_t_per_curve=st)
    assert info["w_bytes_direct"] == 0
    same_search(got, by_the_pair_sum(monkeypatch, b, g, sigma_t_per_curve=st))
