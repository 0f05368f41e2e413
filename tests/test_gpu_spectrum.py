"""The uniform grid through the pair spectrum (csrc/cp_spec.cu): against the
FP64 oracle at the direct form's bar (1e-5 of the curve's peak), at the edges of
its ranges: one- and two-pass transforms, time differences beyond half of the
transform's period (df T > 1/2), grids that start at 0, between or off the
multiples of df (interpolated), equal and unordered times, sigma_t at both ends,
curves that the pair sum evaluates whole.  The best frequency, of the uniform
grid and of the coarse-then-fine search, is the pair sum's own: it equals
cp_best_period_noalloc's (pair sum at every frequency) bit for bit."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1412_1840_gb300 as cp  # noqa: E402

TOL = 1e-5
PLAIN = 6      # most launches of a search whose curves the pair sum evaluates at every frequency


@pytest.fixture(scope="module", autouse=True)
def _need_gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def batch(n_curves, n_lo, n_hi, span, seed=11, shuffle=False, integer=False):
    b = synth.ragged_batch(n_curves, seed=seed, n_lo=n_lo, n_hi=n_hi, span=span)
    if integer:
        b.times[:] = np.floor(b.times)                  # equal times
    if shuffle:
        rng = np.random.default_rng(3)
        for c in range(n_curves):
            s = slice(int(b.offsets[c]), int(b.offsets[c + 1]))
            p = rng.permutation(s.stop - s.start)
            b.times[s], b.mags[s], b.errs[s] = b.times[s][p], b.mags[s][p], b.errs[s][p]
    return b


def run(b, g, **kw):
    dev = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (b.times, b.mags, b.errs)]
    with cp.Plan(*dev, b.offsets, cp.grid_from(g), **kw) as p:
        out = torch.zeros((b.n_curves, g.n_freq), dtype=torch.float32, device="cuda")
        p.periodogram(out)
        p.sync()
        rows = out.cpu().numpy()
        best = p.best_period()
        p.periodogram(out)
        p.sync()
        np.testing.assert_array_equal(rows, out.cpu().numpy())      # deterministic
        return rows, best, p.curve_stats()["sigma_t"].astype(np.float64), p.info()


CASES = [
    # curves, N, span, f_min, df, K, sigma_t
    (192, 60, 90, 40.0, 0.0, 4e-3, 2400, 0.5),        # one pass, grid from 0
    (48, 100, 300, 1500.0, 0.01, 1e-3, 2001, 0.3),   # differences folded: df T = 1.5
    (12, 150, 400, 1500.0, 0.01, 1e-3, 4000, 0.1),    # smallest sigma_t, two passes
    (12, 150, 400, 900.0, 5e-4, 1e-3, 4001, 0.62),    # f_min = df / 2
    (6, 300, 420, 5000.0, 0.0025, 2e-4, 9001, 1.5),  # two harmonics or so, f_min = 12.5 df
    (3, 1500, 2100, 2500.0, 0.002, 1e-4, 700, 0.25),
    # off the multiples of df: interpolated
    (64, 60, 130, 700.0, 0.00143, 1e-3, 3500, 0.5),
    (6, 200, 400, 1733.0, 1.0 / 1733.0, 1e-4, 6000, 0.1),
    (6, 300, 400, 5000.0, 0.0123457, 1e-3, 5000, 0.3),   # longer than the spectra are made for
    # more curves than one launch takes
    (200, 60, 90, 300.0, 0.01, 2e-3, 1500, 0.4),
    # transforms of 2^20 points
    (2, 300, 400, 1500.0, 0.0, 1e-4, 40000, 0.1),
]


@pytest.mark.parametrize("case", CASES)
@pytest.mark.parametrize("form", ["ordered", "shuffled", "integer"])
def test_spectrum_matches_oracle(case, form):
    n_curves, n_lo, n_hi, span, f_min, df, K, st = case
    b = batch(n_curves, n_lo, n_hi, span, shuffle=form == "shuffled", integer=form == "integer")
    g = synth.Grid(f_min, df, K)
    rows, best, sig, info = run(b, g, sigma_t=st)
    assert info["launches_per_search"] > PLAIN
    ks = np.unique(np.r_[0, 1, K - 1, np.random.default_rng(2).choice(K, 160, replace=False), best["best_idx"]])
    ref = oracle.batch_nckp(b, sig, g.freqs()[ks])
    peak = np.maximum(np.abs(ref).max(axis=1), np.abs(rows).max(axis=1))
    err = np.abs(rows[:, ks] - ref).max(axis=1) / peak
    print("max error %.2e of the peak" % err.max())
    assert np.all(err <= TOL), err
    np.testing.assert_array_equal(best["best_idx"], rows.argmax(axis=1))
    np.testing.assert_array_equal(best["best_stat"], rows.max(axis=1))


def via_noalloc(b, g, sigma_t):
    dev = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (b.times, b.mags, b.errs)]
    n = b.n_curves
    out = (torch.zeros(n, dtype=torch.int64, device="cuda"), torch.zeros(n, dtype=torch.float64, device="cuda"),
           torch.zeros(n, dtype=torch.float32, device="cuda"), torch.zeros(n, dtype=torch.uint8, device="cuda"))
    cp.cp_best_period_noalloc(*dev, b.offsets, cp.grid_from(g), sigma_t, *out)
    return dict(zip(("best_idx", "best_freq", "best_stat", "is_periodic"), (o.cpu().numpy() for o in out)))


def same(got, want):
    for k in want:
        np.testing.assert_array_equal(got[k].astype(want[k].dtype), want[k], err_msg=k)


@pytest.mark.parametrize("f_min", [0.01, 0.00977])
@pytest.mark.parametrize("integer", [False, True])
def test_best_frequency_is_the_pair_sums(integer, f_min):
    b = batch(40, 60, 400, 1500.0, seed=12, integer=integer)
    g = synth.Grid(f_min, 1e-3, 2000)
    _, best, _, info = run(b, g, sigma_t=0.3)
    assert info["launches_per_search"] > PLAIN
    same(best, via_noalloc(b, g, 0.3))


# coarse_df T from 0.5 to 4, one peak to 20 (the most that goes through the spectrum), windows that
# overlap and that leave the band
@pytest.mark.parametrize("span,coarse_df,top_k,half,sigma_t", [(500.0, 1e-3, 10, 2e-3, 0.45), (2500.0, 1e-3, 1, 2e-3, 0.3),
                                                               (2500.0, 1.6e-3, 20, 1e-3, 0.25), (1733.0, 7e-4, 5, 5e-3, 0.12)])
@pytest.mark.parametrize("integer", [False, True])
def test_coarse_fine_is_the_pair_sums(span, coarse_df, top_k, half, sigma_t, integer):
    b = batch(64, 150, 300, span, seed=14, integer=integer)
    g = synth.Grid(0.0041, 1e-4, 14501, hierarchical=True, coarse_df=coarse_df, top_k=top_k, fine_df=1.3e-5,
                   fine_halfwidth=half)
    dev = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (b.times, b.mags, b.errs)]
    with cp.Plan(*dev, b.offsets, cp.grid_from(g), sigma_t=sigma_t) as p:
        best = p.best_period()
        assert p.info()["launches_per_search"] > 8
        same(p.best_period(), best)
    same(best, via_noalloc(b, g, sigma_t))


def test_curves_outside_the_spectrums_range():
    """A constant curve (every frequency ties at 0) and curves whose sigma_t
    needs too many harmonics are evaluated by the pair sum, the others of the
    batch by the spectrum; exclusion windows and waves of a small W budget."""
    b = batch(12, 200, 400, 1500.0, seed=13)
    b.mags[b.offsets[4]:b.offsets[5]] = 17.25
    st = np.full(12, 0.3, np.float32)
    st[[1, 7]] = 0.05
    g = synth.Grid(0.01, 1e-3, 2400)
    rows, best, sig, info = run(b, g, sigma_t_per_curve=st)
    assert info["launches_per_search"] > PLAIN
    assert np.all(rows[4] == 0.0) and best["best_idx"][4] == 0 and best["best_stat"][4] == 0.0
    ks = np.arange(0, 2400, 15)
    ref = oracle.batch_nckp(b, sig, g.freqs()[ks])
    keep = [c for c in range(12) if c != 4]
    err = np.abs(rows[keep][:, ks] - ref[keep]).max(axis=1) / np.abs(rows[keep]).max(axis=1)
    assert np.all(err <= TOL), err
    f = g.freqs()
    g.exclude = tuple((x - 2e-3, x + 2e-3) for x in np.unique(best["best_freq"]))
    _, left, _, _ = run(b, g, sigma_t_per_curve=st)
    adm = ~np.any([(f >= lo) & (f <= hi) for lo, hi in g.exclude], axis=0)
    want = [np.flatnonzero(adm)[np.argmax(rows[c][adm])] for c in keep]
    np.testing.assert_array_equal(left["best_idx"][keep], want)


@pytest.mark.parametrize("n", [40, 300, 448])
def test_pair_sum_is_the_same_on_either_block_size(n):
    """Short curves run on blocks of 4 warps once every SM has four of its units
    (below that: 16 warps, on whole or halved units): the sums' order, hence
    every bit, is the same."""
    b = batch(1, n, n, 900.0)
    ks = (2000, 6400, 16 * 4 * 160)         # units of 16 frequencies: fewer than 2 per SM, than 4 per SM, more
    rows = [run(b, synth.Grid(0.01, 1e-4, k), sigma_t=0.08)[0][0] for k in ks]
    for k, row in zip(ks, rows):
        np.testing.assert_array_equal(row, rows[-1][:k])
