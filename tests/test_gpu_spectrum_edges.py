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


def by_the_pair_sum(monkeypatch, b, g, extra_kb, **kw):
    """The same search on a plan that has room for the magnitude-kernel tiles only."""
    nb = (np.diff(b.offsets) + 31) // 32
    tiles = int(np.sum(nb * (nb + 1) // 2)) * 4096
    with monkeypatch.context() as m:
        m.setenv("CP_FAIL_ALLOC_ABOVE_KB", str((tiles >> 10) + extra_kb))
        got, info = search(b, g, **kw)
    assert info["w_bytes_direct"] == tiles
    return got


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
    want = by_the_pair_sum(monkeypatch, b, g, 2560, sigma_t=0.3)
    for key in ("best_idx", "best_freq", "best_stat", "is_periodic"):
        np.testing.assert_array_equal(best[key], want[key], err_msg=key)


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
    want = by_the_pair_sum(monkeypatch, b, g, 1536, sigma_t=0.3)
    for key in ("best_idx", "best_freq", "best_stat", "is_periodic"):
        np.testing.assert_array_equal(best[key], want[key], err_msg=key)
