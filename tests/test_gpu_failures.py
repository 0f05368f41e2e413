"""Failure handling of the C ABI on a GPU, made on the host: an allocation
that the test makes fail (CP_FAIL_ALLOC) must give CP_ENOMEM, release what
the plan had allocated, and leave the next plan unaffected."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1412_1840_gb300 as cp  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _need_gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def test_allocation_failure_reports_enomem_and_leaves_nothing(monkeypatch):
    b = synth.ragged_batch(256, seed=51, n_lo=900, n_hi=1000)    # ~0.5 GB of magnitude-kernel tiles
    g = synth.Grid(0.01, 1e-3, 64)
    grid = cp.grid_from(g)
    td = torch.from_numpy(b.times).cuda()
    md = torch.from_numpy(b.mags).cuda()
    ed = torch.from_numpy(b.errs).cuda()
    with cp.Plan(td, md, ed, b.offsets, grid, sigma_t=0.3) as p:
        want = p.best_period()
    torch.cuda.synchronize()
    free0 = torch.cuda.mem_get_info()[0]
    for k in (1, 2):                       # the device block, then the pinned host block
        monkeypatch.setenv("CP_FAIL_ALLOC", str(k))
        with pytest.raises(cp.CpError) as e:
            cp.Plan(td, md, ed, b.offsets, grid, sigma_t=0.3)
        assert e.value.status == cp.CP_ENOMEM
        torch.cuda.synchronize()
        assert abs(torch.cuda.mem_get_info()[0] - free0) < (64 << 20)
    monkeypatch.delenv("CP_FAIL_ALLOC")
    with cp.Plan(td, md, ed, b.offsets, grid, sigma_t=0.3) as p:
        got = p.best_period()
    for k in ("best_idx", "best_freq", "best_stat", "is_periodic"):
        np.testing.assert_array_equal(got[k], want[k])


@pytest.mark.parametrize("kw", [dict(), dict(hierarchical=True, coarse_df=2e-3, top_k=5, fine_df=1e-4, fine_halfwidth=4e-3),
                                dict(bands=True, n_bands=3, trials_per_band=150)])
def test_no_room_for_the_pair_spectrum_falls_back_to_the_pair_sum(monkeypatch, kw):
    """A plan whose block with the pair spectrum's workspace cannot be allocated
    is made without it, with the same search results; one that has no room for
    the pair sum either reports CP_ENOMEM."""
    b = synth.ragged_batch(64, seed=52, n_lo=300, n_hi=400, span=1500.0)
    g = synth.Grid(0.01, 1e-3, 2000, **kw)
    dev = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (b.times, b.mags, b.errs)]
    out = torch.zeros((b.n_curves, g.n_freq), dtype=torch.float32, device="cuda")

    def run():
        with cp.Plan(*dev, b.offsets, cp.grid_from(g), sigma_t=0.3) as p:
            best = p.best_period()
            p.periodogram(out)
            p.sync()
            return best, out.cpu().numpy(), p.info()

    best, rows, info = run()
    assert info["w_bytes_direct"] == 0
    nb = (np.diff(b.offsets) + 31) // 32
    tiles = int(np.sum(nb * (nb + 1) // 2)) * 4096
    monkeypatch.setenv("CP_FAIL_ALLOC_ABOVE_KB", str((tiles >> 10) + 8192))   # tiles, and 8 MB for the rest
    best2, rows2, info2 = run()
    assert info2["w_bytes_direct"] == tiles
    for k in best:
        np.testing.assert_array_equal(best2[k], best[k], err_msg=k)
    assert np.all(np.abs(rows2 - rows).max(axis=1) <= 1e-5 * np.abs(rows).max(axis=1))
    monkeypatch.setenv("CP_FAIL_ALLOC_ABOVE_KB", str(tiles >> 10))
    with pytest.raises(cp.CpError) as e:
        run()
    assert e.value.status == cp.CP_ENOMEM
