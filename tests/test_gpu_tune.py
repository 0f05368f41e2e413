"""The autotuner on the GPU: its direct-form rates are the pair kernel's."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1412_1840_gb300 import tune as T  # noqa: E402

EX2_PER_S = 10.06e12     # the MUFU's rate (peaks_gb300.json); the pair sum takes one ex2 per pair and frequency


@pytest.fixture(scope="module", autouse=True)
def _need_gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def test_direct_rates_are_the_pair_sums():
    table = T.tune(target_pair_freq=4e9, classes=(8, 32), log=lambda *a: None)
    assert len(table["buckets"]) == len(T.BUCKETS)
    for b in table["buckets"]:
        for rate in list(b["direct"].values()) + [b["direct_sin_form"]]:
            assert 0.0 < rate < EX2_PER_S, b
