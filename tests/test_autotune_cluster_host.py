"""Host-side checks of the autotuner's cluster-block candidates (no GPU needed):
every block size of the form whose warps hold whole pairs (up to 128 threads,
32 among them, which small launches run by default), and blocks per pair only
where a thread has sites to work on."""
import pytest

from paper_2605_25872_gb300 import BatchConfig
from paper_2605_25872_gb300.autotune import candidates


@pytest.mark.parametrize("L", [2, 4, 8, 16, 24])
def test_cluster_candidates_cover_both_forms(L):
    cfg = BatchConfig(L=L, n_samples=4, n_temps=8, n_res=0, er_on=False)
    threads = [s["cluster_threads"] for s in candidates(cfg) if "cluster_threads" in s]
    assert len(threads) == len(set(threads))
    assert [t for t in threads if t <= 128] == [32, 64, 128]
    assert all(t % 32 == 0 and t <= min(512, L ** 3 // 2) for t in threads if t > 128)
    assert any(t > 128 for t in threads) == (L >= 8)
