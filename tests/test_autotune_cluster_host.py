"""Host-side checks of the autotuner's cluster-block candidates (no GPU needed):
every block size of the form whose warps hold whole pairs (up to 128 threads,
32 among them, which small launches run by default), and blocks per pair only
where a thread has sites to work on; and stored shapes hold for the kernels
that they were timed on."""
import shutil

import pytest

from paper_2605_25872_gb300 import BatchConfig, autotune
from paper_2605_25872_gb300.autotune import candidates
from paper_2605_25872_gb300.build import CSRC


@pytest.mark.parametrize("L", [2, 4, 8, 16, 24])
def test_cluster_candidates_cover_both_forms(L):
    cfg = BatchConfig(L=L, n_samples=4, n_temps=8, n_res=0, er_on=False)
    threads = [s["cluster_threads"] for s in candidates(cfg) if "cluster_threads" in s]
    assert len(threads) == len(set(threads))
    assert [t for t in threads if t <= 128] == [32, 64, 128]
    assert all(t % 32 == 0 and t <= min(512, L ** 3 // 2) for t in threads if t > 128)
    assert any(t > 128 for t in threads) == (L >= 8)


def test_stored_shapes_belong_to_the_kernels_they_were_timed_on(tmp_path):
    copy = tmp_path / "csrc"
    shutil.copytree(CSRC, copy)
    assert autotune.kernels_version(str(copy)) == autotune.kernels_version()
    with open(copy / "capi.cu", "a") as f:
        f.write("// another shape rule\n")
    autotune.kernels_version.cache_clear()
    assert autotune.kernels_version(str(copy)) != autotune.kernels_version()
    assert autotune.kernels_version() in autotune._key(BatchConfig(L=8, n_samples=2, n_temps=4), "GPU")
