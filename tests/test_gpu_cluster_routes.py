"""The two forms of the cluster launch -- warps that hold whole pairs, and one
block per pair for launches of few pairs -- give the same labels, spins,
energies and statistics, on overlaps of every kind, both moves and both spin
layouts; and the default picks the block per pair where pairs are few."""
import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu

P = pytest.importorskip("paper_2605_25872_gb300")
from paper_2605_25872_gb300 import Batch, BatchConfig  # noqa: E402
from paper_2605_25872_gb300.build import build  # noqa: E402
from test_gpu_cluster_forms import overlap  # noqa: E402

FORMS = ("equal", "single sites", "pairs", "winding", "wrapped", "random", "random")


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build()


@pytest.mark.parametrize("mode", ["acu", "single"])
@pytest.mark.parametrize("L", [2, 4, 6, 8, 12, 14, 16, 18, 22, 24])
def test_forms_of_the_launch_agree(L, mode):
    bits, off = L in (6, 16, 18), L in (14, 24)
    cfg = BatchConfig(L=L, n_samples=2, n_temps=len(FORMS), t_min=0.2, t_max=0.8, n_replicas=2, n_res=0, er_on=False,
                      cluster=mode, spin_layout="bits" if bits else "bytes")
    spins = W.random_spins((2, cfg.n_lat, cfg.V), 500 + L)
    for k, form in enumerate(FORMS):
        if form != "random":
            spins[:, cfg.n_slot + k] = spins[:, k] * overlap(form, L)
    out = []
    for threads in (0, 128, 32, 160, 512):
        b = Batch(cfg, couplings=W.gaussian_couplings(L, 2, 50 + L, on_grid=not off),
                  seeds=W.sample_seeds(W.SEED_BASE + 50 + L, 2), tuning={"cluster_threads": threads})
        b.import_spins(torch.from_numpy(spins))
        labels = b.cluster_labels().cpu().numpy()
        b.houdayer()
        out.append((labels, b.export_spins().cpu().numpy(), b.cluster_stats.cpu().numpy(), b.energies.cpu().numpy()))
        assert b.poll(10000) == 0
    for o in out[1:]:
        for x, y in zip(o[:3], out[0][:3]):
            np.testing.assert_array_equal(x, y)
        if off:     # the FP64 sums run in another order: at most 3 V + 36 roundings of 2^-53
            J = np.abs(W.gaussian_couplings(L, 2, 50 + L, on_grid=False).astype(np.float64)).sum((1, 2))
            assert (np.abs(o[3] - out[0][3]) <= (2 * 3 * L ** 3 * 2.0 ** -53) * J[:, None]).all()
        else:
            np.testing.assert_array_equal(o[3], out[0][3])


@pytest.mark.parametrize("L", [4, 8, 16, 24])
def test_few_pairs_have_a_block_each(L):
    few = Batch(BatchConfig(L=L, n_samples=1, n_temps=12, n_res=0, er_on=False))
    assert few.get_tuning()["cluster_threads"] > 128
    many = Batch(BatchConfig(L=L, n_samples=160, n_temps=16, n_res=0, er_on=False))
    assert many.get_tuning()["cluster_threads"] <= 128
