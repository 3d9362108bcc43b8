"""The sweep of a batch with few samples (small blocks, couplings in registers)
equals the sweep of the same samples in large blocks bit for bit: spins,
energies and flip counts, for each rule, on full and padded colour rows, with
lattice counts that do not fill the blocks."""
import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu

P = pytest.importorskip("paper_2605_25872_gb300")
from paper_2605_25872_gb300 import Batch, BatchConfig  # noqa: E402
from paper_2605_25872_gb300.build import build  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build()


@pytest.mark.parametrize("rule", ["metropolis", "heatbath", "micsa"])
@pytest.mark.parametrize("L", [2, 4, 6, 10, 12, 14, 16, 18])
def test_small_blocks_equal_large_blocks(L, rule):
    cfg = BatchConfig(L=L, n_samples=3, n_temps=5, n_replicas=3, n_res=3, rule=rule, cluster="off",
                      spin_layout="bits" if L == 10 else "bytes")
    J = W.gaussian_couplings(L, 3, 40 + L, on_grid=L != 6)
    seeds = W.sample_seeds(W.SEED_BASE + L, 3)
    small = Batch(cfg, couplings=J, seeds=seeds)
    large = Batch(cfg, couplings=J, seeds=seeds, tuning={"pt_lattices_per_block": 15, "res_lattices_per_block": 9})
    shapes = [b.get_tuning() for b in (small, large)]
    assert shapes[0]["pt_lattices_per_block"] <= shapes[1]["pt_lattices_per_block"]
    for b in (small, large):
        b.prethermalize(3, first=1, count=2)
        b.sweep(3, 5)
        b.sweep(1, 0)
        b.synchronize()
    np.testing.assert_array_equal(small.export_spins().cpu().numpy(), large.export_spins().cpu().numpy())
    np.testing.assert_array_equal(small.flips.cpu().numpy(), large.flips.cpu().numpy())
    if L != 6:
        np.testing.assert_array_equal(small.energies.cpu().numpy(), large.energies.cpu().numpy())
    else:   # off the grid the FP64 sums run in another order
        np.testing.assert_allclose(small.energies.cpu().numpy(), large.energies.cpu().numpy(), rtol=1e-12, atol=1e-12)
