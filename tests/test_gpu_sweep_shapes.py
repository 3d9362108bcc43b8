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
from paper_2605_25872_gb300 import Batch, BatchConfig, Group  # noqa: E402
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


@pytest.mark.parametrize("rule", ["metropolis", "heatbath", "micsa"])
@pytest.mark.parametrize("L", [6, 8, 10, 12, 14, 16])
def test_reservoir_blocks_in_registers_equal_large_blocks(L, rule):
    # 160 samples: the reservoir's blocks (15 lattices, no multiple of four)
    # run other lattices per thread than the PT clones'; one lattice lane with
    # all of them per thread runs both alike
    S = 160
    cfg = BatchConfig(L=L, n_samples=S, n_temps=4, n_replicas=3, n_res=5, rule=rule, cluster="off",
                      spin_layout="bits" if L == 14 else "bytes")
    J = W.gaussian_couplings(L, S, 60 + L)
    seeds = W.sample_seeds(W.SEED_BASE + L, S)
    lane = L * L * ((L // 2 + 3) // 4)
    out = []
    for tuning in (None, {"res_lattices_per_block": 15, "sweep_threads": lane}):
        b = Batch(cfg, couplings=J, seeds=seeds, tuning=tuning)
        b.sweep(2, 15)      # below the length from which the reservoir has its own blocks
        b.sweep(1, 16)
        b.prethermalize(17)
        b.synchronize()
        out.append((b.export_spins().cpu().numpy(), b.energies.cpu().numpy(), b.flips.cpu().numpy()))
    for x, y in zip(*out):
        np.testing.assert_array_equal(x, y)


@pytest.mark.parametrize("rule", ["metropolis", "micsa"])
def test_group_reservoir_blocks_equal_batches(rule):
    sizes = (6, 8, 10, 12, 14, 16)
    cfgs = [BatchConfig(L=L, n_samples=2, n_temps=5, n_res=3, sweeps_per_emcs=2, res_sweeps_per_emcs=17,
                        rule=rule) for L in sizes]
    pairs = [[Batch(c, couplings=W.gaussian_couplings(c.L, 2, 80 + c.L), seeds=W.sample_seeds(W.SEED_BASE, 2),
                    stream=torch.cuda.Stream()) for c in cfgs] for _ in range(2)]
    g = Group(pairs[0], stream=torch.cuda.Stream())
    g.emcs(2)
    g.synchronize()
    for a, b in zip(*pairs):
        b.emcs(2)
        b.synchronize()
        for name in ("energies", "flips", "obs", "perm"):
            np.testing.assert_array_equal(getattr(a, name).cpu().numpy(), getattr(b, name).cpu().numpy())
        np.testing.assert_array_equal(a.export_spins().cpu().numpy(), b.export_spins().cpu().numpy())
