"""Energies after a cluster move for couplings other than Gaussian ones on the
grid: wide-ranging float32 couplings (every clone's energy is recomputed) and
diluted ones (zeros are on the grid: the energies are updated in integers)."""
import math

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


def domain_pairs(cfg, seed):
    """Spins [S, n_lat, V]: mostly aligned clones whose overlap has domains of
    a few sites inside two large clusters."""
    rng = np.random.Generator(np.random.PCG64(seed))
    L, S = cfg.L, cfg.n_samples
    a = np.where(rng.random((S, cfg.n_slot, cfg.V)) < 0.03, -1, 1)
    z, y, x = np.meshgrid(*[np.arange(L)] * 3, indexing="ij")
    slab = np.where(z < L // 2, 1, -1).reshape(-1)
    b = a * slab * np.where(rng.random(a.shape) < 0.05, -1, 1)
    return np.concatenate([a, b], axis=1).astype(np.int8)


def energy(L, J, s):
    """H = -sum J s s', exactly rounded (J [3, V], s [V])."""
    s = s.reshape(L, L, L).astype(np.float64)
    t = [J[d].reshape(L, L, L).astype(np.float64) * (s * np.roll(s, -1, 2 - d)) for d in range(3)]
    return -math.fsum(np.concatenate([u.ravel() for u in t]))


@pytest.mark.parametrize("L", [12, 18])
def test_off_grid_energies_are_exact(L):
    # Couplings in [2^-13, 2): multiples of 2^-36.  A thread's sum over at most
    # 3 L terms stays below 2^7, so every TwoSum error is at most 2^-18 and
    # their sum at most 54 x 2^-18 < 2^-12: FP32 holds it exactly, and the FP64
    # sums (below 2^16, multiples of 2^-36) are exact in any order.
    cfg = BatchConfig(L=L, n_samples=3, n_temps=5, t_min=0.2, t_max=0.8, n_replicas=2, n_res=0, er_on=False)
    rng = np.random.Generator(np.random.PCG64(70 + L))
    J = np.exp2(rng.uniform(-13.0, 1.0, (3, 3, cfg.V)))
    J = np.maximum(J, rng.uniform(0.0, 1.9, J.shape) * (rng.random(J.shape) < 0.7))
    J = np.clip(J, 2.0 ** -13, 1.99).astype(np.float32)
    b = Batch(cfg, couplings=J, seeds=W.sample_seeds(W.SEED_BASE + 70 + L, 3))
    b.import_spins(torch.from_numpy(domain_pairs(cfg, 71 + L)))
    before = b.export_spins().cpu().numpy()
    b.houdayer()
    after = b.export_spins().cpu().numpy()
    E = b.energies.cpu().numpy()
    moved = (before != after).any(-1)
    assert moved.sum() >= 4
    for s, lat in np.argwhere(moved):
        assert E[s, lat] == energy(L, J[s], after[s, lat]), (s, lat)


@pytest.mark.parametrize("zero", [0.0, -0.0])
@pytest.mark.parametrize("L", [8, 14, 18])
def test_zero_couplings_are_on_the_grid(L, zero):
    # On the grid the move adds an exact difference to the resident energies:
    # a shift planted in both clones' energies is still there afterwards, where
    # a recomputation would drop it.
    cfg = BatchConfig(L=L, n_samples=2, n_temps=6, t_min=0.2, t_max=0.8, n_replicas=2, n_res=0, er_on=False)
    J = W.gaussian_couplings(L, 2, 80 + L)
    J[np.random.Generator(np.random.PCG64(L)).random(J.shape) < 0.5] = zero
    b = Batch(cfg, couplings=J, seeds=W.sample_seeds(W.SEED_BASE + 80 + L, 2))
    b.import_spins(torch.from_numpy(domain_pairs(cfg, 81 + L)))
    before = b.export_spins().cpu().numpy()
    b.energies.add_(1024.0)
    b.houdayer()
    after = b.export_spins().cpu().numpy()
    E = b.energies.cpu().numpy()
    assert (before != after).any(-1).sum() >= 4
    for s in range(2):
        for lat in range(cfg.n_lat):
            assert E[s, lat] == energy(L, J[s], after[s, lat]) + 1024.0, (s, lat)
