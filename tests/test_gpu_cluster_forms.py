"""Cluster moves on overlaps whose clusters take every route of the cluster
kernel: all sites equal, single sites only, thousands of two-site clusters
(more than are flooded one by one, so the union-find takes over), one long
winding path, domains that wrap around the lattice.  Labels, spins, energies
and statistics equal the oracle's (couplings on the grid: every sum is exact)."""
import numpy as np
import pytest
import torch

import oracle as O
import workloads as W

pytestmark = pytest.mark.gpu

P = pytest.importorskip("paper_2605_25872_gb300")
from paper_2605_25872_gb300 import BatchConfig  # noqa: E402
from test_gpu_parity import make, gpu_spins  # noqa: E402


def overlap(form, L):
    z, y, x = np.meshgrid(*[np.arange(L)] * 3, indexing="ij")
    if form == "equal":
        q = np.ones((L, L, L))
    elif form == "single sites":
        q = 1 - 2 * ((x + y + z) & 1)
    elif form == "pairs":
        q = 1 - 2 * ((x // 2 + y + z) & 1)
    elif form == "winding":        # even rows full, odd rows one site at alternating ends; planes joined at a corner
        q = np.where(y % 2 == 0, 1, np.where(x == np.where(y % 4 == 1, 0, L - 1), 1, -1))
        q = np.where(z % 2 == 0, q, np.where((x == 1) & (y == 0), 1, -1))
    else:                          # wrapped: a slab across each periodic boundary
        q = np.where((x < 1) | (x >= L - 1) | (y < 1) | (z >= L - 1), -1, 1)
    return q.astype(np.int8).reshape(-1)


@pytest.mark.parametrize("mode", ["acu", "single"])
@pytest.mark.parametrize("L", [2, 6, 14, 16, 18, 24])
def test_cluster_forms(L, mode):
    forms = ["equal", "single sites", "pairs", "winding", "wrapped"]
    cfg = BatchConfig(L=L, n_samples=1, n_temps=len(forms), t_min=0.2, t_max=0.8, n_replicas=2, n_res=0, er_on=False,
                      cluster=mode, spin_layout="bits" if L == 6 else "bytes")
    gpu, mir = make(cfg, seed=90 + L)
    spins = W.random_spins((1, cfg.n_lat, cfg.V), 3000 + L)
    for k, form in enumerate(forms):
        spins[0, cfg.n_slot + k] = spins[0, k] * overlap(form, L)
    gpu.import_spins(torch.from_numpy(spins))
    smp = mir.samples[0]
    smp.spins[:] = spins[0]
    for lat in range(cfg.n_lat):
        smp.E_lat[lat] = O.energy(L, smp.J, smp.spins[lat])
    lab = gpu.cluster_labels().cpu().numpy()
    sizes = []
    for k in range(len(forms)):
        ref, _ = O.cc_labels(L, spins[0, k], spins[0, cfg.n_slot + k])
        np.testing.assert_array_equal(lab[0, 0, k], ref, err_msg=forms[k])
        sizes.append(np.sort(np.bincount(ref)[np.unique(ref)])[::-1])
    gpu.houdayer()
    mir.houdayer()
    np.testing.assert_array_equal(gpu_spins(gpu), mir.spins())
    np.testing.assert_array_equal(gpu.energies.cpu().numpy(), mir.energies())
    cs = gpu.cluster_stats.cpu().numpy()[0, 0]
    for k, n in enumerate(sizes):
        assert list(cs[k, :3]) == [len(n), n[0], n[1] if len(n) > 1 else 0], forms[k]
    assert gpu.poll(10000) == 0
