"""The cluster step inside a group launch, in both of its forms (a block per pair
where pairs are few, warps that hold whole pairs), equals the batches' own in
the other form; overlaps of thousands of two-site clusters, which the warps
hand to the union-find, among them."""
import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu

P = pytest.importorskip("paper_2605_25872_gb300")
from paper_2605_25872_gb300 import Batch, BatchConfig, Group  # noqa: E402
from paper_2605_25872_gb300.build import build  # noqa: E402
from test_gpu_cluster_forms import overlap  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build()


@pytest.mark.parametrize("sizes,samples,threads", [((4, 6, 8, 10, 12, 14, 16), 2, 128), ((4, 12), 48, 512)])
def test_group_forms_equal_the_batches(sizes, samples, threads):
    made = []
    for tuning in (None, {"cluster_threads": threads}):
        bs = []
        for L in sizes:
            cfg = BatchConfig(L=L, n_samples=samples, n_temps=24, n_res=0, er_on=False, sweeps_per_emcs=0,
                              spin_layout="bits" if L == 8 else "bytes")
            b = Batch(cfg, couplings=W.gaussian_couplings(L, samples, 90 + L),
                      seeds=W.sample_seeds(W.SEED_BASE + 90, samples), stream=torch.cuda.Stream(), tuning=tuning)
            spins = W.random_spins((samples, cfg.n_replicas, cfg.n_slot, cfg.V), 900 + L)
            spins[:, 1, :8] = spins[:, 0, :8] * overlap("pairs", L)
            b.import_spins(torch.from_numpy(spins.reshape(samples, cfg.n_lat, cfg.V)))
            bs.append(b)
        made.append(bs)
    assert all((b.get_tuning()["cluster_threads"] > 128) == (threads <= 128) for b in made[0])
    g = Group(made[0], stream=torch.cuda.Stream())
    assert g.launches_per_emcs == 4
    g.emcs(2)
    g.synchronize()
    for a, b in zip(*made):
        b.emcs(2)
        b.synchronize()
        for name in ("energies", "obs", "perm", "cluster_stats"):
            np.testing.assert_array_equal(getattr(a, name).cpu().numpy(), getattr(b, name).cpu().numpy())
        np.testing.assert_array_equal(a.export_spins().cpu().numpy(), b.export_spins().cpu().numpy())
        assert a.poll(10000) == 0 and b.poll(10000) == 0
