"""A bounded labelling loop that runs out (cluster_iter_cap, no fault) stops its
own pair only: the pair's neighbours in the warp are labelled and moved."""
import numpy as np
import pytest
import torch

import oracle as O
import workloads as W

pytestmark = pytest.mark.gpu

P = pytest.importorskip("paper_2605_25872_gb300")
from paper_2605_25872_gb300 import Batch, BatchConfig, _lib  # noqa: E402
from paper_2605_25872_gb300.build import build  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build()


L = 16
# a flood grows by one site in y per pass at most, so the cluster of all sites
# (reach L / 2) needs more than 2 cap = 4 passes, a site and its six neighbours
# (reach 2 from their first site) at most 3
FORMS = ("star", "all", "all", "star", "star", "all")


def batch():
    cfg = BatchConfig(L=L, n_samples=1, n_temps=len(FORMS), t_min=0.2, t_max=0.8, n_replicas=2, n_res=0, er_on=False)
    z, y, x = np.meshgrid(*[np.arange(L)] * 3, indexing="ij")
    star = 1 - 2 * ((x + y + z) & 1)
    star[5, 6, 7] *= -1
    spins = W.random_spins((1, cfg.n_lat, cfg.V), 12)
    for k, form in enumerate(FORMS):
        spins[0, cfg.n_slot + k] = spins[0, k] * (star.reshape(-1) if form == "star" else 1)
    b = Batch(cfg, couplings=W.gaussian_couplings(L, 1, 11), seeds=W.sample_seeds(W.SEED_BASE + 11, 1))
    b.import_spins(torch.from_numpy(spins))
    b.set_tuning(cluster_iter_cap=2)
    return cfg, b, spins


def test_only_the_pairs_that_ran_out_stay_as_they_were():
    cfg, b, spins = batch()
    e = b.energies.cpu().numpy().copy()
    b.houdayer()
    assert b.poll(10000) == _lib.PTHR_E_NOCONVERGE
    out = b.export_spins().cpu().numpy()[0]
    cs = b.cluster_stats.cpu().numpy()[0, 0]
    for k, form in enumerate(FORMS):
        if form == "star":
            assert list(cs[k, :3]) == [cfg.V - 6, 7, 1]
            assert (out[[k, cfg.n_slot + k]] != spins[0, [k, cfg.n_slot + k]]).any()
        else:
            assert not cs[k].any()
            np.testing.assert_array_equal(out[[k, cfg.n_slot + k]], spins[0, [k, cfg.n_slot + k]])
            np.testing.assert_array_equal(b.energies.cpu().numpy()[0, [k, cfg.n_slot + k]], e[0, [k, cfg.n_slot + k]])


def test_labels_of_a_pair_that_ran_out_are_absent():
    cfg, b, spins = batch()
    lab = b.cluster_labels().cpu().numpy()[0, 0]
    assert b.poll(10000) == _lib.PTHR_E_NOCONVERGE
    for k, form in enumerate(FORMS):
        ref = O.cc_labels(L, spins[0, k], spins[0, cfg.n_slot + k])[0] if form == "star" else -1
        np.testing.assert_array_equal(lab[k], ref if form == "star" else np.full(cfg.V, -1))
