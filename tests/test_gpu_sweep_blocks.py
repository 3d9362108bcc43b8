"""Lattices per sweep block of launches that leave SMs idle: short launches keep
the large blocks, long ones run small blocks, the kind with more lattice
sweeps decides; and the blocks in between give the same results."""
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


def pt_lattices(**kw):
    kw = dict(dict(n_res=0, er_on=False, sweeps_per_emcs=1), **kw)
    return Batch(BatchConfig(**kw)).get_tuning()["pt_lattices_per_block"]


@pytest.mark.parametrize("L,S,NT,large", [(8, 128, 16, 64), (10, 64, 24, 32), (12, 25, 24, 16), (14, 12, 48, 16),
                                          (16, 18, 32, 16)])
def test_one_sweep_on_most_sms_keeps_the_large_blocks(L, S, NT, large):
    assert pt_lattices(L=L, n_samples=S, n_temps=NT) == large


def test_long_launches_of_few_blocks_run_small_blocks():
    for L, S, NT in ((4, 1, 12), (8, 2, 16), (16, 1, 32)):
        assert pt_lattices(L=L, n_samples=S, n_temps=NT, sweeps_per_emcs=10) == 4
    for rule in ("metropolis", "heatbath", "micsa"):    # the reservoir's sweeps
        assert pt_lattices(L=14, n_samples=20, n_temps=48, rule=rule, sweeps_per_emcs=10, n_res=4, er_on=True) == 4


def test_the_kind_with_more_lattice_sweeps_decides():
    assert pt_lattices(L=16, n_samples=60, n_temps=32, sweeps_per_emcs=40, n_res=4, er_on=True,
                       res_sweeps_per_emcs=1) == 16


@pytest.mark.parametrize("rule", ["metropolis", "heatbath", "micsa"])
@pytest.mark.parametrize("L,S,NT,n", [(6, 40, 16, 3), (8, 32, 16, 3), (8, 60, 16, 10), (10, 20, 24, 3), (12, 9, 24, 2),
                                      (16, 6, 32, 3)])
def test_blocks_in_between_equal_one_lane(L, S, NT, n, rule):
    cfg = BatchConfig(L=L, n_samples=S, n_temps=NT, n_res=2, rule=rule, cluster="off")
    J = W.gaussian_couplings(L, S, 30 + L)
    seeds = W.sample_seeds(W.SEED_BASE + 30 + L, S)
    lane = L * L * ((L // 2 + 3) // 4)
    out = []
    for tuning in (None, {"sweep_threads": lane, "pt_lattices_per_block": 7, "res_lattices_per_block": 8}):
        b = Batch(cfg, couplings=J, seeds=seeds, tuning=tuning)
        b.sweep(n, 0)
        b.sweep(1, 5)
        b.synchronize()
        out.append((b.export_spins().cpu().numpy(), b.energies.cpu().numpy(), b.flips.cpu().numpy()))
    for x, y in zip(*out):
        np.testing.assert_array_equal(x, y)


@pytest.mark.parametrize("L,rule,lattices", [(10, "metropolis", 16), (10, "heatbath", 4), (14, "heatbath", 16),
                                             (16, "heatbath", 16)])
def test_default_blocks_run_variants_of_fewer_lattices(L, rule, lattices):
    # lattices per thread of a large launch of PT clones (test_sweep_registers_host.py:
    # the variants of 32 at these sizes spill; L = 10 with the heat bath: couplings in registers)
    t = Batch(BatchConfig(L=L, n_samples=160, n_temps=24, n_res=0, er_on=False, rule=rule)).get_tuning()
    lanes = t["sweep_threads"] // (L * L * ((L // 2 + 3) // 4))
    assert t["pt_lattices_per_block"] <= lattices * lanes


@pytest.mark.parametrize("L,share", [(6, 64), (8, 64), (10, 48)])
def test_a_callers_pt_share_is_kept_beside_reservoir_blocks(L, share):
    cfg = BatchConfig(L=L, n_samples=160, n_temps=16, n_res=1)
    b = Batch(cfg, tuning={"pt_lattices_per_block": share})
    assert b.get_tuning()["pt_lattices_per_block"] == share
