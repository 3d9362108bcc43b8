"""Sweeps with the couplings in registers (at most four lattices per thread) equal
sweeps with them in shared memory (all lattices of a block in one lane), for
every rule, padded and full rows, on and off the coupling grid.  Both shapes
are checked, so that no case compares a form with itself."""
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


def lattices_per_thread(b, lane):
    t = b.get_tuning()
    return -(-max(t["pt_lattices_per_block"], t["res_lattices_per_block"]) // (t["sweep_threads"] // lane))


@pytest.mark.parametrize("on_grid", [True, False])
@pytest.mark.parametrize("rule", ["metropolis", "heatbath", "micsa"])
@pytest.mark.parametrize("L", [6, 8, 10, 12, 14, 16])
def test_registers_equal_shared_memory(L, rule, on_grid):
    cfg = BatchConfig(L=L, n_samples=3, n_temps=6, n_replicas=3, n_res=5, rule=rule, cluster="off", sweeps_per_emcs=3,
                      res_sweeps_per_emcs=5, spin_layout="bits" if L == 8 else "bytes")
    J = W.gaussian_couplings(L, 3, 140 + L, on_grid=on_grid)
    lane = L * L * ((L // 2 + 3) // 4)
    out = []
    for tuning in (None, {"sweep_threads": lane, "pt_lattices_per_block": 15, "res_lattices_per_block": 15}):
        b = Batch(cfg, couplings=J, seeds=W.sample_seeds(W.SEED_BASE + 140 + L, 3), tuning=tuning)
        assert (lattices_per_thread(b, lane) > 4) == (tuning is not None)
        b.sweep(cfg.sweeps_per_emcs, cfg.res_sweeps_per_emcs)
        b.synchronize()
        out.append((b.export_spins().cpu().numpy(), b.flips.cpu().numpy(), b.energies.cpu().numpy()))
    np.testing.assert_array_equal(out[0][0], out[1][0])
    np.testing.assert_array_equal(out[0][1], out[1][1])
    if on_grid:
        np.testing.assert_array_equal(out[0][2], out[1][2])
    else:   # the FP64 sums run in another order: at most 3 V roundings of 2^-53 on either side
        bound = 2 * 3 * L ** 3 * 2.0 ** -53 * np.abs(J.astype(np.float64)).sum((1, 2))
        assert (np.abs(out[0][2] - out[1][2]) <= bound[:, None]).all()
