"""Sweeps in both forms of the block (couplings in registers, couplings in shared
memory) for every rule, run under the release and the range-checked build.

Run as a script (python tests/debug_sweep_scenarios.py OUT.npz) it saves each
scenario's results, its poll status and which forms ran under range checks
(status word 1; 0 in the release build)."""
import os
import sys

import numpy as np

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

import workloads as W  # noqa: E402

SHARED, REGISTERS = 1, 2
# (L, rule, samples, one lattice lane per block, sweeps, forms that run)
SCENARIOS = [(L, rule, 2, lane, (2, 3), SHARED if lane else REGISTERS)
             for L in (6, 10, 16) for rule in ("metropolis", "heatbath", "micsa") for lane in (False, True)]
# large launches whose reservoir blocks alone keep the couplings in registers
SCENARIOS += [(14, rule, 160, False, (1, 17), SHARED | REGISTERS) for rule in ("metropolis", "heatbath", "micsa")]
SCENARIOS += [(18, "metropolis", 2, False, (1, 2), SHARED)]


def run_all():
    import torch
    from paper_2605_25872_gb300 import Batch, BatchConfig, _lib, buffer_info
    out = {}
    for i, (L, rule, S, lane, sweeps, _) in enumerate(SCENARIOS):
        cfg = BatchConfig(L=L, n_samples=S, n_temps=6, n_replicas=3, n_res=5, rule=rule, cluster="off",
                          spin_layout="bits" if L == 16 else "bytes")
        tuning = {"sweep_threads": L * L * ((L // 2 + 3) // 4), "pt_lattices_per_block": 16,
                  "res_lattices_per_block": 15} if lane else None
        b = Batch(cfg, couplings=W.gaussian_couplings(L, S, 700 + i), seeds=W.sample_seeds(W.SEED_BASE + 700 + i, S),
                  tuning=tuning)
        b.sweep(*sweeps)
        b.synchronize()
        off, n = buffer_info(cfg, _lib.BUF_STATUS)
        out[f"cover{i}"] = b.ws[off:off + n].cpu().numpy().view(np.uint32)[1]
        out[f"spins{i}"] = b.export_spins().cpu().numpy()
        out[f"E{i}"] = b.energies.cpu().numpy()
        out[f"flips{i}"] = b.flips.cpu().numpy()
        out[f"poll{i}"] = np.array([b.poll(60000), b.check_canaries()])
        torch.cuda.synchronize()
        b.close()
    return out


if __name__ == "__main__":
    np.savez(sys.argv[1], **run_all())
