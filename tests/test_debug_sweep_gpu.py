"""The range-checked build checks both forms of the sweep block: every scenario of
debug_sweep_scenarios.py runs its forms under checks, none fails, and the
results are those of the release build."""
import os
import subprocess
import sys

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

P = pytest.importorskip("paper_2605_25872_gb300")
from paper_2605_25872_gb300 import _lib  # noqa: E402
from paper_2605_25872_gb300.build import build  # noqa: E402

HERE = os.path.dirname(os.path.abspath(__file__))


def test_both_sweep_forms_run_under_range_checks(tmp_path):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build()
    out = tmp_path / "debug.npz"
    env = dict(os.environ, PTHR_LIBRARY=build(debug=True))
    r = subprocess.run([sys.executable, os.path.join(HERE, "debug_sweep_scenarios.py"), str(out)], env=env,
                       capture_output=True, text=True, timeout=900)
    assert r.returncode == 0, r.stderr[-3000:]
    sys.path.insert(0, HERE)
    import debug_sweep_scenarios as S
    rel = S.run_all()
    got = np.load(out)
    for i, sc in enumerate(S.SCENARIOS):
        assert list(got[f"poll{i}"]) == [_lib.PTHR_OK, -1], sc
        assert int(got[f"cover{i}"]) == sc[-1], sc
        assert int(rel[f"cover{i}"]) == 0
        for k in ("spins", "E", "flips"):
            np.testing.assert_array_equal(got[f"{k}{i}"], rel[f"{k}{i}"], err_msg=str(sc))
