"""The sweep kernel's variants, from the compiler's resource report: launches
without reservoir blocks of their own form have a kernel of one form, and the
variants that the default blocks run do not spill in it."""
import os
import re
import shutil
import subprocess

import pytest

from paper_2605_25872_gb300.build import ARCH, CSRC, ROOT

NVCC = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"


def spills(tmp_path, L, rule, kt):
    """Bytes of spill stores of every kernel that launch_sweep_tpl<L, rule, kt> can launch."""
    src = tmp_path / "v.cu"
    src.write_text('#include "sweep_kernel.cuh"\nnamespace pthr {\ntemplate cudaError_t sweep_detail::launch_sweep_tpl'
                   f"<{L}, {rule}, {kt}>(const SweepArgs &, int, int, size_t, cudaStream_t);\n}}\n")
    r = subprocess.run([NVCC, "-O3", "-std=c++17", *ARCH, "-I", os.path.join(ROOT, "include"), "-I", CSRC, "-Xptxas", "-v",
                        "-c", str(src), "-o", str(tmp_path / "v.o")], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    found = re.findall(r"Function properties for (\S*sweep_kernel\S*)\s+\d+ bytes stack frame, (\d+) bytes spill", r.stderr)
    assert found, r.stderr[-2000:]
    return [int(n) for _, n in found]


@pytest.mark.skipif(not os.path.exists(NVCC), reason="needs nvcc")
def test_launches_of_one_form_have_a_kernel_of_their_own(tmp_path):
    assert len(spills(tmp_path, 12, "PTHR_MICSA", 16)) == 2
    assert len(spills(tmp_path, 16, "PTHR_HEATBATH", 32)) == 2
    assert len(spills(tmp_path, 12, "PTHR_METROPOLIS", 16)) == 1     # never two forms


@pytest.mark.skipif(not os.path.exists(NVCC), reason="needs nvcc")
@pytest.mark.parametrize("rule,variants", [("PTHR_METROPOLIS", [(10, 16), (14, 16), (16, 16)]),
                                           ("PTHR_HEATBATH", [(14, 16), (16, 16)])])
def test_default_variants_do_not_spill(tmp_path, rule, variants):
    for L, kt in variants:
        assert min(spills(tmp_path, L, rule, kt)) == 0, (L, kt)
