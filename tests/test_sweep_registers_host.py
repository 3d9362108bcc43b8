"""The sweep kernel's variants in the compiler's resource report of the build:
launches without reservoir blocks of their own form have a kernel of one form,
and the variants that the default blocks run do not spill in it.  The group
kernels' static and dynamic shared memory fit a block together."""
import os
import re

import pytest

from paper_2605_25872_gb300.build import BUILD, CSRC, build

RULES = {"metropolis": 0, "heatbath": 1, "micsa": 2}


@pytest.fixture(scope="module")
def report():
    build()
    path = os.path.join(BUILD, "ptxas.txt")
    if not os.path.exists(path):
        pytest.skip("the library was built without its resource report")
    with open(path) as f:
        return f.read()


@pytest.fixture(scope="module")
def spills(report):
    """Bytes of spill stores by (L, rule, lattices per thread, both forms)."""
    found = re.findall(r"Function properties for \S*sweep_kernelILi(\d+)ELi(\d+)ELi(\d+)ELb([01])E\S*\s+"
                       r"\d+ bytes stack frame, (\d+) bytes spill", report)
    return {(int(L), int(r), int(k), bool(int(two))): int(n) for L, r, k, two, n in found}


def test_launches_of_one_form_have_a_kernel_of_their_own(spills):
    for L, rule, kt in ((12, "micsa", 16), (16, "heatbath", 32), (16, "metropolis", 16)):
        assert (L, RULES[rule], kt, False) in spills and (L, RULES[rule], kt, True) in spills
    assert (12, RULES["metropolis"], 16, True) not in spills     # never two forms


@pytest.mark.parametrize("rule,variants", [("metropolis", [(10, 16), (14, 16), (16, 16)]),
                                           ("heatbath", [(14, 16), (16, 16)])])
def test_default_variants_do_not_spill(spills, rule, variants):
    for L, kt in variants:
        assert spills[L, RULES[rule], kt, False] == 0, (L, kt)


def test_group_kernels_fit_their_dynamic_limit(report):
    static = [int(n) for n in re.findall(
        r"Compiling entry function '\S*group_(?:sweep|cluster)_kernel\S*' for \S+\n(?:.*\n)*?.*Used .* (\d+) bytes smem", report)]
    assert len(static) == 5
    with open(os.path.join(CSRC, "capi.cu")) as f:
        limit = int(re.search(r"GROUP_DYNAMIC_SMEM = (\d+) \* 1024", f.read()).group(1)) * 1024
    assert max(static) + limit <= 227 * 1024
