"""Where the dequantising kernel learns early that it has rows (csrc/tc_plan.h), compiled for the host: from a count that this step or pass
wrote, never above its own, whatever earlier ones left behind - and positive in a pass whose host knows that there are rows, but for the
block right behind the first that only some of them left at."""
import ctypes
import itertools
import os
import subprocess

import pytest

from tests.test_tc_plan import ROOT

SHIM = r"""
#include "tc_plan.h"
extern "C" int hint(int all, int at, int before, int settled) { return river::exit_rows_hint(all != 0, at, before, settled != 0); }
"""


@pytest.fixture(scope="module")
def hint(tmp_path_factory):
    d = tmp_path_factory.mktemp("hint")
    (d / "shim.cpp").write_text(SHIM)
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", os.path.join(ROOT, "paper_2604_18396_b200", "csrc"),
                           str(d / "shim.cpp"), "-o", str(d / "shim.so")])
    return ctypes.CDLL(str(d / "shim.so")).hint


@pytest.mark.parametrize("L", [1, 2, 5])
def test_passes_whose_depths_are_known(hint, L):
    for depths in itertools.product(range(L + 1), repeat=3):
        n_riv = [None] * (L + 1)  # (None: what an earlier step left)
        at, before, gone, left_at = 0, 0, depths.count(0), 0
        n_riv[0] = gone
        for l in range(1, L + 1):  # noqa: E741
            everyone = gone == len(depths)
            e = hint(everyone, at, before, at < l - 1)
            seen = len(depths) if e < 0 else n_riv[e]
            assert seen is not None and seen <= gone and (e != l - 1 or l == 1), (depths, l)
            if gone and (everyone or left_at < l - 1):
                assert seen > 0, (depths, l)
            if l < L and depths.count(l):
                left_at = left_at if gone else l
                before, at, gone = at, l, gone + depths.count(l)
                n_riv[l] = gone


@pytest.mark.parametrize("L", [1, 2, 5])
def test_steps(hint, L):
    """Every entry is written: never above the count entering the block, and the entry is complete when the block before it starts."""
    for exits in itertools.product(range(L + 1), repeat=3):
        count = [sum(e <= l for e in exits) for l in range(L + 1)]
        at = before = 0
        for l in range(1, L + 1):  # noqa: E741
            e = hint(0, at, before, at < l - 1)
            assert e == max(0, l - 2) and count[e] <= count[l - 1]
            before, at = at, l
