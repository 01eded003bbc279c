"""The launch rule of small steps' projections (csrc/stream_plan.h), compiled for the host."""
import ctypes
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SHIM = r"""
#include "stream_plan.h"
extern "C" int small(int sms, int rows, int tasks, int K, int R, int *o) {
    river::StreamGeom g{0, 0};
    const bool is = river::stream_small_share(sms, rows, tasks, K, R, g);
    o[0] = g.threads; o[1] = g.grid; o[2] = R == 2 ? river::kStreamPieces<2> : river::kStreamPieces<4>;
    return is ? 1 : 0;
}
"""
SMS = 148


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    d = tmp_path_factory.mktemp("plan")
    (d / "shim.cpp").write_text(SHIM)
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", os.path.join(ROOT, "paper_2604_18396_b200", "csrc"),
                           str(d / "shim.cpp"), "-o", str(d / "shim.so")])
    return ctypes.CDLL(str(d / "shim.so"))


@pytest.mark.parametrize("R,K_from,K_to", [(4, 32, 4096), (2, 4096, 8192 + 32)])
@pytest.mark.parametrize("tasks", [1, 64, 148, 149, 700, 148 * 9, 148 * 16, 148 * 16 + 1])
def test_the_warps_hold_a_row(plan, tasks, R, K_from, K_to):
    """A CTA of a one-row step holds the row in registers whatever its length, every warp has a task and every CTA one."""
    o = (ctypes.c_int * 3)()
    share = -(-tasks // SMS)
    for K in range(K_from, K_to, 32):
        is_small = plan.small(SMS, 1, tasks, K, R, o)
        assert bool(is_small) == (share <= 16)
        if is_small:
            threads, grid, pieces = o
            assert threads * pieces * 4 >= K, K
            assert grid == min(tasks, SMS) and threads % 32 == 0 and max(128, 32 * share) <= threads <= 512
            assert threads <= 32 * max(4, share) or (threads - 32) * pieces * 4 < K  # and no warp more than that


def test_only_steps_of_few_rows(plan):
    """More rows than one pass takes keep the geometry whose warps all stage."""
    o = (ctypes.c_int * 3)()
    assert [plan.small(SMS, n, 148, 512, 4, o) for n in (1, 2, 3, 4, 5, 8, 64, 256, 1024)] == [1, 1, 1, 1, 0, 0, 0, 0, 0]
