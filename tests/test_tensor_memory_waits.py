"""Who may hold tensor memory while it waits.  A CTA that keeps columns until the grids before its own have finished must not be what a
CTA of those grids waits for in its allocation, without end: so every kernel that allocates lets the next grid start only behind its
allocation, and gives the columns back before it waits for its cluster or, at its end, for another grid."""
import os
import re

import pytest

from tests.test_tc_plan import ROOT

CSRC = os.path.join(ROOT, "paper_2604_18396_b200", "csrc")
KERNELS = [("gemm_tc.cuh", "tc_gemm_kernel"), ("gemm_tc_w4.cuh", "tc_gemm_w4_kernel"), ("gemm_tc_wide.cuh", "tc_gemm_wide_kernel"),
           ("attn_prefill_tc.cuh", "attn_prefill_tc_kernel")]


def body(name, what):
    s = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
    i = re.search(r"\b%s\(" % what, s).start()
    return s[i:s.index("\n}\n", i)]


def test_every_kernel_that_allocates_is_here():
    found = {f for f in os.listdir(CSRC) if "tcgen05.alloc" in open(os.path.join(CSRC, f)).read()}
    assert found == {f for f, _ in KERNELS}


@pytest.mark.parametrize("name,kernel", KERNELS)
def test_the_next_grid_starts_behind_the_allocation(name, kernel):
    b = body(name, kernel)
    alloc = [m.start() for m in re.finditer(r"tcgen05\.alloc", b)]
    assert len(alloc) == 1
    for m in re.finditer(r"pdl_launch\(\);", b):
        before = b[:m.start()]
        # behind the allocation, in the warp that made it - or where the CTA leaves without one
        leaves = re.match(r"pdl_launch\(\);\s*(if \(a\.overlap\) )?pdl_wait\(\);\s*return;", b[m.start():])
        same_warp = alloc[0] < m.start() and "\n    }" not in before[alloc[0]:]
        later = alloc[0] < m.start() and "pdl_wait();" in before[alloc[0]:]  # (late_release: past the wait, too)
        assert leaves or same_warp or later, before[-200:]
    assert "pdl_launch();" in b[alloc[0]:]


def test_columns_go_back_before_the_cluster_is_waited_for():
    b = body("gemm_tc.cuh", "tc_finish")
    assert 0 < b.index("tcgen05.dealloc") < b.index("barrier.cluster")
    for name, kernel in KERNELS[:2]:
        k = body(name, kernel)
        assert "barrier.cluster" not in k[:k.index("tc_finish(")]
