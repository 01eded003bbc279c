"""Row tiles of the batch projections (csrc/tc_plan.h), compiled for the host: when a step's rows are dealt out over several CTAs, that
their sums stay those of all rows together, and that whatever shares an SM finds its tensor memory there."""
import ctypes
import os
import subprocess

import pytest

from tests.test_tc_plan import ROOT, SHAPES, SMS, ceil_div

SHIM = r"""
#include "tc_plan.h"
extern "C" {
int row_tile(int sms, int np, int tiles, int K, int decode) { return river::tc_row_tile(sms, np, tiles, K, decode != 0); }
int tc_splits(int sms, int np, int tiles, int K, int decode) { return river::tc_plan(sms, np, tiles, K, true, decode != 0).splits; }
int pass_rows(int sms, int tiles, int K) { return river::tc_tiled_pass_rows(sms, tiles, K); }
int pass_splits(int sms, int pass_rows, int tiles, int K, int f16, int n) { return river::tc_pass_splits(sms, pass_rows, tiles, K, f16 != 0, n); }
int segment(int sms, int pass_rows, int tiles, int K, int f16) { return river::tc_wide_segment(sms, pass_rows, tiles, K, f16 != 0); }
int tc_columns(int np, int nt) { river::TcFootprint f[6]; return river::most_columns(f, river::step_footprints(np, nt, f)); }
long w4_smem(int sms, int np, int nt, int tiles, int K, int decode, int *o) {
    const river::W4Plan all = river::w4_plan(sms, np, tiles, K, decode != 0), p = river::w4_row_plan(all, np, nt);
    o[0] = p.occ; o[1] = p.n_stages; o[2] = p.splits; o[3] = p.sets; o[4] = p.cols; o[5] = p.wide; o[6] = all.splits; o[7] = all.sets;
    const long smem = (long)river::w4_smem_request(p, np, nt);
    river::TcFootprint f[7];
    const int n = river::step_footprints(np, nt, f);
    f[n] = {(size_t)smem, p.cols};
    o[8] = smem ? river::most_columns(f, n + 1) : 0;
    return smem;
}
}
"""


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    d = tmp_path_factory.mktemp("rows")
    (d / "shim.cpp").write_text(SHIM)
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", os.path.join(ROOT, "paper_2604_18396_b200", "csrc"),
                           str(d / "shim.cpp"), "-o", str(d / "shim.so")])
    lib = ctypes.CDLL(str(d / "shim.so"))
    lib.w4_smem.restype = ctypes.c_long
    return lib


@pytest.mark.parametrize("np", range(16, 257, 16))
def test_tiles_fit_beside_each_other_and_sum_the_same(plan, np):
    o = (ctypes.c_int * 9)()
    for nt in [t for t in (16, 32, 64) if t < np] + [np]:
        assert plan.tc_columns(np, nt) <= 512
        for tiles, K in SHAPES:
            for decode in (0, 1):
                if K % 256:
                    continue
                smem = plan.w4_smem(SMS, np, nt, tiles, K, decode, o)
                assert 0 < smem <= 227 * 1024 and o[8] <= 512 and o[0] * o[4] <= 512, (nt, tiles, K)
                assert (o[2], o[3]) == (o[6], o[7]) and o[4] >= o[3] * (2 * nt if o[5] else nt) + 32 * o[1] and o[1] >= 2 and o[1] % 2 == 0


def test_row_tiles_of_the_shapes(plan):
    widest = {"tiny": (16, 256), "mini8": (24, 512), "1b": (128, 2048), "8b": (224, 4096)}
    got = {s: [plan.row_tile(SMS, np, t, K, 0) for np in (16, 32, 64, 112, 128, 256)] for s, (t, K) in widest.items()}
    assert got["8b"] == got["1b"] == [16, 32, 64, 112, 128, 256]
    for s, (t, K) in widest.items():
        for np in range(16, 257, 16):
            for decode in (0, 1):
                nt = plan.row_tile(SMS, np, t, K, decode)
                assert nt == np or t * plan.tc_splits(SMS, np, t, K, decode) * ceil_div(np, nt) <= 2 * SMS
    assert got["mini8"][:5] == [16, 16, 16, 32, 32] and got["tiny"][:5] == [16, 16, 16, 16, 16], got


def test_short_passes_of_dealt_out_rows(plan):
    assert [plan.pass_rows(SMS, t, K) for t, K in ((16, 256), (24, 512), (128, 2048), (224, 4096))] == [192, 192, 0, 0]


@pytest.mark.parametrize("n", [225, 256, 600, 830, 1024])
def test_long_passes_on_the_batch_kernel_sum_no_longer(plan, n):
    taken = []
    for tiles, K in SHAPES:
        for f16 in (0, 1):
            if K % 256:
                continue
            s = plan.pass_splits(SMS, 256, tiles, K, f16, n)
            if s:
                taken.append((tiles, K))
                kb = K // 64
                per = [kb * (i + 1) // s - kb * i // s for i in range(s)]
                assert s <= 8 and min(per) >= 2 and max(ceil_div(p, 2) for p in per) <= plan.segment(SMS, 256, tiles, K, f16), (tiles, K)
                assert tiles * s * ceil_div(n, 64) <= 2 * SMS
    assert (4, 1536) in taken and (4, 1024) in taken and (2, 1024) in taken  # O and down of the mini and the tiny shape
    assert not any(t >= 16 for t, _ in taken)
