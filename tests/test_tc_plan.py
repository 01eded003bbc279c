"""The rules that cut the tensor-core projections' work (csrc/tc_plan.h), compiled for the host: how many inputs one sum inside
the tensor cores takes, at most."""
import ctypes
import itertools
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SHIM = r"""
#include "tc_plan.h"
extern "C" {
int pick(int sms, int tiles, int kb, int slots, int min_kb) { return river::tc_pick_splits(sms, tiles, kb, slots, min_kb); }
void w4(int sms, int np, int tiles, int K, int decode, int *o) {
    const river::W4Plan p = river::w4_plan(sms, np, tiles, K, decode != 0);
    o[0] = p.occ; o[1] = p.n_stages; o[2] = p.splits; o[3] = p.wide; o[4] = p.sets; o[5] = p.cols;
}
int tc_splits(int sms, int np, int tiles, int K) { return river::tc_plan(sms, np, tiles, K, true, false).splits; }
void tc(int sms, int np, int tiles, int K, int most, int *o) {
    const river::TcPlan p = river::tc_plan(sms, np, tiles, K, true, false, most);
    o[0] = p.occ; o[1] = p.splits; o[2] = p.halves; o[3] = river::tc_stages_at(np, p.occ);
}
void w4_most(int sms, int np, int tiles, int K, int most, int *o) {
    const river::W4Plan p = river::w4_plan(sms, np, tiles, K, false, most);
    o[0] = p.occ; o[1] = p.splits; o[2] = p.sets; o[3] = p.cols; o[4] = p.wide; o[5] = p.n_stages;
}
int ends_fit(int sms, int rows, int ends, int d, int q, int F, int f16) { return river::tc_ends_fit(sms, rows, ends, d, q, F, f16 != 0); }
int long_pass_rows(int d, int L, int exit_blocks, int max_rows) { return river::tc_long_pass_rows(d, L, exit_blocks, max_rows); }
int wide_segment(int sms, int rows, int tiles, int K, int f16) { return river::tc_wide_segment(sms, rows, tiles, K, f16 != 0); }
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


def ceil_div(a, b):
    return -(-a // b)


# (128-feature tiles, K) of the repository's shapes - QKV, O, gate/up, down - and others of the same range
SHAPES = sorted({(4, 256), (2, 256), (16, 256), (2, 1024), (12, 512), (4, 1024), (24, 512), (4, 1536), (24, 2048), (16, 2048), (128, 2048),
                 (16, 8192), (48, 4096), (32, 4096), (224, 4096), (32, 14336)} | set(itertools.product((1, 3, 8, 20, 56, 100, 147), (2048, 2304, 5120, 16384))))


@pytest.mark.parametrize("np", range(16, 257, 16))
def test_exit_layer_sums_take_no_more_inputs_than_a_split_over_every_slot(plan, np):
    o = (ctypes.c_int * 6)()
    for tiles, K in SHAPES:
        raw = K // 256
        for decode in (0, 1):
            plan.w4(SMS, np, tiles, K, decode, o)
            occ, stages, splits, wide, sets, cols = o
            every_slot = plan.pick(SMS, tiles, raw, SMS * occ, 2 if raw <= 8 else 4)
            assert 1 <= splits <= 8 and splits <= raw and stages >= 2 and stages % 2 == 0 and occ * cols <= 512
            assert cols >= sets * (2 * np if wide else np) + 32 * stages and (sets == 1 or wide)
            # k-blocks that one accumulator takes, at most: a CTA's raw tiles hold four each, two halves of them with two accumulators
            assert ceil_div(4 * ceil_div(raw, splits), sets) <= 4 * ceil_div(raw, every_slot), (tiles, K, decode)
    # 64 rows of the 8B shape's down projection, of its QKV, and the 1B shape's gate/up
    for tiles, K, longest in ((32, 14336, 1792), (48, 4096, 1024), (128, 2048, 1024)):
        plan.w4(SMS, np, tiles, K, 1, o)
        assert np > 128 or 256 * ceil_div(ceil_div(K // 256, o[2]), o[4]) <= longest, (tiles, K)


@pytest.mark.parametrize("chunk", [128, 160, 200, 256])
def test_long_pass_sums_are_no_longer_than_short_passes(plan, chunk):
    o = (ctypes.c_int * 6)()
    np = ceil_div(chunk, 16) * 16
    for tiles, K in SHAPES:
        kb = K // 64
        for f16 in (0, 1):
            if f16:
                plan.w4(SMS, np, tiles, K, 0, o)
                longest = 4 * ceil_div(kb // 4, o[2])
            else:
                longest = ceil_div(kb, plan.tc_splits(SMS, np, tiles, K))
            assert 1 <= plan.wide_segment(SMS, chunk, tiles, K, f16) <= min(16, longest), (tiles, K, f16)


@pytest.mark.parametrize("chunk", [128, 200, 256])
@pytest.mark.parametrize("np", range(16, 97, 16))
def test_prompt_ends_sums_are_no_longer_than_the_long_pass_they_end(plan, np, chunk):
    """What a long pass computes at its prompt ends on the kernels of decode steps: no accumulator sums more k-blocks than the pair
    kernel's, within the limits of a launch."""
    o = (ctypes.c_int * 6)()
    for tiles, K in SHAPES:
        kb = K // 64
        most = plan.wide_segment(SMS, chunk, tiles, K, 0)
        plan.tc(SMS, np, tiles, K, most, o)
        occ, splits, halves, stages, _, _ = o
        if splits:
            assert ceil_div(ceil_div(kb, splits), 1 + halves) <= most, (tiles, K)
            assert splits <= 8 and splits <= kb and stages >= 2 and (not halves or (occ == 2 and np <= 64))
        else:
            assert ceil_div(kb, 8 * (2 if np <= 64 else 1)) > most, (tiles, K)
        most = plan.wide_segment(SMS, chunk, tiles, K, 1)
        plan.w4_most(SMS, np, tiles, K, most, o)
        occ, splits, sets, cols, wide, stages = o
        if splits:
            assert 4 * ceil_div(kb // 4, splits) // sets <= most, (tiles, K)
            assert splits <= 8 and splits <= kb // 4 and (sets == 1 or wide)
            assert occ * cols <= 512 and cols >= sets * (2 * np if wide else np) + 32 * stages
        else:
            assert ceil_div(kb // 4, 8) * 4 > most * (2 if np <= 32 else 1), (tiles, K)


def test_which_prompt_ends_take_the_kernels_of_decode_steps(plan):
    fit = lambda d, q, F, f16: [n for n in (1, 4, 5, 32, 33, 64, 65, 96, 97, 200) if plan.ends_fit(SMS, 256, n, d, q, F, f16)]  # noqa: E731
    assert fit(512, 1024, 1536, 0) == fit(512, 1024, 1536, 1) == fit(2048, 2048, 8192, 0) == fit(2048, 2048, 8192, 1) == [1, 4, 5, 32, 33, 64, 65, 96]
    assert fit(4096, 4096, 14336, 0) == [1, 4, 5, 32, 33, 64] and fit(4096, 4096, 14336, 1) == [1, 4, 5, 32]
    assert fit(8192, 8192, 28672, 0) == [1, 4] and fit(8192, 8192, 28672, 1) == []  # its down projection needs more splits than a cluster has


def test_rows_of_a_long_pass(plan):
    assert [plan.long_pass_rows(d, 2, x, 256) for d, x in ((256, 0), (512, 2), (1024, 0), (2048, 2), (3072, 0), (4096, 0), (4096, 1), (8192, 2))] == [
        129, 129, 145, 205, 145, 161, 257, 257]
    assert plan.long_pass_rows(4096, 32, 32, 128) == 129  # never more than one short pass can hold, nor than the batch kernels take
    assert plan.long_pass_rows(4096, 32, 32, 1024) == 257
