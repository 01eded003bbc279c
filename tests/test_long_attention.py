"""Which attention kernel a long pass takes (csrc/tc_plan.h), compiled for the host: both sides of a mean look-back of 64 and of 128."""
import ctypes
import os
import subprocess

import pytest

from tests.test_tc_plan import ROOT, SMS, ceil_div

SHIM = r"""
#include "tc_plan.h"
extern "C" int on_tcgen05(int sms, int warp_ctas, int n, long long seen) { return river::tc_long_attention(sms, warp_ctas, n, seen); }
"""


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    d = tmp_path_factory.mktemp("attn")
    (d / "shim.cpp").write_text(SHIM)
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", os.path.join(ROOT, "paper_2604_18396_b200", "csrc"),
                           str(d / "shim.cpp"), "-o", str(d / "shim.so")])
    lib = ctypes.CDLL(str(d / "shim.so"))
    lib.on_tcgen05.argtypes = [ctypes.c_int, ctypes.c_int, ctypes.c_int, ctypes.c_longlong]
    return lambda lens, hkv: bool(lib.on_tcgen05(SMS, ceil_div(sum(lens), 16) * hkv, sum(lens), sum(n * (n + 1) // 2 for n in lens)))


# (two KV heads, 1184 rows and fewer: the warp-level kernel's CTAs are one per SM at most; eight KV heads: more)
@pytest.mark.parametrize("lens,hkv,taken", [([126, 126], 2, False), ([127, 127], 2, True), ([146, 97], 2, False), ([147, 97], 2, True),
                                            ([200, 60], 2, True), ([191, 191], 2, True), ([16] * 40, 2, False), ([1024], 2, True),
                                            ([160] * 5, 8, False), ([254, 254], 8, False), ([255, 255], 8, True), ([1024], 8, True),
                                            ([296], 8, True), ([127, 127], 8, True), ([127] * 3, 8, False)])
def test_by_mean_look_back(rule, lens, hkv, taken):
    assert rule(lens, hkv) is taken
