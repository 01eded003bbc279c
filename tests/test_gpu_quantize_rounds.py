"""The refinement rounds of river_quantize_w4 that leave operations out, against the quantiser oracle: groups whose
residuals reach the soft threshold, whose codes need clamping, far from zero, tiny, constant, and matrices of one group."""
import numpy as np
import pytest
import torch

from oracle import quant_oracle as qo
from tests.test_gpu_quantize import _near_bf16_boundary
from workloads import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("group", [32, 64, 128])
@pytest.mark.parametrize("out,groups,std,offset,outlier", [
    (1, 1, 0.02, 0.0, 1.0), (3, 5, 0.02, 0.0, 8.0), (129, 3, 1.0, 0.0, 1.0), (17, 4, 6.0, 0.0, 3.0), (16, 4, 1e-5, 0.0, 1.0),
    (16, 4, 0.3, 40.0, 1.0), (16, 4, 0.02, -1.0, 20.0)])
def test_rounds_match_oracle(group, out, groups, std, offset, outlier):
    from paper_2604_18396_b200 import binding
    w = synth.normal(23, group + out, (out, group * groups), std, "cuda") + offset
    w[:, ::29] *= outlier
    if out > 3:
        w[2, :group] = w[2, 0]
    w = w.bfloat16().contiguous()
    codes, scale, zero = binding.quantize_w4(w, group, 20)
    c_o, s_o, z_o, zf = qo.quantize_w4(w.float().cpu().numpy(), group, 20, return_float_zero=True)
    assert np.array_equal(scale.float().cpu().numpy(), s_o)
    # (as in test_gpu_quantize.py: where the soft threshold acts, the power's last bit may turn a rounding to bf16 over)
    near = _near_bf16_boundary(zf)
    zg = zero.float().cpu().numpy()
    assert np.array_equal(zg[~near], z_o[~near])
    same = np.repeat(~near, group // 2, axis=1)
    assert np.array_equal(codes.cpu().numpy()[same], c_o[same])
