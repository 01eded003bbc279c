"""river_quantize_w4 ends a group's refinement at a zero-point that a round gives back: against the quantiser oracle, which runs every
round, for few and for many rounds - where the soft threshold, which falls with the rounds, reaches some groups only in late ones."""
import numpy as np
import pytest

from oracle import quant_oracle as qo
from tests.test_gpu_quantize import _near_bf16_boundary
from workloads import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("group", [32, 64, 128])
@pytest.mark.parametrize("iters,std", [(1, 0.02), (3, 0.02), (60, 0.02), (300, 0.02), (60, 0.2), (300, 0.2), (5, 4.0), (20, 1.0)])
def test_as_if_every_round_had_run(group, iters, std):
    from paper_2604_18396_b200 import binding
    w = synth.normal(31, group + iters, (67, group * 3), std, "cuda").bfloat16().contiguous()
    codes, scale, zero = binding.quantize_w4(w, group, iters)
    c_o, s_o, z_o, zf = qo.quantize_w4(w.float().cpu().numpy(), group, iters, return_float_zero=True)
    assert np.array_equal(scale.float().cpu().numpy(), s_o)
    # (as in test_gpu_quantize.py: where the soft threshold acts, the power's last bit may turn a rounding to bf16 over)
    near = _near_bf16_boundary(zf)
    assert near.mean() < 0.1
    assert np.array_equal(zero.float().cpu().numpy()[~near], z_o[~near])
    same = np.repeat(~near, group // 2, axis=1)
    assert np.array_equal(codes.cpu().numpy()[same], c_o[same])


@pytest.mark.parametrize("group", [32, 64, 128])
@pytest.mark.parametrize("std,mix", [(1e-22, 1.0), (1e22, 1.0), (0.02, 0.0), (0.02, 1e-25)])
def test_quotients_outside_the_range_of_the_reciprocal(group, std, mix):
    """Weights so small or large that the remainder of a quotient could underflow (these groups divide), and some such weights, or
    zeros, among ordinary ones."""
    from paper_2604_18396_b200 import binding
    w = synth.normal(37, group, (19, group * 3), 1.0, "cuda").float() * std
    if mix != 1.0:
        w[:, ::5] *= mix
    w = w.bfloat16().contiguous()
    codes, scale, zero = binding.quantize_w4(w, group, 5)
    c_o, s_o, z_o, zf = qo.quantize_w4(w.float().cpu().numpy(), group, 5, return_float_zero=True)
    assert np.array_equal(scale.float().cpu().numpy(), s_o)
    near = _near_bf16_boundary(zf)
    assert near.mean() < 0.1
    assert np.array_equal(zero.float().cpu().numpy()[~near], z_o[~near])
    same = np.repeat(~near, group // 2, axis=1)
    assert np.array_equal(codes.cpu().numpy()[same], c_o[same])
