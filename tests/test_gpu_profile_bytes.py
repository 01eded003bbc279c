"""The algorithmic bytes that river_profile_read reports for a long prefill pass, whose last block runs behind QKV at the prompt
ends only: K and V of all positions are written there, but only the prompt ends attend, on one weight set."""
import pytest

from paper_2604_18396_b200 import River, make_config
from tests.gpu_harness import draw_model
from workloads import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("depth", [None, 2])
def test_bytes_of_a_long_pass(depth):
    shape, _, (bb, rv) = draw_model("mini8")
    n, L = 200, shape.L
    r = River(make_config(shape, max_seqs=1, max_pages_per_seq=16, n_pages=16, max_batch=8, prefill_chunk=256), bb, rv)
    tok = synth.tokens(97, 0, n, shape.V).int().cuda()
    r.profile(True)
    r.prefill([0], tok, [0, n], depth)
    got = {x["name"]: x["alg_bytes_total"] for x in r.profile_read()}
    r.profile(False)
    kv, qdim = shape.Hkv * shape.dh, shape.Hq * shape.dh
    w4 = 0.25 + 2.0 / shape.group
    sets = sum(1.0 if l < (L if depth is None else depth) else w4 for l in range(L))  # weight bytes relative to bf16, over the blocks
    assert got["prefill_attn"] == pytest.approx(4.0 * kv * ((L - 1) * n * (n + 1) / 2 + n))
    assert got["o_proj_resid"] == pytest.approx(2.0 * qdim * shape.d * sets)
    assert got["qkv_rope_kv"] == pytest.approx(2.0 * (qdim + 2 * kv) * shape.d * sets + L * n * 4.0 * kv)
    r.close()
