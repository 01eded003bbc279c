"""What a long pass attends with at its prompt ends - the split-KV kernel over rows of the pass - against the oracle's logits: head dims
and group sizes, ends whose contexts make one split and many, more ends than a decode step has rows, on either weight set."""
import pytest
import torch

from tests.gpu_harness import Pair
from workloads import rtn_w4, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dh,gq,lens,depth", [(64, 1, [300, 1, 64, 65], None), (64, 8, [129, 700], None), (128, 4, [1000], 1), (128, 2, [17] * 40, None),
                                              (128, 8, [300, 129, 2], 1), (64, 4, [5] * 130, 1)])
def test_logits_of_the_ends(dh, gq, lens, depth):
    hkv = max(1, 512 // dh // gq, 128 // dh)
    shape = synth.ModelShape("e", 2, 256, hkv * gq, hkv, dh, 256, 1024, seed=7, resid_decay=1.0)
    bb = synth.make_backbone(shape, "cpu")
    for lay in bb["layers"]:  # scores of a few units, so that the running maximum moves
        lay["wq"] *= 12.0
    rv = rtn_w4.make_river(bb, shape.group)
    to = lambda x: x.cuda() if isinstance(x, torch.Tensor) else (  # noqa: E731
        {k: to(v) for k, v in x.items()} if isinstance(x, dict) else type(x)(to(v) for v in x))
    p = Pair((shape, (bb, rv), (to(bb), to(rv))), len(lens), max(lens) + 8, max(8, len(lens)), prefill_chunk=256, kv_store=1, page_shuffle_seed=5)
    p.prefill(list(range(len(lens))), [synth.tokens(49, b, n, shape.V).numpy() for b, n in enumerate(lens)], depth, logits=True)
    assert p.gpu.stats().device_error == 0
    p.close()
