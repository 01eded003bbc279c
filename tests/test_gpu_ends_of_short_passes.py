"""Short passes of 193 to 208 rows on the exit layers whose prompt ends go through the LM head's tensor-core kernel: the dequantising
kernel's CTAs ask for all of an SM's tensor memory there, the head's, of 16 and of 48 rows, for some of it beside them."""
import pytest
import torch

from tests.gpu_harness import Pair
from workloads import rtn_w4, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lens", [[40] * 5, [4] * 40 + [5] * 8])
def test_logits_of_the_ends(lens):
    shape = synth.ModelShape("e", 2, 1024, 16, 4, 64, 4096, 8192, entry_layer=0, seed=7, resid_decay=1.0)
    bb = synth.make_backbone(shape, "cpu")
    rv = rtn_w4.make_river(bb, shape.group)
    to = lambda x: x.cuda() if isinstance(x, torch.Tensor) else (  # noqa: E731
        {k: to(v) for k, v in x.items()} if isinstance(x, dict) else type(x)(to(v) for v in x))
    p = Pair((shape, (bb, rv), (to(bb), to(rv))), len(lens), max(lens) + 8, len(lens), prefill_chunk=256, kv_store=1, page_shuffle_seed=5)
    p.prefill(list(range(len(lens))), [synth.tokens(53, b, n, shape.V).numpy() for b, n in enumerate(lens)], 0, logits=True)
    assert p.gpu.stats().device_error == 0
    p.close()
