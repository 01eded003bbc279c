"""Two contexts on one device: what one context sets up for a kernel must not take anything from the other's launches."""
import pytest
import torch

from paper_2604_18396_b200 import River, make_config
from tests.gpu_harness import draw_model
from workloads import synth

pytestmark = pytest.mark.gpu


def test_contexts_with_other_prompt_lengths_do_not_disturb_each_other():
    # a projection of 60 rows asks for more shared memory (three stages of 32 KB per CTA) than one of 12 (at most four of 20 KB), so a
    # limit that the second context set for its own launches alone would be too low for the first one's next prompt
    shape, _, (bb, rv) = draw_model("mini8")
    cfg = make_config(shape, max_seqs=1, max_pages_per_seq=8, n_pages=8, max_batch=8, prefill_chunk=64)
    a, b = River(cfg, bb, rv), River(cfg, bb, rv)
    tok = synth.tokens(3, 0, 60, shape.V).cuda()
    out = [torch.empty((1, shape.V), device="cuda") for _ in range(2)]
    a.prefill([0], tok, [0, 60], None, out[0])
    b.prefill([0], tok[:12].contiguous(), [0, 12])
    a.release(0)
    a.prefill([0], tok, [0, 60], None, out[1])
    torch.cuda.synchronize()
    assert torch.equal(out[0], out[1])
    a.close()
    b.close()
