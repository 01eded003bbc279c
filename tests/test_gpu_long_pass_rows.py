"""Prompts on both sides of the row counts from which a pass is a long one, where that is not the smallest count there is."""
import pytest
import torch

from tests.gpu_harness import Pair
from workloads import rtn_w4, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def model():
    shape = synth.ModelShape("k", 3, 1024, 16, 4, 64, 2048, 1024, seed=13, resid_decay=0.5)
    bb = synth.make_backbone(shape, "cuda")
    rv = rtn_w4.make_river(bb, shape.group)
    to = lambda x, dev: x.to(dev) if isinstance(x, torch.Tensor) else (  # noqa: E731
        {k: to(v, dev) for k, v in x.items()} if isinstance(x, dict) else type(x)(to(v, dev) for v in x))
    return shape, (to(bb, "cpu"), to(rv, "cpu")), (bb, rv)


# 145 rows on the backbone, 185 with two blocks of three on the exit layers; chunks of 128 keep short passes to 128 rows
@pytest.mark.parametrize("chunk,lens,depth", [(256, [144], None), (256, [145], None), (256, [184], 1), (256, [100, 85], 1), (128, [130], 1)])
def test_prompts_match_oracle(model, chunk, lens, depth):
    shape = model[0]
    p = Pair(model, len(lens), max(lens) + 8, 8, prefill_chunk=chunk, kv_store=1, storage_yardstick=True)
    p.prefill(list(range(len(lens))), [synth.tokens(81, b, n, shape.V).numpy() for b, n in enumerate(lens)], depth)
    for b, n in enumerate(lens):
        p.compare_kv(b, n, f"chunk {chunk} prompts {lens} depth {depth}")
    assert p.gpu.stats().device_error == 0
    p.close()
