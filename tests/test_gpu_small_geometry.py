"""Steps whose projections have inputs that no power of two divides evenly (the warps of a CTA hold a row with some to spare) and a few
weight rows per SM: one row and several, both weight sets, against the oracle."""
import numpy as np
import pytest
import torch

from tests.gpu_harness import INF, Pair
from workloads import rtn_w4, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows", [1, 3])
@pytest.mark.parametrize("d,heads,F", [(1408, 22, 4864), (896, 14, 1152), (576, 9, 4352)])
def test_ragged_inputs(d, heads, F, rows):
    shape = synth.ModelShape("g", 3, d, heads, heads, 64, F, 300, seed=17, resid_decay=0.5)
    bb = synth.make_backbone(shape, "cuda")
    rv = rtn_w4.make_river(bb, shape.group)
    to = lambda x, dev: x.to(dev) if isinstance(x, torch.Tensor) else (  # noqa: E731
        {k: to(v, dev) for k, v in x.items()} if isinstance(x, dict) else type(x)(to(v, dev) for v in x))
    p = Pair((shape, (to(bb, "cpu"), to(rv, "cpu")), (bb, rv)), rows, 40, 4, kv_store=1, storage_yardstick=True, flags=1)
    slots = list(range(rows))
    p.prefill(slots, [synth.tokens(107, b, 4 + b, shape.V).numpy() for b in slots])
    for t in range(4):
        tk = synth.tokens(107, 60 + t, rows, shape.V).numpy()
        forced = np.array([3 if (b + t) % 2 else 1 for b in slots], np.int32)
        o, g = p.oracle_step(slots, tk, INF, forced), p.gpu_step(slots, tk, INF, forced)
        p.compare_lists(rows)
        p.compare_logits(g.logits, o.logits, f"step {t}")
    for b in slots:
        p.compare_kv(b, 8 + b)
    p.close()
