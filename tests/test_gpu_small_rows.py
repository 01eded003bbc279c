"""Steps of two to four rows where their shared memory decides the launches: every row count has its own kernel instance, and
three and more rows of a K too long to be staged whole take two launches of half the inputs."""
import numpy as np
import pytest
import torch

from tests.gpu_harness import INF, Pair
from workloads import rtn_w4, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows", [2, 3, 4])
@pytest.mark.parametrize("F", [1024, 13184])  # 13184: the down projection's rows do not fit together; its half is an odd number of groups
def test_row_counts_and_long_inputs(rows, F):
    shape = synth.ModelShape("s", 3, 256, 4, 2, 64, F, 1024, seed=9, resid_decay=0.5)
    bb = synth.make_backbone(shape, "cpu")
    rv = rtn_w4.make_river(bb, shape.group)
    to = lambda x: x.cuda() if isinstance(x, torch.Tensor) else (  # noqa: E731
        {k: to(v) for k, v in x.items()} if isinstance(x, dict) else type(x)(to(v) for v in x))
    lens = [17, 5, 33, 9][:rows]
    p = Pair((shape, (bb, rv), (to(bb), to(rv))), rows, 64, 4)
    slots = list(range(rows))
    p.prefill(slots, [synth.tokens(53, b, n, shape.V).numpy() for b, n in enumerate(lens)])
    for t in range(4):
        tk = synth.tokens(53, 10 + t, rows, shape.V).numpy()
        forced = np.array([1 + (b + t) % 3 for b in range(rows)], np.int32)  # both weight sets, and each alone, over the blocks
        o, g = p.oracle_step(slots, tk, INF, forced), p.gpu_step(slots, tk, INF, forced)
        assert np.array_equal(g.exit_layer, o.exit_layer)
        p.compare_logits(g.logits, o.logits, f"step {t}")
    for b, n in enumerate(lens):
        p.compare_kv(b, n + 4)
    p.close()
