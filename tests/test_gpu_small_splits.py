"""Steps of one to four rows whose contexts lie around the 64 positions a split of the small-step attention has at least, rows of one
step on different sides of it, and a captured step replayed while the number of splits grows."""
import numpy as np
import pytest

from tests.gpu_harness import INF, Pair, draw_model
from workloads import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mini8():
    return draw_model("mini8")


@pytest.mark.parametrize("lens", [[61], [1], [126], [63, 1], [62, 130, 5], [64, 65, 200, 16]])
def test_contexts_around_a_split(mini8, lens):
    shape, rows = mini8[0], len(lens)
    p = Pair(mini8, rows, max(lens) + 8, 4, kv_store=1, storage_yardstick=True, flags=1)
    slots = list(range(rows))
    p.prefill(slots, [synth.tokens(101, b, n, shape.V).numpy() for b, n in enumerate(lens)])
    for t in range(6):
        tk = synth.tokens(101, 300 + t, rows, shape.V).numpy()
        forced = np.array([1 + (b + t) % shape.L for b in slots], np.int32)
        o, g = p.oracle_step(slots, tk, INF, forced), p.gpu_step(slots, tk, INF, forced)
        assert np.array_equal(g.exit_layer, o.exit_layer)
        p.compare_logits(g.logits, o.logits, f"step {t}")
    for b, n in enumerate(lens):
        p.compare_kv(b, n + 6)
    p.close()
