"""Steps and short prefill passes whose rows are dealt out over several CTAs of a projection, against the oracle: row counts on both
sides of a tile's edge, lists of the two weight sets that end inside a tile, at its edge and before the last tile."""
import numpy as np
import pytest

from tests.gpu_harness import INF, Pair, draw_model
from workloads import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def models():
    return {n: draw_model(n) for n in ("mini8", "tiny")}


@pytest.mark.parametrize("name,rows", [("mini8", n) for n in (17, 32, 33, 48, 64, 65, 97, 128)] + [("tiny", n) for n in (16, 31, 100, 129)])
def test_steps_match_oracle(models, name, rows):
    shape = models[name][0]
    p = Pair(models[name], rows, 24, rows, kv_store=1, storage_yardstick=True, page_shuffle_seed=4)
    slots = list(range(rows))
    lens = [1 + b % 5 for b in slots]
    p.prefill(slots, [synth.tokens(81, b, n, shape.V).numpy() for b, n in enumerate(lens)])
    L = shape.L
    for t, gone in enumerate((0, rows, rows // 2, rows - 16, 1)):  # rows that leave after the first block they may
        tk = synth.tokens(81, 500 + t, rows, shape.V).numpy()
        lo = max(1, shape.entry_layer)
        forced = np.full(rows, L, np.int32)
        forced[np.random.default_rng(t).permutation(rows)[:gone]] = lo
        o, g = p.oracle_step(slots, tk, INF, forced), p.gpu_step(slots, tk, INF, forced)
        assert np.array_equal(g.exit_layer, o.exit_layer)
        p.compare_lists(rows)
        p.compare_logits(g.logits, o.logits, f"{rows} rows, {gone} gone")
    for b in (0, rows // 2, rows - 1):
        p.compare_kv(b, lens[b] + 5)
    assert p.gpu.stats().device_error == 0
    p.close()


@pytest.mark.parametrize("lens,depth", [([40], None), ([16, 17], 3), ([100, 20], 2), ([128], None)])
def test_short_passes_match_oracle(models, lens, depth):
    shape = models["mini8"][0]
    p = Pair(models["mini8"], len(lens), max(lens) + 8, 8, prefill_chunk=128, kv_store=1, storage_yardstick=True, page_shuffle_seed=3)
    p.prefill(list(range(len(lens))), [synth.tokens(82, b, n, shape.V).numpy() for b, n in enumerate(lens)], depth, logits=True)
    for b, n in enumerate(lens):
        p.compare_kv(b, n)
    p.close()
