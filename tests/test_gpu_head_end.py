"""The end of a small step: the LM head's last CTA merges the greedy tokens, notes the last block's score and the final row lists.
Vocabularies with fewer tasks than CTAs, with shares that differ by one, and one row against several (other kernels)."""
import numpy as np
import pytest
import torch

from tests.gpu_harness import INF, Pair
from workloads import rtn_w4, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows", [1, 2, 3, 4])
@pytest.mark.parametrize("V", [12, 300, 4100])
def test_tokens_scores_and_lists(rows, V):
    shape = synth.ModelShape("h", 3, 256, 4, 2, 64, 512, V, seed=13, resid_decay=0.5)
    bb = synth.make_backbone(shape, "cpu")
    bb["lm_head"][V // 2] = bb["lm_head"][V - 1]  # equal logits: the lower id wins
    rv = rtn_w4.make_river(bb, shape.group)
    to = lambda x: x.cuda() if isinstance(x, torch.Tensor) else (  # noqa: E731
        {k: to(v) for k, v in x.items()} if isinstance(x, dict) else type(x)(to(v) for v in x))
    p = Pair((shape, (bb, rv), (to(bb), to(rv))), rows, 40, 4, flags=1)
    slots = list(range(rows))
    p.prefill(slots, [synth.tokens(91, b, 5 + 3 * b, V).numpy() for b in slots])
    for t in range(4):  # (the third is the first replayed one)
        tk = synth.tokens(91, 50 + t, rows, V).numpy()
        forced = np.array([3 if (b + t) % 2 else 1 for b in slots], np.int32)
        o, g = p.oracle_step(slots, tk, INF, forced), p.gpu_step(slots, tk, INF, forced)
        p.compare_lists(rows)
        p.compare_logits(g.logits, o.logits, f"step {t}")
        assert np.array_equal(g.next_tok, np.argmax(g.logits, axis=1))  # (the first of equal ones)
        deep = forced == 3
        assert np.allclose(g.scores[deep, 2], o.scores[deep, 2], atol=1e-3) and np.isnan(g.scores[~deep, 2]).all()
    p.close()


@pytest.mark.parametrize("rows", [5, 9])
def test_more_rows_than_the_last_cta_merges(rows):
    """Steps whose LM head the CUDA-core kernel computes for five and more rows: a kernel with a CTA per row merges the tokens."""
    V = 300
    shape = synth.ModelShape("h", 3, 256, 4, 2, 64, 512, V, seed=13, resid_decay=0.5)
    bb = synth.make_backbone(shape, "cpu")
    bb["lm_head"][V // 2] = bb["lm_head"][V - 1]
    rv = rtn_w4.make_river(bb, shape.group)
    to = lambda x: x.cuda() if isinstance(x, torch.Tensor) else (  # noqa: E731
        {k: to(v) for k, v in x.items()} if isinstance(x, dict) else type(x)(to(v) for v in x))
    p = Pair((shape, (bb, rv), (to(bb), to(rv))), rows, 40, rows)
    slots = list(range(rows))
    p.prefill(slots, [synth.tokens(93, b, 2 + b, V).numpy() for b in slots])
    for t in range(2):
        tk = synth.tokens(93, 50 + t, rows, V).numpy()
        forced = np.array([3 if (b + t) % 2 else 1 for b in slots], np.int32)
        o, g = p.oracle_step(slots, tk, INF, forced), p.gpu_step(slots, tk, INF, forced)
        p.compare_lists(rows)
        p.compare_logits(g.logits, o.logits, f"step {t}")
        assert np.array_equal(g.next_tok, np.argmax(g.logits, axis=1))
        assert p.gpu.stats().launches_last_step == 1 + 6 * shape.L + 2  # (LM head and merge)
    assert sum(p.gpu.exit_histogram()) == 2 * rows
    p.close()
