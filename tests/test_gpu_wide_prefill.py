"""Long prefill passes (hundreds of rows through the pair kernels) against the oracle: cache, logits and unified depth."""
import numpy as np
import pytest
import torch

from tests.gpu_harness import INF, Pair, draw_model
from workloads import rtn_w4, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mini8():
    return draw_model("mini8")


# 129 rows: the shortest long pass; 225 / 300: last tiles of a few rows; several prompts in one pass and across two passes;
# 1150: a full pass and a rest of 126 rows for the batch kernels
@pytest.mark.parametrize("lens,depth", [([129], None), ([225], 2), ([40, 300, 9, 200], None), ([300, 17], 4), ([1150], None),
                                        ([700, 600], 3)])
def test_long_passes_match_oracle(mini8, lens, depth):
    shape = mini8[0]
    p = Pair(mini8, len(lens), max(lens) + 8, 8, prefill_chunk=256, kv_store=1, storage_yardstick=True, page_shuffle_seed=3)
    slots = list(range(len(lens)))
    p.prefill(slots, [synth.tokens(41, b, n, shape.V).numpy() for b, n in enumerate(lens)], depth)
    for b, n in enumerate(lens):
        p.compare_kv(b, n, f"lens {lens} depth {depth}")
    tk = synth.tokens(41, 99, len(lens), shape.V).numpy()
    o = p.oracle_step(slots, tk, INF)
    g = p.gpu_step(slots, tk, INF)
    p.compare_logits(g.logits, o.logits, "step after the prompts")
    assert p.gpu.stats().device_error == 0
    p.close()


def test_mixed_depths_in_one_pass(mini8):
    """Depth chosen per prompt by Eq. 1: one pass holds rows on both weight sets; the same prompts one by one, in short
    passes, choose the same depths and give the same cache and logits."""
    from paper_2604_18396_b200 import River, make_config
    shape, _, (bb, rv) = mini8
    lens = [150, 260, 90]
    toks = [synth.tokens(43, b, n, shape.V) for b, n in enumerate(lens)]
    offs = np.concatenate([[0], np.cumsum(lens)]).tolist()

    def context(chunk):
        return River(make_config(shape, max_seqs=3, max_pages_per_seq=20, n_pages=60, max_batch=8, prefill_chunk=chunk), bb, rv)

    long, short = context(256), context(64)
    all_tok = torch.cat(toks).cuda()
    # a threshold that separates the prompts: between the lowest and the highest of their smallest scores, found by trying
    seen = {}
    for tau in np.linspace(0.80, 0.999, 24):
        lg = torch.empty((3, shape.V), device="cuda")
        d = long.prefill([0, 1, 2], all_tok, offs, -1, lg, tau=float(tau))
        d2 = []
        lg2 = torch.empty((3, shape.V), device="cuda")
        for b in range(3):
            d2 += short.prefill([b], toks[b].cuda(), [0, lens[b]], -1, lg2[b:b + 1], tau=float(tau))
        torch.cuda.synchronize()
        seen[tuple(d)] = tau
        if d == d2:  # (a score within rounding of tau may pick another depth: nothing to compare then)
            assert (lg - lg2).abs().max() <= 2e-2
            for b, n in enumerate(lens):
                for l in range(1, shape.L + 1):
                    for x, y in zip(long.read_kv(b, l, 0, n), short.read_kv(b, l, 0, n)):
                        x, y = x.float(), y.float()
                        assert torch.isfinite(x).all()
                        assert ((x - y).norm() / y.norm()).item() <= 1e-2
        for c in (long, short):
            for b in (2, 1, 0):
                c.release(b)
    assert len(seen) > 1 and any(len(set(k)) > 1 for k in seen), f"no threshold separates the prompts: {list(seen)}"
    long.close()
    short.close()


@pytest.mark.parametrize("dh,gq", [(64, 1), (64, 2), (64, 4), (64, 8), (128, 1), (128, 2), (128, 4), (128, 8)])
def test_long_pass_attention_geometries(dh, gq):
    """Every head dim and group size of the attention kernel, prompts that end inside and on the edges of its query tiles
    (128 / gq positions), key tiles (64) and pages (16): the second block's cache shows the attention of every position."""
    hkv = max(1, 512 // dh // gq, 128 // dh)
    shape = synth.ModelShape("a", 2, 256, hkv * gq, hkv, dh, 256, 1024, seed=7, resid_decay=1.0)
    bb = synth.make_backbone(shape, "cpu")
    for lay in bb["layers"]:  # scores of a few units, so that the running maximum moves from tile to tile
        lay["wq"] *= 12.0
    rv = rtn_w4.make_river(bb, shape.group)
    to = lambda x: x.cuda() if isinstance(x, torch.Tensor) else (  # noqa: E731
        {k: to(v) for k, v in x.items()} if isinstance(x, dict) else type(x)(to(v) for v in x))
    lens = [400, 129, 1, 448, 16, 30]
    p = Pair((shape, (bb, rv), (to(bb), to(rv))), 6, 456, 8, prefill_chunk=256, kv_store=1, storage_yardstick=True, page_shuffle_seed=5)
    p.prefill(list(range(6)), [synth.tokens(47, b, n, shape.V).numpy() for b, n in enumerate(lens)])
    for b, n in enumerate(lens):
        p.compare_kv(b, n, f"dh {dh} gq {gq} prompt {n}")
    assert p.gpu.stats().device_error == 0
    p.close()
