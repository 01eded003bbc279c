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


# 193 rows: the shortest long pass; 225 / 300: last tiles of a few rows; several prompts in one pass and across two passes;
# 1150: a full pass and a rest of 126 rows for the batch kernels
@pytest.mark.parametrize("lens,depth", [([193], None), ([225], 2), ([40, 300, 9, 200], None), ([300, 17], 4), ([1150], None),
                                        ([700, 600], 3)])
def test_long_passes_match_oracle(mini8, lens, depth):
    shape = mini8[0]
    p = Pair(mini8, len(lens), max(lens) + 8, 8, prefill_chunk=256, kv_store=1, storage_yardstick=True, page_shuffle_seed=3)
    slots = list(range(len(lens)))
    p.prefill(slots, [synth.tokens(41, b, n, shape.V).numpy() for b, n in enumerate(lens)], depth, logits=True)
    for b, n in enumerate(lens):
        p.compare_kv(b, n, f"lens {lens} depth {depth}")
    tk = synth.tokens(41, 99, len(lens), shape.V).numpy()
    o = p.oracle_step(slots, tk, INF)
    g = p.gpu_step(slots, tk, INF)
    p.compare_logits(g.logits, o.logits, "step after the prompts")
    assert p.gpu.stats().device_error == 0
    p.close()


def test_mixed_depths_in_one_pass(mini8):
    """Depth chosen per prompt by Eq. 1, thresholds between the per-block minima of the oracle's scores (never within 2.5e-3 of
    one, so the depths are unambiguous): one pass of 145 rows (a long one: short passes end at prefill_chunk) holds rows on both weight
    sets; depths, logits and cache."""
    shape = mini8[0]
    lens, L, lo = [60, 45, 40], shape.L, max(shape.entry_layer, 1)
    prompts = [synth.tokens(43, b, n, shape.V).numpy() for b, n in enumerate(lens)]
    probe = Pair(mini8, 1, max(lens) + 2, 4)
    mins = []
    for pr in prompts:
        sc = np.stack([probe.oracle.decode_step([0], [tk], INF)["scores"][0] for tk in pr])
        probe.oracle.release(0)
        mins.append(sc[:, lo - 1:L - 1].min(axis=0))
    probe.close()
    mins = np.stack(mins)
    edges = np.sort(mins.ravel())
    taus = [float(t) for t in 0.5 * (edges[:-1] + edges[1:]) if np.abs(mins - t).min() > 2.5e-3]
    first = lambda t: [next((lo + i for i in range(L - lo) if m[i] > t), L) for m in mins]  # noqa: E731
    mixed = [t for t in taus if len(set(first(t))) > 1]
    assert mixed, "no threshold separates the prompts"
    for tau in mixed[::max(1, len(mixed) // 4)]:
        p = Pair(mini8, 3, max(lens) + 2, 8, prefill_chunk=128, page_shuffle_seed=9)
        want = [p.oracle.prefill_auto(b, pr, tau) for b, pr in enumerate(prompts)]
        offs = np.concatenate([[0], np.cumsum(lens)]).tolist()
        lg = torch.empty((3, shape.V), device="cuda")
        got = p.gpu.prefill([0, 1, 2], torch.from_numpy(np.concatenate(prompts)).int().cuda(), offs, -1, lg, tau=tau)
        torch.cuda.synchronize()
        assert got == [w[2] for w in want] and len(set(got)) > 1, (tau, got, [w[2] for w in want])
        p.compare_logits(lg.cpu().numpy(), np.stack([w[0] for w in want]), f"tau {tau}")
        for b, n in enumerate(lens):
            p.compare_kv(b, n, f"tau {tau}")
        p.close()


@pytest.mark.parametrize("exit_mode", [0, 1])
@pytest.mark.parametrize("depth", [0, 2, None])
def test_long_pass_from_the_first_block_on(mini8, depth, exit_mode):
    """Every row on the exit layers from block 1 on (depth 0), from block 3 on, never; both exit modes, and steps behind them."""
    shape = mini8[0]
    lens = [200, 3]
    p = Pair(mini8, 2, 210, 4, exit_mode, entry_layer=0, prefill_chunk=256, kv_store=1, storage_yardstick=True)
    p.prefill([0, 1], [synth.tokens(44, b, n, shape.V).numpy() for b, n in enumerate(lens)], depth, logits=True)
    for t in range(2):
        tk = synth.tokens(44, 90 + t, 2, shape.V).numpy()
        o, g = p.oracle_step([0, 1], tk, -2.0), p.gpu_step([0, 1], tk, -2.0)
        assert np.array_equal(g.exit_layer, o.exit_layer)
        p.compare_logits(g.logits, o.logits, f"step {t}")
    for b, n in enumerate(lens):
        p.compare_kv(b, n + 2)
    p.close()


def test_gate_and_up_in_either_order_in_memory(mini8):
    """One map covers the gate and the up matrix whichever of them lies first: the same bits both ways."""
    from paper_2604_18396_b200 import River, make_config
    shape, _, (bb, rv) = mini8
    tok = synth.tokens(45, 0, 150, shape.V).cuda()
    out = []
    for up_first in (False, True):
        layers = []
        for lay in bb["layers"]:
            both = torch.stack((lay["wu"], lay["wg"]) if up_first else (lay["wg"], lay["wu"]))
            layers.append(dict(lay, wg=both[1 if up_first else 0], wu=both[0 if up_first else 1]))
        r = River(make_config(shape, max_seqs=1, max_pages_per_seq=10, n_pages=10, max_batch=8, prefill_chunk=128),
                  dict(bb, layers=layers), rv)
        lg = torch.empty((1, shape.V), device="cuda")
        r.prefill([0], tok, [0, 150], None, lg)
        kv = r.read_kv(0, shape.L, 0, 150)
        torch.cuda.synchronize()
        out.append((lg.clone(), kv[0].clone(), kv[1].clone()))
        r.close()
    assert torch.isfinite(out[0][0]).all()
    assert all(torch.equal(x, y) for x, y in zip(*out))


@pytest.mark.parametrize("dh,gq", [(64, 1), (64, 2), (64, 4), (64, 8), (128, 1), (128, 2), (128, 4), (128, 8)])
def test_long_pass_attention_geometries(dh, gq):
    """Every head dim and group size of the attention kernel, prompts that end inside and on the edges of its query tiles
    (128 / gq positions), key tiles (128, in two streams) and pages (16): the second block's cache shows the attention of every position."""
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
