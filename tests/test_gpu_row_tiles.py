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


# (192 rows and one more: the last short passes, the first long ones)
@pytest.mark.parametrize("lens,depth,chunk", [([40], None, 128), ([16, 17], 3, 128), ([100, 20], 2, 128), ([128], None, 128), ([192], None, 256),
                                              ([170, 23], None, 256), ([90, 102], 1, 256), ([193], 1, 256), ([150, 30], 0, 256)])
def test_short_passes_match_oracle(models, lens, depth, chunk):
    shape = models["mini8"][0]
    p = Pair(models["mini8"], len(lens), max(lens) + 8, 8, entry_layer=0 if depth == 0 else None, prefill_chunk=chunk, kv_store=1, storage_yardstick=True, page_shuffle_seed=3)
    p.prefill(list(range(len(lens))), [synth.tokens(82, b, n, shape.V).numpy() for b, n in enumerate(lens)], depth, logits=True)
    for b, n in enumerate(lens):
        p.compare_kv(b, n)
    p.close()


@pytest.mark.parametrize("name,lens,depth", [("mini8", [257], None), ("mini8", [320, 5], 1), ("tiny", [640], 1), ("tiny", [300, 33], None)])
def test_long_passes_match_oracle(models, name, lens, depth):
    """O and down of long passes on the batch kernel: last row tiles of one row, full ones, both weight sets."""
    shape = models[name][0]
    p = Pair(models[name], len(lens), max(lens) + 8, 8, prefill_chunk=256, kv_store=1, storage_yardstick=True, page_shuffle_seed=3)
    p.prefill(list(range(len(lens))), [synth.tokens(84, b, n, shape.V).numpy() for b, n in enumerate(lens)], depth, logits=True)
    for b, n in enumerate(lens):
        p.compare_kv(b, n)
    assert p.gpu.stats().device_error == 0
    p.close()


def test_mixed_depths(models):
    """Depths chosen per prompt by Eq. 1: passes of 120 and of 250 rows with rows on both weight sets, whose kernels are launched for
    the sets that have rows."""
    import torch
    shape = models["mini8"][0]
    L, lo = shape.L, max(shape.entry_layer, 1)
    for lens in ([50, 40, 30], [100, 90, 60]):
        prompts = [synth.tokens(83, b, n, shape.V).numpy() for b, n in enumerate(lens)]
        probe = Pair(models["mini8"], 1, max(lens) + 2, 4, kv_store=1)
        mins = []
        for pr in prompts:
            sc = np.stack([probe.oracle.decode_step([0], [tk], INF)["scores"][0] for tk in pr])
            probe.oracle.release(0)
            mins.append(sc[:, lo - 1:L - 1].min(axis=0))
        probe.close()
        mins = np.stack(mins)
        edges = np.sort(mins.ravel())
        first = lambda t: [next((lo + i for i in range(L - lo) if m[i] > t), L) for m in mins]  # noqa: E731
        taus = [float(t) for t in 0.5 * (edges[:-1] + edges[1:]) if np.abs(mins - t).min() > 2.5e-3 and len(set(first(t))) > 1]
        assert taus, "no threshold separates the prompts"
        for tau in taus[::max(1, len(taus) // 2)]:
            # (kv_store: the cache as both store it, 16 bits; of this many positions its roundings alone pass the plain bound)
            p = Pair(models["mini8"], 3, max(lens) + 2, 8, prefill_chunk=256, page_shuffle_seed=9, kv_store=1)
            want = [p.oracle.prefill_auto(b, pr, tau) for b, pr in enumerate(prompts)]
            offs = np.concatenate([[0], np.cumsum(lens)]).tolist()
            lg = torch.empty((3, shape.V), device="cuda")
            got = p.gpu.prefill([0, 1, 2], torch.from_numpy(np.concatenate(prompts)).int().cuda(), offs, -1, lg, tau=tau)
            torch.cuda.synchronize()
            assert got == [w[2] for w in want] and len(set(got)) > 1
            p.compare_logits(lg.cpu().numpy(), np.stack([w[0] for w in want]), f"tau {tau}")
            for b, n in enumerate(lens):
                p.compare_kv(b, n, f"tau {tau}")
            p.close()
