"""Exit-layer projections of decode steps whose K is long enough for one CTA per SM: their runs of k-blocks summed in two
accumulators (up to 32 operand rows), with one CTA and with several per tile, an odd number of raw tiles, and the row count
from which a run keeps one accumulator and its old length."""
import numpy as np
import pytest
import torch

from tests.gpu_harness import INF, Pair
from workloads import rtn_w4, synth

pytestmark = pytest.mark.gpu

# gate/up of 120 tiles over eight and nine raw tiles of codes (one CTA per tile); QKV of 48 tiles over sixteen (clusters of three)
SHAPES = {"gateup8": (2048, 8, 2, 7680), "gateup9": (2304, 8, 2, 7680), "qkv16": (4096, 16, 16, 256)}


@pytest.fixture(scope="module", params=sorted(SHAPES))
def model(request):
    d, hq, hkv, F = SHAPES[request.param]
    shape = synth.ModelShape("h", 2, d, hq, hkv, 128, F, 1024, seed=11, resid_decay=0.5)
    bb = synth.make_backbone(shape, "cuda")
    rv = rtn_w4.make_river(bb, shape.group)
    to = lambda x, dev: x.to(dev) if isinstance(x, torch.Tensor) else (  # noqa: E731
        {k: to(v, dev) for k, v in x.items()} if isinstance(x, dict) else type(x)(to(v, dev) for v in x))
    return shape, (to(bb, "cpu"), to(rv, "cpu")), (bb, rv)


@pytest.mark.parametrize("rows", [5, 17, 32, 33])
def test_steps_match_oracle(model, rows):
    shape = model[0]
    p = Pair(model, rows, 16, rows, kv_store=1, storage_yardstick=True)
    slots = list(range(rows))
    p.prefill(slots, [synth.tokens(71, b, 1 + b % 2, shape.V).numpy() for b in range(rows)])
    for t in range(3):
        tk = synth.tokens(71, 100 + t, rows, shape.V).numpy()
        forced = np.array([2 if t == 2 and b % 3 else 1 for b in range(rows)], np.int32)  # all on the exit layer; some
        o, g = p.oracle_step(slots, tk, INF, forced), p.gpu_step(slots, tk, INF, forced)
        assert np.array_equal(g.exit_layer, o.exit_layer)
        p.compare_logits(g.logits, o.logits, f"step {t}")
    for b in range(rows):
        p.compare_kv(b, p.gpu.seq_len(b))
    assert p.gpu.stats().device_error == 0
    p.close()


@pytest.mark.parametrize("rows", [8, 24, 40, 61])
def test_sums_of_long_inputs(rows):
    """QKV of 4096 inputs on exit-layer weights that are exact in f16 (powers of two times small integers), activations in hi and lo
    parts: what is left is the error of the sums.  2.0e-7 of the result's norm with 1365 inputs per sum, 1.5e-7 with 1024 or fewer."""
    from paper_2604_18396_b200 import River, make_config
    shape = synth.ModelShape("q", 1, 4096, 32, 8, 128, 256, 1024, seed=12, resid_decay=1.0)
    g = torch.Generator(device="cuda").manual_seed(rows)
    dims = {"wq": (4096, 4096), "wk": (1024, 4096), "wv": (1024, 4096), "wo": (4096, 4096), "wg": (256, 4096), "wu": (256, 4096), "wd": (4096, 256)}
    w4, lay = {}, {"attn_norm": torch.ones(4096, dtype=torch.bfloat16, device="cuda")}
    lay["ffn_norm"] = lay["attn_norm"]
    full = {}
    for n, (o, i) in dims.items():
        codes = torch.randint(0, 256, (o, i // 2), generator=g, device="cuda", dtype=torch.uint8)
        w4[n] = (codes, torch.full((o, i // 64), 2.0 ** -8, device="cuda").bfloat16(), torch.full((o, i // 64), 7.0, device="cuda").bfloat16())
        full[n] = ((torch.stack((codes & 15, codes >> 4), -1).view(o, i).double() - 7.0) * 2.0 ** -8)
        lay[n] = full[n].bfloat16()
    emb = torch.zeros((1024, 4096), dtype=torch.bfloat16, device="cuda")
    r = River(make_config(shape, max_seqs=rows, max_pages_per_seq=1, n_pages=rows, max_batch=rows, entry_layer=0),
              {"embed": emb, "lm_head": emb, "final_norm": lay["attn_norm"], "layers": [lay]}, [w4])
    one = torch.zeros((1, 1024), dtype=torch.bfloat16, device="cuda")
    for b in range(rows):
        r.write_kv(b, 1, 0, one, one)  # position 0: no rotation
    h = (torch.randn((rows, 4096), generator=g, device="cuda") * 64).round() / 64  # (the sum of their squares is exact in 32 bits)
    q = torch.empty((rows, 4096), device="cuda")
    r.project_kv(1, True, list(range(rows)), h, q)
    torch.cuda.synchronize()
    x = h.double() * torch.rsqrt((h.double() ** 2).mean(-1, keepdim=True) + shape.rms_eps)
    want = x @ full["wq"].T
    assert ((q.double() - want).norm() / want.norm()).item() <= 1.75e-7
    r.close()
