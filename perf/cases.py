"""Timing cases of the early-exit decode library: whole steps, prompts, single stages and the exit layers' quantiser.

Every case goes through the public binding (`paper_2604_18396_b200`), with inputs drawn from a seed on the GPU:
`listed()` names the cases, `draw(rng)` makes more of the same ranges, `prepare` builds what a program holds before the
call (weights, cache history, context), `run` makes ONE pass, `exact` states the result in 64-bit plain torch.

Model shapes are the repository's own (4-layer tiny model, `mini8`, the 1B- and 8B-class decoders), some with fewer
blocks than the full depth so that a case with its own weights and cache prepares quickly; a block's shape, which is what
the kernels see, is never reduced.  Rows that leave the backbone do so by threshold: tau = -2 lets a row go at the
first block the model allows (`entry_layer`), tau = +inf never, so no score can lie near its threshold.
"""
from __future__ import annotations

import math
import random

import torch

from paper_2604_18396_b200 import River, make_config
from paper_2604_18396_b200 import binding

INF = float("inf")
EPS, THETA, GROUP, PAGE = 1e-5, 10000.0, 64, 16
RESETS = 512  # decode steps a state takes before its sequences go back to their prompts

#        (layers, hidden, query heads, KV heads, head dim, FFN, vocabulary)
SHAPES = {
    "tiny": (4, 256, 4, 2, 64, 1024, 1024),
    "mini8": (6, 512, 8, 2, 128, 1536, 4096),
    "1b": (16, 2048, 32, 8, 64, 8192, 128256),
    "8b": (32, 4096, 32, 8, 128, 14336, 128256),
}
MATS = ("wq", "wk", "wv", "wo", "wg", "wu", "wd")


class _Shape:
    def __init__(self, case):
        L, self.d, self.Hq, self.Hkv, self.dh, self.F, self.V = SHAPES[case["shape"]]
        self.L = case.get("layers", L)
        self.entry_layer = case.get("entry", 1)
        self.rms_eps, self.rope_theta, self.group = EPS, THETA, GROUP

    def dims(self):
        q, kv = self.Hq * self.dh, self.Hkv * self.dh
        return {"wq": (q, self.d), "wk": (kv, self.d), "wv": (kv, self.d), "wo": (self.d, q), "wg": (self.F, self.d),
                "wu": (self.F, self.d), "wd": (self.d, self.F)}

    def params(self):
        return sum(a * b for a, b in self.dims().values())


def listed():
    return [
        # the smallest call there is: one token of a model that fits in cache; launches and latency are all of it
        {"name": "decode_tiny_r1", "kind": "decode", "shape": "tiny", "rows": 1, "lo": 32, "hi": 32, "exits": False},
        # one chat session on the 8B-class decoder, the token leaving the backbone half way (the headline workload)
        {"name": "decode_8b_r1", "kind": "decode", "shape": "8b", "rows": 1, "lo": 1024, "hi": 1024, "exits": True, "entry": 16},
        # a few sessions at once, contexts of unequal length, every token at full depth
        {"name": "decode_8b_r3", "kind": "decode", "shape": "8b", "layers": 8, "rows": 3, "lo": 100, "hi": 2000, "exits": False},
        # a small serving batch of the 1B-class decoder, half of the rows on the exit layers
        {"name": "decode_1b_r8", "kind": "decode", "shape": "1b", "rows": 8, "lo": 512, "hi": 512, "exits": True, "entry": 4},
        # the wide ragged serving batch, full depth: weights and cache both count
        {"name": "decode_8b_r64", "kind": "decode", "shape": "8b", "layers": 8, "rows": 64, "lo": 256, "hi": 4096, "exits": False},
        # the same batch with an odd row count and half of it on the exit layers: both weight sets in most blocks
        {"name": "decode_8b_r61_exits", "kind": "decode", "shape": "8b", "layers": 8, "rows": 61, "lo": 256, "hi": 2048, "exits": True, "entry": 2},
        # short ragged prompts on a small model, several per call
        {"name": "prefill_mini8_ragged", "kind": "prefill", "shape": "mini8", "prompts": 5, "lo": 9, "hi": 333, "depth": 6},
        # prompts that leave the backbone early (sequence-level exit): the exit layers' weights carry most blocks
        {"name": "prefill_1b_exit", "kind": "prefill", "shape": "1b", "layers": 8, "prompts": 2, "lo": 300, "hi": 900, "depth": 3, "entry": 2},
        # the usual prompt of the headline workload
        {"name": "prefill_8b_1024", "kind": "prefill", "shape": "8b", "layers": 8, "prompts": 1, "lo": 1024, "hi": 1024, "depth": 8},
        # the longest prompt of the wide batch, an odd length: attention over thousands of positions
        {"name": "prefill_8b_4001", "kind": "prefill", "shape": "8b", "layers": 4, "prompts": 1, "lo": 4001, "hi": 4001, "depth": 4},
        # one block's attention of a batch with long contexts, as the attention microbenchmark asks for it
        {"name": "attn_8b_16x8k", "kind": "attention", "Hq": 32, "Hkv": 8, "dh": 128, "rows": 16, "lo": 8192, "hi": 8192},
        # building an exit layer: the largest matrix of an 8B-class block through the zero-point refinement
        {"name": "quantize_8b_down", "kind": "quantize", "out": 4096, "in": 14336, "group": 64, "iters": 20},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("decode", "decode", "decode", "prefill", "prefill", "prefill", "attention", "quantize"))
    if kind == "quantize":
        group = rng.choice((32, 64, 128))
        return {"kind": kind, "out": _log(rng, 16, 8192), "in": group * _log(rng, 1, 8192 // group), "group": group,
                "iters": rng.choice((0, 5, 20))}
    if kind == "attention":
        Hkv, dh = rng.choice((2, 8)), rng.choice((64, 128))
        rows = _log(rng, 1, 100)
        hi = _log(rng, 16, max(17, min(16000, 130000 // rows)))
        return {"kind": kind, "Hq": 4 * Hkv, "Hkv": Hkv, "dh": dh, "rows": rows, "lo": rng.randint(1, hi), "hi": hi}
    shape, layers = rng.choice((("tiny", 4), ("mini8", 6), ("1b", 4), ("8b", 2)))
    entry = rng.randint(1, layers - 1)
    if kind == "decode":
        hi = _log(rng, 4, 2000)
        return {"kind": kind, "shape": shape, "layers": layers, "rows": _log(rng, 1, 150), "lo": rng.randint(1, hi), "hi": hi,
                "exits": rng.random() < 0.5, "entry": entry}
    hi = _log(rng, 4, 1500)
    return {"kind": kind, "shape": shape, "layers": layers, "prompts": _log(rng, 1, 6), "lo": rng.randint(1, hi), "hi": hi,
            "depth": rng.choice((layers, entry)), "entry": entry}


# ------------------------------------------------------------------------------------------------- inputs from a seed
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _normal(g, shape, std, dtype=torch.bfloat16):
    return torch.empty(shape, dtype=dtype, device="cuda").normal_(0.0, std, generator=g)


def _w4(w):
    """Min/max round-to-nearest 4-bit copy of a bf16 matrix: (codes u8, scale bf16, zero bf16)."""
    out, n = w.shape
    x = w.float().view(out, n // GROUP, GROUP)
    mn, mx = x.amin(2, keepdim=True), x.amax(2, keepdim=True)
    s = ((mx - mn) / 15.0).bfloat16().float()
    z = (-mn / s).bfloat16().float()
    q = (x / s).add_(z).round_().clamp_(0, 15).to(torch.uint8).view(out, n)
    return q[:, 0::2] | (q[:, 1::2] << 4), s.bfloat16().view(out, -1), z.bfloat16().view(out, -1)


def _model(case, seed):
    s, g = _Shape(case), _gen(seed)
    decay = 0.125 ** (1.0 / max(s.L - 1, 1))  # the blocks' contributions to the residual stream fall with depth
    one = lambda: (1.0 + _normal(g, (s.d,), 0.1)).bfloat16()  # noqa: E731
    bb = {"embed": _normal(g, (s.V, s.d), 0.02), "lm_head": _normal(g, (s.V, s.d), 0.02), "final_norm": one(), "layers": []}
    need = case.get("exits") or case.get("depth", s.L) < s.L
    river, rest = [], None
    for l in range(s.L):
        lay = {"attn_norm": one(), "ffn_norm": one()}
        for n, dim in s.dims().items():
            lay[n] = _normal(g, dim, 0.02 * (decay ** l if n in ("wo", "wd") else 1.0))
        bb["layers"].append(lay)
        if l < s.entry_layer:
            river.append(None)
        elif need:
            river.append({n: _w4(lay[n]) for n in MATS})
        else:  # no row ever leaves: the blocks share one copy
            rest = rest or {n: _w4(lay[n]) for n in MATS}
            river.append(rest)
    return s, bb, river


def _lengths(case, n):
    r = random.Random(n * 7919 + case["hi"])  # the lengths belong to the case: every seed has the same sizes
    return [r.randint(case["lo"], case["hi"]) for _ in range(n)]


def _decode_inputs(case, seed):
    s, bb, river = _model(case, seed)
    rows = case["rows"]
    lens, g = _lengths(case, rows), _gen(seed + 1)
    w = s.Hkv * s.dh
    hist = [[(_normal(g, (n, w), 1.0), _normal(g, (n, w), 1.0)) for _ in range(s.L)] for n in lens]
    tok = torch.randint(0, s.V, (rows,), generator=g, device="cuda", dtype=torch.int32)
    leaves = [case["exits"] and b % 2 == 0 for b in range(rows)]
    tau = torch.tensor([-2.0 if x else INF for x in leaves], device="cuda")
    return s, bb, river, lens, hist, tok, tau, leaves


def _prefill_inputs(case, seed):
    s, bb, river = _model(case, seed)
    lens = _lengths(case, case["prompts"])
    tok = torch.randint(0, s.V, (sum(lens),), generator=_gen(seed + 1), device="cuda", dtype=torch.int32)
    return s, bb, river, lens, tok


def _attention_inputs(case, seed):
    lens, g = _lengths(case, case["rows"]), _gen(seed)
    w = case["Hkv"] * case["dh"]
    hist = [(_normal(g, (n, w), 1.0), _normal(g, (n, w), 1.0)) for n in lens]
    return lens, hist, _normal(g, (case["rows"], case["Hq"] * case["dh"]), 1.0, torch.float32)


def _pages(n):
    return (n + PAGE - 1) // PAGE


def _write_history(st):
    for b, layers in enumerate(st["hist"]):
        for l, (k, v) in enumerate(layers):
            st["river"].write_kv(b, l + 1, 0, k, v)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "quantize":
        return {"kind": kind, "w": _normal(_gen(seed), (case["out"], case["in"]), 0.02), "group": case["group"],
                "iters": case["iters"]}
    if kind == "attention":
        lens, hist, q = _attention_inputs(case, seed)
        one = dict(case, shape="tiny", layers=1)  # a one-block model that only carries the cache
        s = _Shape(one)
        s.Hq, s.Hkv, s.dh, s.d, s.F, s.V, s.entry_layer = case["Hq"], case["Hkv"], case["dh"], 256, 256, 1024, 0
        g = _gen(seed + 2)
        lay = {n: _normal(g, dim, 0.02) for n, dim in s.dims().items()}
        lay["attn_norm"] = lay["ffn_norm"] = torch.ones(s.d, dtype=torch.bfloat16, device="cuda")
        bb = {"embed": _normal(g, (s.V, s.d), 0.02), "lm_head": _normal(g, (s.V, s.d), 0.02),
              "final_norm": torch.ones(s.d, dtype=torch.bfloat16, device="cuda"), "layers": [lay]}
        cfg = make_config(s, max_seqs=len(lens), max_pages_per_seq=_pages(max(lens)), n_pages=sum(map(_pages, lens)),
                          max_batch=len(lens))
        st = {"kind": kind, "river": River(cfg, bb, [{n: _w4(lay[n]) for n in MATS}]), "q": q, "out": torch.empty_like(q),
              "slots": list(range(len(lens))), "hist": [[kv] for kv in hist]}
        _write_history(st)
        return st
    if kind == "prefill":
        s, bb, river, lens, tok = _prefill_inputs(case, seed)
        cfg = make_config(s, max_seqs=len(lens), max_pages_per_seq=_pages(max(lens)), n_pages=sum(map(_pages, lens)),
                          max_batch=8, prefill_chunk=256)
        offs = [0]
        for n in lens:
            offs.append(offs[-1] + n)
        return {"kind": kind, "river": River(cfg, bb, river), "tok": tok, "offs": offs, "slots": list(range(len(lens))),
                "depth": case["depth"], "logits": torch.empty((len(lens), s.V), dtype=torch.float32, device="cuda")}
    s, bb, river, lens, hist, tok, tau, _ = _decode_inputs(case, seed)
    rows = case["rows"]
    cfg = make_config(s, max_seqs=rows, max_pages_per_seq=_pages(max(lens) + RESETS),
                      n_pages=sum(_pages(n + RESETS) for n in lens), max_batch=max(rows, 8),
                      flags=binding.RIVER_F_GRAPH)  # as the benchmark runs it
    st = {"kind": kind, "river": River(cfg, bb, river), "hist": hist, "tok": tok, "tau": tau, "slots": list(range(rows)), "steps": 0,
          "logits": torch.empty((rows, s.V), dtype=torch.float32, device="cuda"),
          "next": torch.empty(rows, dtype=torch.int32, device="cuda"),
          "exit": torch.empty(rows, dtype=torch.int32, device="cuda")}
    _write_history(st)
    return st


def run(st):
    kind = st["kind"]
    if kind == "quantize":
        return binding.quantize_w4(st["w"], st["group"], st["iters"])
    rv = st["river"]
    if kind == "attention":
        rv.attention(1, st["slots"], st["q"], st["out"])
        return st["out"]
    if kind == "prefill":
        if rv.seq_len(0):  # the request before this one is over: its pages go back, in the order that hands them out again
            for s in reversed(st["slots"]):
                rv.release(s)
        rv.prefill(st["slots"], st["tok"], st["offs"], st["depth"], st["logits"])
        return {"logits": st["logits"], "kv": rv.kv_pool}
    if st["steps"] == RESETS:
        for s in reversed(st["slots"]):
            rv.release(s)
        _write_history(st)
        st["steps"] = 0
    rv.decode_step(st["slots"], st["tok"], st["tau"], None, st["logits"], st["next"], st["exit"])
    st["steps"] += 1
    return {"logits": st["logits"], "exit": st["exit"]}


# ------------------------------------------------------------------------------------------------- sizes and bounds
def _mean_len(case):
    return 0.5 * (case["lo"] + case["hi"])


def work(case):
    kind = case["kind"]
    if kind == "quantize":
        n = case["out"] * case["in"]
        return {"bytes": n * (2.0 + 0.5 + 4.0 / case["group"]), "flops": 0.0}
    n = _mean_len(case)
    if kind == "attention":
        q = case["Hq"] * case["dh"]
        return {"bytes": case["rows"] * (n * case["Hkv"] * case["dh"] * 4.0 + 8.0 * q), "flops": case["rows"] * 4.0 * n * q}
    s = _Shape(case)
    q, kv_tok, P = s.Hq * s.dh, 4.0 * s.Hkv * s.dh, s.params()
    w4 = 0.5 + 4.0 / GROUP
    head = 2.0 * s.V * s.d
    if kind == "decode":
        rows = case["rows"]
        n_leave = (rows + 1) // 2 if case["exits"] else 0
        bf = s.L if n_leave < rows else s.entry_layer
        bits4 = s.L - s.entry_layer if n_leave else 0
        return {"bytes": P * (2.0 * bf + w4 * bits4) + rows * s.L * (n + 2) * kv_tok + head + rows * (2.0 * s.d + 4.0 * s.V),
                "flops": rows * (2.0 * P * s.L + 4.0 * n * q * s.L + head)}
    T, m = case["prompts"] * n, case["depth"]
    return {"bytes": P * (2.0 * m + w4 * (s.L - m)) + T * (s.L * kv_tok + 2.0 * s.d) + head + case["prompts"] * 4.0 * s.V,
            "flops": T * (2.0 * P * s.L + 2.0 * n * q * s.L) + case["prompts"] * head}


def tolerance(case):
    # About four times the distance from `exact` that was measured over these ranges: attention 3.4e-6, steps up to 1.7e-4
    # (the 1B-class decoder, half of the rows on f16 exit-layer weights), prompts up to 1.2e-3 (cached K and V: bf16 values
    # whose rounding a difference in the last bits of 32-bit sums turns over, block after block).
    return "exact" if case["kind"] == "quantize" else {"rel": {"attention": 1.5e-5, "decode": 7e-4, "prefill": 5e-3}[case["kind"]]}


# ------------------------------------------------------------------------------------------------- 64-bit statement
def _rms(x, gain):
    return x * torch.rsqrt((x * x).mean(-1, keepdim=True) + EPS) * gain.double()


def _rope(x, pos, dh):  # x [T, H, dh], rotate-half
    f = THETA ** (-2.0 * torch.arange(dh // 2, dtype=torch.float64, device=x.device) / dh)
    a = pos.double()[:, None] * f
    c, s = a.cos()[:, None], a.sin()[:, None]
    lo, hi = x[..., :dh // 2], x[..., dh // 2:]
    return torch.cat((lo * c - hi * s, hi * c + lo * s), -1)


def _full(w):  # a bf16 matrix, or (codes, scale, zero), in 64 bits
    if isinstance(w, torch.Tensor):
        return w.double()
    codes, scale, zero = w
    q = torch.stack((codes & 15, codes >> 4), -1).view(codes.shape[0], -1, GROUP).double()
    return ((q - zero.double()[..., None]) * scale.double()[..., None]).view(codes.shape[0], -1)


def _attend(q, k, v, pos, s):
    """q [T, Hq, dh] at positions pos against k, v [n, Hkv, dh] (position = index), causal."""
    out = torch.empty_like(q)
    g = s.Hq // s.Hkv
    for h in range(s.Hkv):
        for t in range(0, q.shape[0], 1024):
            p = pos[t:t + 1024]
            m = torch.arange(k.shape[0], device=q.device)[None] > p[:, None]
            for j in range(h * g, (h + 1) * g):
                a = (q[t:t + 1024, j] @ k[:, h].T) * s.dh ** -0.5
                out[t:t + 1024, j] = a.masked_fill_(m, -INF).softmax(-1) @ v[:, h]
    return out


def _block(s, lay, wts, h, pos, seqs, cache):
    """One decoder block in 64 bits over rows h: `wts` its matrices (either weight set), `seqs` [(rows, cached k, cached v)];
    K and V are bf16 values, as the cache stores them."""
    x = _rms(h, lay["attn_norm"])
    T = h.shape[0]
    q = _rope((x @ _full(wts["wq"]).T).view(T, s.Hq, s.dh), pos, s.dh)
    k = _rope((x @ _full(wts["wk"]).T).view(T, s.Hkv, s.dh), pos, s.dh).bfloat16().double()
    v = (x @ _full(wts["wv"]).T).view(T, s.Hkv, s.dh).bfloat16().double()
    o = torch.empty_like(q)
    for rows, kc, vc in seqs:
        kk = k[rows] if kc is None else torch.cat((kc.double().view(-1, s.Hkv, s.dh), k[rows]))
        vv = v[rows] if vc is None else torch.cat((vc.double().view(-1, s.Hkv, s.dh), v[rows]))
        o[rows] = _attend(q[rows], kk, vv, pos[rows], s)
        if cache is not None:
            cache(rows, k[rows], v[rows])
    h = h + o.view(T, -1) @ _full(wts["wo"]).T
    y = _rms(h, lay["ffn_norm"])
    gate = y @ _full(wts["wg"]).T
    return h + (gate * torch.sigmoid(gate) * (y @ _full(wts["wu"]).T)) @ _full(wts["wd"]).T


def exact(case, seed):
    kind = case["kind"]
    if kind == "quantize":
        return None  # whole numbers in a fixed order of 32-bit operations
    if kind == "attention":
        lens, hist, q = _attention_inputs(case, seed)
        s = _Shape(dict(shape="tiny"))
        s.Hq, s.Hkv, s.dh = case["Hq"], case["Hkv"], case["dh"]
        out = torch.empty(q.shape, dtype=torch.float64, device="cuda")
        for b, (k, v) in enumerate(hist):
            at = torch.tensor([lens[b] - 1], device="cuda")
            out[b] = _attend(q[b].double().view(1, s.Hq, s.dh), k.double().view(-1, s.Hkv, s.dh),
                             v.double().view(-1, s.Hkv, s.dh), at, s).view(-1)
        return out
    if kind == "prefill":
        s, bb, river, lens, tok = _prefill_inputs(case, seed)
        first, pages, seqs, pos, r = {}, 0, [], [], 0
        for n in lens:
            first[r] = pages
            seqs.append((slice(r, r + n), None, None))
            pos.append(torch.arange(n, device="cuda"))
            r, pages = r + n, pages + _pages(n)
        pos = torch.cat(pos)
        pool = torch.full((s.L, pages, 2, s.Hkv, PAGE, s.dh), float("nan"), dtype=torch.float64, device="cuda")
        h = bb["embed"][tok.long()].double()
        for l in range(s.L):
            def cache(rows, k, v):
                p = torch.arange(k.shape[0], device="cuda")
                pool[l, first[rows.start] + p // PAGE, 0, :, p % PAGE] = k
                pool[l, first[rows.start] + p // PAGE, 1, :, p % PAGE] = v
            h = _block(s, bb["layers"][l], bb["layers"][l] if l < case["depth"] else river[l], h, pos, seqs, cache)
        h = h[torch.tensor([q[0].stop - 1 for q in seqs], device="cuda")]
        return {"logits": _rms(h, bb["final_norm"]) @ bb["lm_head"].double().T, "kv": pool.view(-1)}
    s, bb, river, lens, hist, tok, tau, leaves = _decode_inputs(case, seed)
    pos = torch.tensor(lens, device="cuda")
    h = bb["embed"][tok.long()].double()
    for l in range(s.L):
        new = torch.empty_like(h)
        for gone in (False, True):
            at = [b for b in range(case["rows"]) if (leaves[b] and l >= s.entry_layer) == gone]
            if not at:
                continue
            i = torch.tensor(at, device="cuda")
            seqs = [(slice(j, j + 1), *hist[b][l]) for j, b in enumerate(at)]
            new[i] = _block(s, bb["layers"][l], river[l] if gone else bb["layers"][l], h[i], pos[i], seqs, None)
        h = new
    return {"logits": _rms(h, bb["final_norm"]) @ bb["lm_head"].double().T, "exit": None}
