"""The step metadata is laid out for decode steps and short prefill passes, and for long passes, in turn: steps replayed as a
graph before and after a long pass, and what a short prompt uploads in a context that can run long passes."""
import os
import subprocess
import sys

import numpy as np
import pytest

from paper_2604_18396_b200 import binding
from tests.gpu_harness import INF, Pair, draw_model
from workloads import synth

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def mini8():
    return draw_model("mini8")


def test_steps_in_a_graph_around_long_and_short_passes(mini8):
    shape = mini8[0]
    lens = [21, 7, 300, 4, 170, 33]
    p = Pair(mini8, 6, 320, 6, prefill_chunk=256, kv_store=1, storage_yardstick=True, page_shuffle_seed=2, flags=binding.RIVER_F_GRAPH)
    prompts = [synth.tokens(61, b, n, shape.V).numpy() for b, n in enumerate(lens)]
    t = 0

    def steps(slots, n):
        nonlocal t
        for _ in range(n):
            tk = synth.tokens(61, 100 + t, len(slots), shape.V).numpy()
            lo = max(1, shape.entry_layer)
            forced = np.array([lo + (b + t) % (shape.L + 1 - lo) for b in range(len(slots))], np.int32)
            o, g = p.oracle_step(slots, tk, INF, forced), p.gpu_step(slots, tk, INF, forced)
            assert np.array_equal(g.exit_layer, o.exit_layer)
            p.compare_logits(g.logits, o.logits, f"step {t}")
            t += 1

    p.prefill([0, 1], prompts[:2])               # a short pass
    steps([0, 1], 3)                             # the second step is captured, the third replayed
    p.prefill([2], prompts[2:3])                 # a long pass: the other layout, on the device and in the staging blocks
    steps([0, 1], 2)                             # the graph from before it
    steps([0, 1, 2], 3)
    p.prefill([3, 4, 5], prompts[3:], 4)         # 207 rows of three prompts, a long pass, leaving after block 4
    steps([3, 4, 5, 0, 1, 2], 3)                 # six rows: the batch kernels
    steps([0, 1], 1)
    for b in range(6):
        p.compare_kv(b, p.gpu.seq_len(b))
    assert p.gpu.stats().device_error == 0
    p.close()


UPLOAD = """
import json, sys, torch
from torch.profiler import ProfilerActivity, profile
from paper_2604_18396_b200 import River, binding, make_config
from tests.gpu_harness import draw_model
from workloads import synth
shape, _, (bb, rv) = draw_model("mini8")
for flags in (0, binding.RIVER_F_NO_W4TC):  # (the flag leaves the context without long passes)
    r = River(make_config(shape, max_seqs=2, max_pages_per_seq=32, n_pages=64, max_batch=8, prefill_chunk=256, flags=flags), bb, rv)
    tok = synth.tokens(67, 0, 300, shape.V).cuda()
    r.prefill([1], tok, [0, 300])
    torch.cuda.synchronize()
    with profile(activities=[ProfilerActivity.CPU, ProfilerActivity.CUDA]) as prof:
        r.prefill([0], tok[:20].contiguous(), [0, 20])
        torch.cuda.synchronize()
    prof.export_chrome_trace(sys.argv[1])
    ev = json.load(open(sys.argv[1]))["traceEvents"]
    print(sum(e["args"]["bytes"] for e in ev if "HtoD" in e.get("name", "") and "bytes" in e.get("args", {})))
    r.close()
"""


def test_a_short_prompt_uploads_no_more_than_without_long_passes(tmp_path):
    # (in a process of its own: the trace then holds this context's copies and nothing else)
    out = subprocess.run([sys.executable, "-c", UPLOAD, str(tmp_path / "t.json")], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert out.returncode == 0, out.stderr[-2000:]
    with_long, without = (int(x) for x in out.stdout.split()[-2:])
    assert 0 < with_long <= without
