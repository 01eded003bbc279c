"""river_release and river_prefill wait for nothing: prompts whose pages go back, and out again, while the kernels that fill and read
them are still queued, against the same calls with a synchronisation after each; and what a caller on another stream than the
context's may do behind them without one."""
import pytest
import torch

from paper_2604_18396_b200 import River, binding, make_config
from tests.gpu_harness import draw_model
from workloads import synth

pytestmark = pytest.mark.gpu

HOLD = 60_000_000  # cycles (30 ms) that a kernel of torch's keeps the context's stream busy: the host is far ahead meanwhile


def hold(r):
    with torch.cuda.stream(r.stream):
        torch.cuda._sleep(HOLD)
        ev = torch.cuda.Event()
        ev.record()
    return ev


# long passes, several of them; short passes (the batch kernels; at four rows and fewer the decode attention); depths by Eq. 1; the
# strategy that gives a released slot its full depth back; a stream of the context's own
@pytest.mark.parametrize("lens,depth,strategy,flags", [([300, 9, 200], None, 0, 0), ([1100, 40], 3, 0, 0), ([20, 30], 4, 0, 0), ([3, 1], None, 0, 0),
                                                       ([60, 45], -1, 0, 0), ([20, 7], None, 2, 0), ([20, 7], None, 3, 0),
                                                       ([300, 9, 200], None, 0, binding.RIVER_F_GRAPH)])
def test_pages_handed_on_while_in_use(lens, depth, strategy, flags):
    shape, _, (bb, rv) = draw_model("mini8")
    pages = sum((n + 16) // 16 for n in lens)
    offs = [0]
    for n in lens:
        offs.append(offs[-1] + n)
    slots, B = list(range(len(lens))), len(lens)
    toks = [torch.cat([synth.tokens(71 + turn, b, n, shape.V) for b, n in enumerate(lens)]).int().cuda() for turn in range(5)]
    first = [t[:B].contiguous() for t in toks]
    tau = torch.full((B,), 0.9, device="cuda")
    out = {}
    for wait in (True, False):
        r = River(make_config(shape, max_seqs=B, max_pages_per_seq=80, n_pages=pages, max_batch=8, prefill_chunk=256,
                              kv_strategy=strategy, flags=flags), bb, rv)
        got = out[wait] = []
        torch.cuda.synchronize()
        held = None
        for turn in range(5):
            lg = torch.empty((B, shape.V), device="cuda")
            if turn:
                for s in (slots if turn % 2 else slots[::-1]):
                    r.release(s)
                assert wait or not held.query(), "release waited for the device"
            d = r.prefill(slots, toks[turn], offs, depth, lg, tau=0.5 + 0.1 * turn if depth == -1 else float("inf"))
            if turn and depth != -1:  # (a depth that the device finds is waited for)
                assert wait or not held.query(), "prefill waited for the device"
            if not wait:
                held = hold(r)  # what follows is queued behind it when the next turn's releases come
            nxt, ex = torch.empty(B, dtype=torch.int32, device="cuda"), torch.empty(B, dtype=torch.int32, device="cuda")
            lg2 = torch.empty_like(lg)
            r.decode_step(slots, first[turn], tau, None, lg2, nxt, ex)
            kv = [r.read_kv(b, shape.L, 0, 1) for b in slots]
            if wait:
                torch.cuda.synchronize()
            got.append((d, lg, lg2, nxt, ex, [x for pair in kv for x in pair]))
        torch.cuda.synchronize()
        assert r.stats().device_error == 0
        r.close()
    for a, b in zip(out[True], out[False]):
        assert a[0] == b[0]
        assert all(torch.equal(x, y) for x, y in zip(a[1:5], b[1:5]))
        assert all(torch.equal(x, y) for x, y in zip(a[5], b[5]))


def test_outputs_behind_release_and_prefill_on_a_stream_of_its_own():
    """A context with its own stream: torch's current stream reads a prompt's logits once its slot is released, a step's once the next
    prompt is queued, and memory that a prompt's tensors leave is not written before the prompt has read them - all without a
    synchronisation by the host."""
    shape, _, (bb, rv) = draw_model("mini8")
    r = River(make_config(shape, max_seqs=2, max_pages_per_seq=20, n_pages=40, max_batch=8, prefill_chunk=256, flags=binding.RIVER_F_GRAPH), bb, rv)
    prompt = synth.tokens(73, 0, 300, shape.V).int().cuda()
    other = torch.full_like(prompt, 1)
    step_tok, tau = prompt[:1].contiguous(), torch.full((1,), float("inf"), device="cuda")
    nxt, ex = torch.empty(1, dtype=torch.int32, device="cuda"), torch.empty(1, dtype=torch.int32, device="cuda")
    want, want_step = torch.empty((1, shape.V), device="cuda"), torch.empty((1, shape.V), device="cuda")
    r.prefill([0], prompt, [0, 300], None, want)
    r.decode_step([0], step_tok, tau, None, want_step, nxt, ex)
    torch.cuda.synchronize()
    r.release(0)
    for turn in range(3):
        lg, lg2 = torch.full_like(want, float("nan")), torch.full_like(want, float("nan"))
        torch.cuda.synchronize()
        held = hold(r)
        tok = prompt.clone()
        r.prefill([0], tok, [0, 300], None, lg)
        if turn == 2:
            del tok
            again = torch.empty_like(prompt).copy_(other)  # (takes tok's memory, were it free)
        r.decode_step([0], step_tok, tau, None, lg2, nxt, ex)
        if turn == 1:
            r.prefill([1], prompt[:20].contiguous(), [0, 20])
        r.release(0)
        if turn == 1:
            r.release(1)
        got, got_step = lg.clone(), lg2.clone()
        assert not held.query(), "the host waited"
        torch.cuda.synchronize()
        assert torch.equal(got, want) and torch.equal(got_step, want_step), turn
    # (the steps before a prompt, read behind it)
    lg2 = torch.full_like(want, float("nan"))
    r.prefill([0], prompt, [0, 300])
    torch.cuda.synchronize()
    held = hold(r)
    r.decode_step([0], step_tok, tau, None, lg2, nxt, ex)
    r.prefill([1], prompt, [0, 300])
    got = lg2.clone()
    assert not held.query(), "the host waited"
    torch.cuda.synchronize()
    assert torch.equal(got, want_step)
    assert r.stats().device_error == 0
    r.close()
