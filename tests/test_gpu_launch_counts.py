"""river_stats_t.launches_last_step against the kernels that ran on the device, over every kind of step and prefill pass."""
import numpy as np
import pytest
import torch
from torch.profiler import ProfilerActivity, profile

from paper_2604_18396_b200 import River, binding, make_config
from tests.gpu_harness import draw_model
from workloads import synth

pytestmark = pytest.mark.gpu


def kernels(f):
    torch.cuda.synchronize()
    with profile(activities=[ProfilerActivity.CPU, ProfilerActivity.CUDA]) as prof:
        f()
        torch.cuda.synchronize()
    return sum(1 for e in prof.events() if e.device_type == torch.autograd.DeviceType.CUDA and "river::" in e.name)


@pytest.mark.parametrize("rows,flags,strategy", [(1, 0, 0), (3, 0, 0), (6, 0, 0), (6, binding.RIVER_F_SERIAL_TC, 0),
                                                 (6, binding.RIVER_F_NO_W4TC, 0), (2, 0, 1), (6, 0, 1), (6, 0, 3)])
def test_decode_steps(rows, flags, strategy):
    shape, _, (bb, rv) = draw_model("tiny")
    r = River(make_config(shape, max_seqs=8, max_pages_per_seq=2, n_pages=16, max_batch=8, flags=flags, kv_strategy=strategy), bb, rv)
    tok = synth.tokens(91, 0, 8, shape.V).int().cuda()
    slots = list(range(rows))
    r.prefill(slots, tok[:rows].contiguous(), list(range(rows + 1)))
    tau = torch.tensor([-2.0 if b % 2 else float("inf") for b in slots], device="cuda")
    nx, ex = (torch.empty(rows, dtype=torch.int32, device="cuda") for _ in range(2))
    step = lambda: r.decode_step(slots, tok[:rows].contiguous(), tau, None, None, nx, ex)  # noqa: E731
    step()
    n = kernels(step)
    assert n > 0 and n == r.stats().launches_last_step
    r.close()


@pytest.mark.parametrize("lens,tau", [([20], 0.0), ([150], 0.0), ([60, 45, 40], 0.9), ([60, 45, 40], 2.0),
                                      ([200], 0.0), ([90, 65, 60], 0.9), ([90, 65, 60], 2.0)])
def test_prefill_passes(lens, tau):
    """Short passes and (200 rows and more) long ones.  tau 0.9 lies between the prompts' scores often enough for rows on both weight
    sets; 2: every row on the backbone."""
    shape, _, (bb, rv) = draw_model("mini8")
    r = River(make_config(shape, max_seqs=3, max_pages_per_seq=13, n_pages=39, max_batch=8, prefill_chunk=256), bb, rv)
    tok = torch.cat([synth.tokens(43, b, n, shape.V) for b, n in enumerate(lens)]).int().cuda()
    offs = np.concatenate([[0], np.cumsum(lens)]).tolist()
    before = r.stats().launches_total
    n = kernels(lambda: r.prefill(list(range(len(lens))), tok, offs, -1, None, tau=tau))
    assert n > 0 and n == r.stats().launches_total - before
    r.close()
