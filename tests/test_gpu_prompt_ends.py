"""The last block of a long prefill pass runs behind QKV at the prompt ends only, on the kernels of decode steps: one, four, five and
more ends (the kernels change there), on either weight set, a pass whose ends are in the next one, against the oracle."""
import numpy as np
import pytest

from tests.gpu_harness import Pair, draw_model
from workloads import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mini8():
    return draw_model("mini8")


@pytest.mark.parametrize("depth", [6, 2])
@pytest.mark.parametrize("lens", [[150], [1030], [90, 3, 40, 31], [40, 30, 30, 20, 30], [17] * 20])
def test_logits_and_cache(mini8, lens, depth):
    shape = mini8[0]
    p = Pair(mini8, len(lens), max(lens) + 8, len(lens), kv_store=1, storage_yardstick=True, prefill_chunk=256)
    p.prefill(list(range(len(lens))), [synth.tokens(97, b, n, shape.V).numpy() for b, n in enumerate(lens)], depth, logits=True)
    for b, n in enumerate(lens):
        p.compare_kv(b, n)
    assert p.gpu.stats().device_error == 0
    p.close()
