"""Long passes whose rows look back at 64 positions on average, or a few less or more (tests/test_long_attention.py has which attention
kernel they take), against the oracle."""
import pytest

from tests.gpu_harness import Pair, draw_model
from workloads import synth

pytestmark = pytest.mark.gpu


# mean look-back 63.5 and 64 (equal prompts), 63.7, 64.1 and 84 with a short prompt beside a long one, 96
@pytest.mark.parametrize("name,lens", [("mini8", [126, 126]), ("mini8", [127, 127]), ("mini8", [146, 97]), ("mini8", [147, 97]), ("mini8", [200, 60]), ("tiny", [191, 191])])
def test_prompts_match_oracle(name, lens):
    m = draw_model(name)
    p = Pair(m, len(lens), max(lens) + 8, 8, prefill_chunk=256, kv_store=1, storage_yardstick=True, page_shuffle_seed=3)
    p.prefill(list(range(len(lens))), [synth.tokens(85, b, n, m[0].V).numpy() for b, n in enumerate(lens)], None, logits=True)
    for b, n in enumerate(lens):
        p.compare_kv(b, n)
    p.close()
