"""GPU parity of the staged tail beside the short pools of many (sequence, KV head) pairs, on
both sides of the rule that gives the tails a kernel of their own (a quarter of the wave's
slots), against the oracle within the documented tolerance."""
import pytest

from paper_2608_28911_gb300 import synthetic
from parity import ATOL, RTOL_L2, Pair, attention_errors

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("base,levels,B,H,T,n", [
    (0, (6, 5), 19, 4, 300, 77),    # 76 pairs: in the pools' grid
    (0, (6, 5), 11, 7, 300, 77),    # 77: apart
    (2, (6, 5), 16, 8, 520, 1),
    (0, (6, 5), 76, 2, 200, 33),    # 152 pairs
    (0, (4, 4), 11, 7, 300, 77),    # general kernel: after its wave
])
def test_tail_beside_many_short_pools(base, levels, B, H, T, n):
    p = Pair(base, levels[0], levels[1], B, 1, H, 4 * H, T, 26, 100, seed=970 + T)
    p.quantize()
    k, v = synthetic.kv(971, B, 1, H, n)
    p.stage(k, v, synthetic.scores_zipf(972, B, n))
    err, rel = attention_errors(*p.decode(0))
    assert err <= ATOL and rel <= RTOL_L2, (err, rel)
    assert int(p.cache.dev_error.item()) == 0
