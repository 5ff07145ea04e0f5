"""GPU parity of decode attention over long caches whose tokens are all in one pool, with one
to four (sequence, KV head) pairs: each pair's one segment is spread over as many CTAs as the
partial slots allow.  Both entry points against the oracle's binary64 attention within the
documented tolerance (max-abs 2e-3, relative L2 1e-3), and nothing written past the
workspace."""
import math

import pytest

import oracle
from paper_2608_28911_gb300 import synthetic
from parity import ATOL, RTOL_L2, Pair, attention_errors

pytestmark = pytest.mark.gpu

T = 20000


@pytest.mark.parametrize("base,levels,r", [
    (0, (6, 5), (1, 1)),     # fast kernel, every token high
    (0, (8, 3), (1, 1)),     # general kernel
    (2, (6, 5), (1, 1)),     # rotated affine
    (0, (6, 5), (0, 1)),     # every token low
])
@pytest.mark.parametrize("H", [1, 2, 4])
@pytest.mark.parametrize("n", [0, 77])
def test_long_cache_with_an_empty_pool(base, levels, r, H, n):
    import torch
    from paper_2608_28911_gb300 import semkv
    p = Pair(base, levels[0], levels[1], 1, 1, H, 4 * H, T, r[0], r[1], seed=900 + H)
    p.quantize()
    if n:
        k, v = synthetic.kv(901, 1, 1, H, n)
        p.stage(k, v, synthetic.scores_zipf(902, 1, n))
    q = synthetic.queries(903 + H, 1, 4 * H)
    scale = 1.0 / math.sqrt(128)
    ref = oracle.decode_attention(p.oc, 0, synthetic.f16_bits(q), scale)
    qd = torch.from_numpy(q).to(p.dev)
    out = torch.full((1, 4 * H, 128), float("nan"), dtype=torch.float32, device=p.dev)
    words = semkv.semkv_decode_workspace_bytes(p.cache) // 4
    canary = -1234.5
    big = torch.full((words + 4096,), canary, dtype=torch.float32, device=p.dev)
    semkv.semkv_decode_attention(p.desc, p.cache, 0, qd, out, scale, big[:words])
    got = [out.cpu().numpy().copy()]
    assert bool((big[words:] == canary).all()), "decode wrote past the workspace"
    out.fill_(float("nan"))
    semkv.semkv_decode_attention_noalloc(p.desc, p.cache, 0, qd, out, scale)
    got.append(out.cpu().numpy())
    for g in got:
        err, rel = attention_errors(g, ref)
        assert err <= ATOL and rel <= RTOL_L2, (err, rel)
    assert int(p.cache.dev_error.item()) == 0
