"""GPU edge sizes of the staged tail: one token, around the 32-token rounding of its logits,
the largest stage, group sizes that do not divide the warps, beside every pool kernel (fast
and general affine, TurboQuant, the 16-warp kernel's separate launch) and without pools; and
the four-level byte lookups at ragged pool sizes.  Attention against the oracle, or binary64
attention where there are no pools, within the documented tolerance."""
import math

import numpy as np
import pytest

import oracle
from paper_2608_28911_gb300 import synthetic
from parity import ATOL, RTOL_L2, Pair, attention_errors

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("base,levels,B,H,G,T,n", [
    (0, (6, 5), 1, 8, 4, 700, 1),        # 8-warp fast kernel
    (0, (6, 5), 2, 2, 3, 90, 33),
    (0, (6, 5), 20, 8, 4, 2200, 31),     # 16-warp fast kernel: the tail in its own launch
    (0, (4, 4), 1, 3, 8, 333, 32),       # general kernel, groups of eight
    (0, (6, 5), 3, 8, 4, 14700, 47),     # 8-warp kernels over long ranges: a launch of its own
    (0, (4, 4), 3, 8, 4, 14700, 47),
    (0, (8, 3), 2, 1, 5, 17, 200),
    (2, (6, 5), 1, 2, 1, 50, 1024),      # the largest stage
    (1, (4, 3), 2, 2, 8, 257, 65),       # TurboQuant kernel
    (1, (5, 4), 1, 2, 3, 40, 7),         # its CUDA-core path beside the tensor-core one
    (3, (4, 3), 1, 2, 4, 100, 40),       # dense rotation
])
def test_staged_tail_beside_every_pool_kernel(base, levels, B, H, G, T, n):
    p = Pair(base, levels[0], levels[1], B, 1, H, H * G, T, 1, 2, seed=600 + n, block=1024)
    p.quantize()
    if base == oracle.BASE_TQ_DENSE:
        p.adopt_gpu_records()
    k, v = synthetic.kv(601 + n, B, 1, H, n)
    p.stage(k, v, synthetic.scores_zipf(602 + n, B, n))
    for seed in (0, 1):
        err, rel = attention_errors(*p.decode(0, seed))
        assert err <= ATOL and rel <= RTOL_L2, (err, rel)
    assert int(p.cache.dev_error.item()) == 0


@pytest.mark.parametrize("base", [0, 1, 2])
@pytest.mark.parametrize("n,G", [(1, 4), (32, 8), (100, 3)])
def test_staged_tokens_without_pools(base, n, G):
    import torch
    from paper_2608_28911_gb300 import semkv
    B, H = 2, 3
    signs = synthetic.signs(5, 1, H) if base else None
    desc = semkv.QuantDesc(base, 4, 3, signs=signs)
    cache = semkv.KVCache(desc, B, 1, H, H * G, hi_cap=16, lo_cap=16)
    k, v = synthetic.kv(700 + n, B, 1, H, n)
    cache.stage_k[:, :, :, :n] = torch.from_numpy(k).cuda()
    cache.stage_v[:, :, :, :n] = torch.from_numpy(v).cuda()
    cache.s.stage_n = n
    q = synthetic.queries(701 + n, B, H * G)
    out = torch.full((B, H * G, 128), -7.0, dtype=torch.float32, device="cuda")
    scale = 1.0 / math.sqrt(128)
    semkv.semkv_decode_attention(desc, cache, 0, torch.from_numpy(q).cuda(), out, scale, cache.workspace())
    torch.cuda.synchronize()
    q64 = q.astype(np.float64).reshape(B, H, G, 128)
    lg = np.einsum("bhgd,bhtd->bhgt", q64, k[:, 0].astype(np.float64)) * scale
    w = np.exp(lg - lg.max(-1, keepdims=True))
    ref = np.einsum("bhgt,bhtd->bhgd", w / w.sum(-1, keepdims=True), v[:, 0].astype(np.float64))
    err, rel = attention_errors(out.cpu().numpy(), ref.reshape(B, H * G, 128))
    assert err <= ATOL and rel <= RTOL_L2, (err, rel)


@pytest.mark.parametrize("base", [0, 1, 2])
@pytest.mark.parametrize("G", [1, 4, 8])
@pytest.mark.parametrize("T", [1, 15, 16, 17, 400])
def test_four_level_lookups_at_ragged_sizes(base, G, T):
    p = Pair(base, 4, 4, 1, 1, 2, 2 * G, T, 0, 1, seed=800 + T)
    p.quantize()
    err, rel = attention_errors(*p.decode(0))
    assert err <= ATOL and rel <= RTOL_L2, (err, rel)
