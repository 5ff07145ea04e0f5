"""GPU edge sizes of the rows quantizer (TQ and rotated affine, 8-slot tiles, two lanes per
row): pools of one slot to a few tiles, records that start off a 16-byte boundary (odd block
appends), both pools and every level count, and rows whose parameters are limited or
subnormal beside ordinary ones (the rows that still need their codes clamped).  Records are
compared bit for bit with the oracle."""
import numpy as np
import pytest

import oracle
from paper_2608_28911_gb300 import synthetic
from parity import Pair

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("base", [1, 2])
@pytest.mark.parametrize("L_hi,L_lo,T,r,blk", [
    (4, 3, 1, (0, 1), 1),       # one slot, then one at a time
    (6, 5, 7, (1, 2), 3),
    (8, 7, 9, (1, 3), 5),
    (2, 4, 16, (1, 2), 7),
    (5, 6, 33, (1, 1), 9),      # the high pool only, until blocks add low slots
    (3, 8, 130, (26, 100), 31),
])
def test_rows_tiles_and_unaligned_appends_bit_exact(base, L_hi, L_lo, T, r, blk):
    import torch
    from paper_2608_28911_gb300 import semkv
    n = 3 * blk
    p = Pair(base, L_hi, L_lo, 2, 2, 3, 6, T, r[0], r[1], seed=900 + T, block=blk, extra_cap=n)
    p.quantize()
    p.assert_records_equal()
    k, v = synthetic.kv(901 + T, 2, 2, 3, n)
    s = synthetic.scores_zipf(902 + T, 2, n)
    for i in range(3):
        at = slice(i * blk, (i + 1) * blk)
        p.stage(k[:, :, :, at], v[:, :, :, at], s[:, at])
        semkv.semkv_append_block(p.desc, p.cache, 1, 2)
        oracle.append_block(p.oc, 1, 2)
    torch.cuda.synchronize()
    p.assert_records_equal()
    p.assert_untouched_past_counts()
    assert int(p.cache.dev_error.item()) == 0


@pytest.mark.parametrize("L", [2, 3, 4, 5, 6, 7, 8])
def test_rotated_rows_with_limited_and_subnormal_parameters(L):
    """Rows of one warp's tile that take the clamped codes beside rows that do not: values
    near fp16's largest (offset and step limited), tiny values (subnormal steps, whose
    rounding is coarse), constant and zero rows."""
    import torch
    from paper_2608_28911_gb300 import semkv
    p = Pair(2, L, L, 1, 1, 2, 4, 40, 0, 1, seed=77)
    rng = np.random.default_rng(5)
    for x in (p.k, p.v):
        x[0, 0, :, 3] = np.float16(60000.0) * np.sign(rng.standard_normal((2, 128)))
        x[0, 0, :, 5] = np.float16(65504.0)
        x[0, 0, :, 12] = (rng.integers(-3, 4, (2, 128)) * 2.0 ** -24).astype(np.float16)
        x[0, 0, :, 13] = (rng.integers(-40, 41, (2, 128)) * 2.0 ** -24).astype(np.float16)
        x[0, 0, :, 20] = 0.0
        x[0, 0, :, 21] = np.float16(-2.5)
    p.quantize()
    torch.cuda.synchronize()
    p.assert_records_equal()


@pytest.mark.parametrize("base,L_hi,L_lo", [(1, 4, 3), (1, 2, 8), (2, 6, 5), (2, 3, 7)])
@pytest.mark.parametrize("T,mixed", [(1, False), (7, True), (8, True), (9, True), (257, False)])
def test_fake_rows_tile_edges_bit_exact(base, L_hi, L_lo, T, mixed):
    """Fake quantization of the rotated bases at the edges of its 8-token tiles, with a row of
    limited parameters, one of subnormal steps and a zero row."""
    import torch
    from paper_2608_28911_gb300 import semkv
    B, NL, H = 2, 2, 3
    k, v = synthetic.kv(300 + T, B, NL, H, T)
    rng = np.random.default_rng(T)
    k[0, 0, 1, T // 2] = np.float16(60000.0) * np.sign(rng.standard_normal(128)).astype(np.float16)
    k[1, 1, 0, 0] = (rng.integers(-3, 4, 128) * 2.0 ** -24).astype(np.float16)
    v[1, 0, 2, T - 1] = 0.0
    ih = (rng.random((B, T)) < 0.4).astype(np.uint8) if mixed else None
    sg = synthetic.signs(301 + T, NL, H)
    kw = dict(signs=sg)
    if base == 1:
        kw["cb_hi"], kw["cb_lo"] = [oracle.lloyd_max_gaussian(L)[1:3] for L in (L_hi, L_lo)]
    desc = semkv.QuantDesc(base, L_hi, L_lo, signs=sg)
    kt, vt = torch.from_numpy(k).cuda(), torch.from_numpy(v).cuda()
    n, pad, canary = kt.numel(), 64, 0x7BCD
    big = [torch.full((n + 2 * pad,), canary, dtype=torch.int16, device="cuda") for _ in range(2)]
    ko, vo = [x[pad:pad + n].view(torch.float16).view(kt.shape) for x in big]
    semkv.semkv_fake_quant(desc, kt, vt, ko, vo, is_high=None if ih is None else torch.from_numpy(ih).cuda())
    torch.cuda.synchronize()
    for x in big:
        g = x.cpu().numpy()
        assert np.all(g[:pad] == canary) and np.all(g[pad + n:] == canary)
    want = oracle.fake_quant(base, L_hi, L_lo, synthetic.f16_bits(k), synthetic.f16_bits(v),
                             is_high=ih, **kw)
    for got, w in zip((ko, vo), want):
        assert np.array_equal(got.cpu().numpy().view(np.uint16), w)


@pytest.mark.parametrize("L_hi,L_lo,T,r,blk,shift", [
    (6, 5, 1, (0, 1), 1, 0),       # one slot, then one at a time
    (2, 3, 5, (1, 2), 3, 4),       # rows on 8-byte boundaries
    (8, 7, 9, (1, 3), 5, 0),
    (5, 4, 67, (1, 1), 9, 4),      # the high pool only, until blocks add low slots
    (3, 2, 131, (26, 100), 30, 0),
])
def test_affine_units_and_unaligned_appends_bit_exact(L_hi, L_lo, T, r, blk, shift):
    """The affine quantizer's 4-slot units: remainders, records that start off a 16-byte
    boundary, prompt rows on 8-byte boundaries only, NaN and infinity beside ordinary rows
    of the same unit, limited and subnormal steps."""
    import torch
    from paper_2608_28911_gb300 import semkv
    n = 2 * blk
    p = Pair(0, L_hi, L_lo, 2, 1, 2, 4, T, r[0], r[1], seed=400 + T, block=blk, extra_cap=n)
    rng = np.random.default_rng(T)
    for x in (p.k, p.v):
        x[0, 0, 0, T // 2, 7] = np.nan
        x[0, 0, 1, T - 1] = np.float16(65504.0) * np.sign(rng.standard_normal(128)).astype(np.float16)
        x[1, 0, 0, 0] = (rng.integers(-9, 10, 128) * 2.0 ** -24).astype(np.float16)
        x[1, 0, 1, T - 1, 3] = np.inf
    if shift:  # the same rows at an address that is 8 modulo 16
        d = p.dev
        p.o_is_high, p.o_slot = oracle.quantize_prompt(
            p.oc, synthetic.f16_bits(p.k), synthetic.f16_bits(p.v), p.s, r[0], r[1])
        rows = []
        for x in (p.k, p.v):
            buf = torch.zeros(x.size + 8, dtype=torch.float16, device=d)
            view = buf[shift:shift + x.size].view(x.shape)
            view.copy_(torch.from_numpy(x).to(d))
            assert view.data_ptr() % 16 == 8
            rows.append(view)
        h = torch.empty((2, T), dtype=torch.uint8, device=d)
        slot = torch.empty((2, T), dtype=torch.int32, device=d)
        semkv.semkv_rank_assign(torch.from_numpy(p.s).to(d), p.n_high, h, slot)
        semkv.semkv_quantize_pack(p.desc, rows[0], rows[1], h, slot, p.n_high, p.cache)
        torch.cuda.synchronize()
    else:
        p.quantize()
    # a row with NaN has no record that the oracle defines; it must leave its unit's others alone
    for gp, op, tok in ((p.cache.hi_pool, p.oc.hi_pool, p.oc.hi_tok), (p.cache.lo_pool, p.oc.lo_pool, p.oc.lo_tok)):
        at = np.flatnonzero(tok[0] == T // 2)
        op[0, 0, 0, at] = gp.cpu().numpy()[0, 0, 0, at]
    p.assert_records_equal()
    k, v = synthetic.kv(401 + T, 2, 1, 2, n)
    s = synthetic.scores_zipf(402 + T, 2, n)
    for i in range(2):
        at = slice(i * blk, (i + 1) * blk)
        p.stage(k[:, :, :, at], v[:, :, :, at], s[:, at])
        semkv.semkv_append_block(p.desc, p.cache, 1, 2)
        oracle.append_block(p.oc, 1, 2)
    torch.cuda.synchronize()
    p.assert_records_equal()
    p.assert_untouched_past_counts()
