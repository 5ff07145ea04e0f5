"""The work a user of the packed KV cache has it do, as measured cases.

Four kinds of call sequences, each through the Python binding of the C ABI:

  decode  one token's attention over a cache that is already packed, every layer once
  step    a generation step that closes a block: append the staged tokens, then decode
  prompt  Algorithm 1 on a prompt: value-norm scores, top-r selection, quantize and pack
  fake    the quality protocol: quantize every row and reconstruct it to fp16

K, V and queries are fp16 N(0,1) with four outlier channels per (layer, KV head) scaled by
8; scores are Zipf(1.1) integers, whose many ties are what the selection meets.
"""
import math

import numpy as np
import torch

from paper_2608_28911_gb300 import semkv

D = 128
SCALE = 1.0 / math.sqrt(D)
BLOCK = 128
AFFINE, TQ, AFFINE_HAD, TQ_DENSE = 0, 1, 2, 3


def _case(name, kind, base, levels, B, T, H=8, G=4, layers=1, r=(26, 100), staged=0):
    return {"name": name, "kind": kind, "base": base, "hi": levels[0], "lo": levels[1],
            "batch": B, "tokens": T, "kv_heads": H, "group": G, "layers": layers,
            "r_num": r[0], "r_den": r[1], "staged": staged}


def listed():
    return [
        # a single chat session early on: short context, part of a block still in fp16
        _case("decode-4k-staged", "decode", AFFINE, (6, 5), 1, 4096, staged=77),
        # one session at 32K: the whole cache is 22 MB, launches and merges count
        _case("decode-32k", "decode", AFFINE, (6, 5), 1, 32768),
        # a serving batch at long context, one layer: the throughput case
        _case("decode-16x64k", "decode", AFFINE, (6, 5), 16, 65536),
        # one token through all 32 layers of an 8B model at 128K
        _case("decode-32layers-128k", "decode", AFFINE, (6, 5), 1, 131072, layers=32),
        # the TurboQuant-MSE base at its published operating point, r = 75%
        _case("decode-tq-32k", "decode", TQ, (4, 3), 1, 32768, r=(3, 4)),
        # a batch of ragged length on the rotated affine base
        _case("decode-rotated-8x16k", "decode", AFFINE_HAD, (6, 5), 8, 16411),
        # a uniform grid point on a model with eight query heads per KV head
        _case("decode-uniform4-g8", "decode", AFFINE, (4, 4), 2, 12345, G=8, r=(0, 1)),
        # the generation step of a batch at which every sequence's block is full
        _case("step-16x16k", "step", AFFINE, (6, 5), 16, 16384, staged=BLOCK),
        # prompts of a batch, the main base: the largest prefill
        _case("prompt-4x64k", "prompt", AFFINE, (6, 5), 4, 65536),
        # one prompt on the TurboQuant-MSE base
        _case("prompt-tq-32k", "prompt", TQ, (4, 3), 1, 32768, r=(3, 4)),
        # ragged prompts of a small batch on the rotated affine base
        _case("prompt-rotated-3x20k", "prompt", AFFINE_HAD, (6, 5), 3, 20011),
        # the quality protocol over four layers on the rotated affine base
        _case("fake-rotated-4layers", "fake", AFFINE_HAD, (6, 5), 1, 16384, layers=4),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["decode", "decode", "decode", "step", "prompt", "prompt", "fake"])
    base = rng.choice([AFFINE, AFFINE, AFFINE, TQ, AFFINE_HAD, TQ_DENSE])
    if kind == "fake" and base == TQ_DENSE:
        base = TQ  # fake quantization has no dense rotation
    if base in (TQ, TQ_DENSE):
        levels, r = rng.choice([((4, 3), (3, 4)), ((4, 3), (26, 100)), ((4, 4), (0, 1)), ((3, 2), (1, 2))])
    else:
        levels, r = rng.choice([((6, 5), (26, 100)), ((6, 5), (26, 100)), ((6, 5), (35, 100)),
                                ((5, 5), (0, 1)), ((8, 7), (1, 4)), ((4, 3), (1, 2))])
    B = _log_int(rng, 1, 16)
    H = rng.choice([1, 2, 4, 8, 8])
    G = rng.choice([1, 2, 4, 4, 4, 8])
    T = _log_int(rng, 512, 65536)
    layers = rng.choice([1, 1, 1, 2, 4])
    while B * layers * H * T > 8 * 8 * 65536:  # no dearer than the largest listed case
        if B > 1:
            B = (B + 1) // 2
        elif layers > 1:
            layers //= 2
        else:
            break
    staged = {"decode": rng.choice([0, rng.randint(1, BLOCK - 1)]), "step": BLOCK}.get(kind, 0)
    c = _case("", kind, base, levels, B, T, H, G, layers, r, staged)
    del c["name"]
    return c


# ------------------------------------------------------------------ inputs ------

def _gen(seed, stream, layer=0):
    g = torch.Generator(device="cuda")
    g.manual_seed((seed * 1009 + stream) * 4099 + layer)
    return g


def _kv_layer(c, seed, layer, T, stream=0):
    """K and V of one layer: fp16 [B][H][T][128]."""
    B, H = c["batch"], c["kv_heads"]
    g = _gen(seed, 1 + stream, layer)
    gain = torch.ones((2, 1, H, 1, D), device="cuda")
    idx = torch.rand((H, D), generator=g, device="cuda").argsort(dim=1)[:, :4]
    gain.view(2, H, D).scatter_(2, idx.expand(2, H, 4), 8.0)
    out = []
    for r in range(2):
        x = torch.randn((B, H, T, D), generator=g, device="cuda")
        out.append(x.mul_(gain[r]).half())
    return out


def _kv(c, seed, T, stream=0):
    B, NL, H = c["batch"], c["layers"], c["kv_heads"]
    k = torch.empty((B, NL, H, T, D), dtype=torch.float16, device="cuda")
    v = torch.empty_like(k)
    for l in range(NL):
        k[:, l], v[:, l] = _kv_layer(c, seed, l, T, stream)
    return k, v


def _zipf(c, seed, n, stream):
    r = np.random.default_rng([seed, stream])
    return r.zipf(1.1, size=(c["batch"], n)).astype(np.float32)


def _n_high(c, n):
    return n * c["r_num"] // c["r_den"]


def _block_high(c, n):
    return (2 * c["r_num"] * n + c["r_den"]) // (2 * c["r_den"])


def _signs(c, seed):
    g = _gen(seed, 11)
    return (torch.randint(0, 2, (c["layers"], c["kv_heads"], D), generator=g, device="cuda") * 2 - 1).to(torch.int8)


def _rotations(c, seed):
    g = _gen(seed, 12)
    x = torch.randn((c["layers"], c["kv_heads"], D, D), generator=g, device="cuda", dtype=torch.float64)
    q, r = torch.linalg.qr(x)
    q = q * torch.where(torch.diagonal(r, dim1=-2, dim2=-1) < 0, -1.0, 1.0)[..., None, :]
    return (math.sqrt(D) * q).half().cpu().numpy()


def _queries(c, seed):
    g = _gen(seed, 13)
    shape = (c["layers"], c["batch"], c["kv_heads"] * c["group"], D)
    return torch.randn(shape, generator=g, device="cuda").half()


def _desc(c, seed):
    b = c["base"]
    signs = _signs(c, seed).cpu() if b in (TQ, AFFINE_HAD) else None
    rot = _rotations(c, seed) if b == TQ_DENSE else None
    return semkv.QuantDesc(b, c["hi"], c["lo"], signs=signs, rotation=rot)


def _new_cache(c, desc, T, extra=0):
    n = _n_high(c, T)
    return semkv.KVCache(desc, c["batch"], c["layers"], c["kv_heads"], c["kv_heads"] * c["group"],
                         hi_cap=n + extra, lo_cap=T - n + extra, block=BLOCK)


def prepare(case, seed):
    c, T = case, case["tokens"]
    st = {"case": c, "desc": _desc(c, seed)}
    flags = dict(dtype=torch.uint8, device="cuda")
    ints = dict(dtype=torch.int32, device="cuda")
    if c["kind"] == "fake":
        st["k"], st["v"] = _kv(c, seed, T)
        st["k_out"], st["v_out"] = torch.empty_like(st["k"]), torch.empty_like(st["v"])
        st["is_high"] = torch.from_numpy(_fake_flags(c, seed)).cuda()
        return st
    st["n_high"] = _n_high(c, T)
    st["is_high"] = torch.empty((c["batch"], T), **flags)
    st["slot"] = torch.empty((c["batch"], T), **ints)
    st["cache"] = _new_cache(c, st["desc"], T, BLOCK if c["kind"] == "step" else 0)
    if c["kind"] == "prompt":
        st["k"], st["v"] = _kv(c, seed, T)
        st["scores"] = torch.empty((c["batch"], T), dtype=torch.float32, device="cuda")
        return st
    scores = torch.from_numpy(_zipf(c, seed, T, 21)).cuda()
    semkv.semkv_rank_assign(scores, st["n_high"], st["is_high"], st["slot"])
    k, v = _kv(c, seed, T)
    cache = st["cache"]
    semkv.semkv_quantize_pack(st["desc"], k, v, st["is_high"], st["slot"], st["n_high"], cache)
    del k, v
    n = c["staged"]
    if n:
        sk, sv = _kv(c, seed, n, stream=2)
        cache.stage_k[:, :, :, :n] = sk
        cache.stage_v[:, :, :, :n] = sv
        cache.stage_score[:, :n] = torch.from_numpy(_zipf(c, seed, n, 22)).cuda()
        cache.s.stage_n = n
    st["q"] = _queries(c, seed)
    st["out"] = torch.empty(st["q"].shape, dtype=torch.float32, device="cuda")
    st["ws"] = cache.workspace()
    return st


# -------------------------------------------------------------------- run -------

def run(state):
    c, desc = state["case"], state["desc"]
    if c["kind"] == "fake":
        semkv.semkv_fake_quant(desc, state["k"], state["v"], state["k_out"], state["v_out"],
                               state["is_high"])
        return {"k": state["k_out"], "v": state["v_out"]}
    cache = state["cache"]
    if c["kind"] == "prompt":
        semkv.semkv_score_kv_norm(state["v"], state["scores"])
        semkv.semkv_rank_assign(state["scores"], state["n_high"], state["is_high"], state["slot"])
        semkv.semkv_quantize_pack(desc, state["k"], state["v"], state["is_high"], state["slot"],
                                  state["n_high"], cache)
        return {"scores": state["scores"], "is_high": state["is_high"], "slot": state["slot"],
                "hi_pool": cache.hi_pool, "lo_pool": cache.lo_pool,
                "hi_tok": cache.hi_tok, "lo_tok": cache.lo_tok}
    outs = {}
    if c["kind"] == "step":
        # the block's slots are taken again on every pass
        cache.s.hi_count = state["n_high"]
        cache.s.lo_count = c["tokens"] - state["n_high"]
        cache.s.n_tokens = c["tokens"]
        cache.s.stage_n = c["staged"]
        semkv.semkv_append_block(desc, cache, c["r_num"], c["r_den"])
        outs = {"hi_pool": cache.hi_pool, "lo_pool": cache.lo_pool, "hi_tok": cache.hi_tok,
                "lo_tok": cache.lo_tok}
    q, out, ws = state["q"], state["out"], state["ws"]
    for l in range(c["layers"]):
        semkv.semkv_decode_attention(desc, cache, l, q[l], out[l], SCALE, ws)
    outs["out"] = out
    return outs


# ------------------------------------------------------------------- work -------

_ROW = {2: 16, 3: 26, 4: 32, 5: 38, 6: 42, 7: 48, 8: 48}


def work(case):
    c, T = case, case["tokens"]
    par = 4 if c["base"] in (TQ, TQ_DENSE) else 8
    rec = {"hi": 2 * _ROW[c["hi"]] + par, "lo": 2 * _ROW[c["lo"]] + par}
    rows = c["batch"] * c["layers"] * c["kv_heads"]
    heads = rows * c["group"]
    n = _n_high(c, T)
    packed = rows * (n * rec["hi"] + (T - n) * rec["lo"])
    rotate = 2 * D * 7 if c["base"] in (TQ, AFFINE_HAD) else 2 * D * D if c["base"] == TQ_DENSE else 0
    if c["kind"] == "fake":
        return {"bytes": 2 * rows * T * 2 * D * 2 + c["batch"] * T,
                "flops": 2 * rows * T * (2 * rotate / 2 + 8 * D)}
    if c["kind"] == "prompt":
        return {"bytes": 2 * rows * T * D * 2 + packed + c["batch"] * T * (4 + 1 + 4 + 4),
                "flops": 2 * rows * T * (rotate / 2 + 6 * D) + 2 * rows * T * D}
    m = c["staged"]
    moved, tokens = packed + heads * D * (2 + 4), T + m
    if c["kind"] == "step":
        h = _block_high(c, m)
        new = rows * (h * rec["hi"] + (m - h) * rec["lo"])
        moved += 2 * rows * m * D * 2 + new + c["batch"] * m * (4 + 4)
    else:
        moved += 2 * rows * m * D * 2
    return {"bytes": moved, "flops": 4 * heads * tokens * D}


# ---------------------------------------------------------- 64-bit results ------
# Codes are what the record format says they are: binary32 arithmetic on fp16 rows.  What
# is computed from the codes (attention, reconstruction) is taken in 64 bits.

def _fwht(x):
    h = 1
    while h < D:
        y = x.view(*x.shape[:-1], D // (2 * h), 2, h)
        a, b = y[..., 0, :], y[..., 1, :]
        x = torch.stack((a + b, a - b), dim=-2).view(x.shape)
        h *= 2
    return x


def _param(x):
    return x.half().clamp(-65504, 65504)


def _floor16(x):
    """fp16 rounded toward minus infinity, at least -65504."""
    h = x.half()
    up = h.float() > x
    bits = h.view(torch.int16)
    down = torch.where(h > 0, bits - 1, torch.where(h < 0, bits + 1, torch.full_like(bits, -32767)))
    return torch.where(up, down.view(torch.float16), h).clamp(min=-65504)


def _codebook(L):
    erf, c = math.erf, [2.0 * (-1.0 + 2.0 * (i + 0.5) / L) for i in range(L)]
    pdf = lambda x: math.exp(-0.5 * x * x) / math.sqrt(2 * math.pi) if math.isfinite(x) else 0.0  # noqa: E731
    cdf = lambda x: 0.5 * (1.0 + erf(x / math.sqrt(2))) if math.isfinite(x) else float(x > 0)  # noqa: E731
    for _ in range(20000):
        t = [-math.inf] + [0.5 * (a + b) for a, b in zip(c, c[1:])] + [math.inf]
        new = [(pdf(t[i]) - pdf(t[i + 1])) / (cdf(t[i + 1]) - cdf(t[i])) for i in range(L)]
        moved = max(abs(a - b) for a, b in zip(new, c))
        c = new
        if moved < 1e-15:
            break
    c = [0.5 * (a - b) for a, b in zip(c, reversed(c))]
    thr = [0.5 * (a + b) for a, b in zip(c, c[1:])]
    return (torch.tensor(c, dtype=torch.float32, device="cuda"),
            torch.tensor(thr, dtype=torch.float32, device="cuda"))


def _dequant(x, L, base, sign):
    """Rows x [T][128] fp16 at L levels, as the 64-bit values their records stand for."""
    f = x.float()
    if base == TQ:
        f = f * sign.float()
        p = f.view(-1, 32, 4).square()
        p = ((p[..., 0] + p[..., 1]) + p[..., 2]) + p[..., 3]
        for off in (16, 8, 4, 2, 1):
            p = p[:, :off] + p[:, off:2 * off]
        n = _param(p[:, 0].sqrt()).float()
        inv = torch.where(n != 0, 1.0 / n, torch.zeros_like(n))
        u = _fwht(f) * inv[:, None]
        cb, thr = _codebook(L)
        code = (u[..., None] > thr).sum(-1)
        code = torch.where(n[:, None] != 0, code, torch.zeros_like(code))
        y = cb.double()[code] * (n.double() / D)[:, None]
        return _fwht(y) * sign.double()
    if base == AFFINE_HAD:
        f = _fwht(f * sign.float()) * torch.tensor(float.fromhex("0x1.6a09e6p-4"), device="cuda")
    mn, mx = f.amin(1), f.amax(1)
    z = _floor16(mn) if base == AFFINE_HAD else mn.half()
    z = torch.where(z == 0, torch.zeros_like(z), z)
    s = _param((mx - (z.float() if base == AFFINE_HAD else mn)) / (L - 1))
    inv = torch.where(s.float() > 0, 1.0 / s.float(), torch.zeros_like(mn))
    code = ((f - z.float()[:, None]) * inv[:, None]).round().clamp(0, L - 1)
    y = z.double()[:, None] + s.double()[:, None] * code.double()
    if base == AFFINE_HAD:
        y = _fwht(y) * sign.double() / math.sqrt(D)
    return y


def _top(scores, n):
    """Flags of the n largest of each row, ties to the lower index."""
    order = np.argsort(-scores, axis=1, kind="stable")[:, :n]
    flags = np.zeros(scores.shape, np.uint8)
    np.put_along_axis(flags, order, 1, axis=1)
    return flags


def _fake_flags(c, seed):
    return _top(_zipf(c, seed, c["tokens"], 21), _n_high(c, c["tokens"]))


def _rows64(c, x, high, sign):
    """Rows x [T][128] fp16, each at its token's level count, as 64-bit values."""
    y = torch.empty(x.shape, dtype=torch.float64, device="cuda")
    for L, sel in ((c["hi"], high), (c["lo"], ~high)):
        if bool(sel.any()):
            y[sel] = _dequant(x[sel], L, c["base"], sign)
    return y


def exact(case, seed):
    c, T = case, case["tokens"]
    B, NL, H, G, m = c["batch"], c["layers"], c["kv_heads"], c["group"], c["staged"]
    if c["base"] == TQ_DENSE and c["kind"] != "prompt":
        return None  # its codes come from a product on the tensor cores
    if c["kind"] == "prompt":
        total = torch.zeros((B, T), dtype=torch.float64, device="cuda")
        for l in range(NL):
            v = _kv_layer(c, seed, l, T)[1]
            for h in range(H):
                total += v[:, h].double().square().sum(-1)
        return {"scores": total.sqrt(), "is_high": None, "slot": None, "hi_pool": None,
                "lo_pool": None, "hi_tok": None, "lo_tok": None}
    signs = _signs(c, seed)
    high = torch.from_numpy(_top(_zipf(c, seed, T, 21), _n_high(c, T)).astype(bool)).cuda()
    if c["kind"] == "fake":
        out = {r: torch.empty((B, NL, H, T, D), dtype=torch.float64, device="cuda") for r in "kv"}
        for l in range(NL):
            for r, x in zip("kv", _kv_layer(c, seed, l, T)):
                for b in range(B):
                    for h in range(H):
                        out[r][b, l, h] = _rows64(c, x[b, h], high[b], signs[l, h])
        return out
    q = _queries(c, seed).double()
    out = torch.empty(q.shape, dtype=torch.float64, device="cuda")
    staged_high = (torch.from_numpy(_top(_zipf(c, seed, m, 22), _block_high(c, m)).astype(bool)).cuda()
                   if c["kind"] == "step" else None)
    for l in range(NL):
        k, v = _kv_layer(c, seed, l, T)
        if m:
            sk, sv = _kv_layer(c, seed, l, m, stream=2)
        for b in range(B):
            for h in range(H):
                rows = []
                for i, x in enumerate((k, v)):
                    y = _rows64(c, x[b, h], high[b], signs[l, h])
                    if m:
                        s = (sk, sv)[i][b, h]
                        y = torch.cat((y, _rows64(c, s, staged_high[b], signs[l, h])
                                       if staged_high is not None else s.double()))
                    rows.append(y)
                a = torch.softmax(q[l, b, h * G:(h + 1) * G] @ rows[0].T * SCALE, dim=1)
                out[l, b, h * G:(h + 1) * G] = a @ rows[1]
    outs = {"out": out}
    if c["kind"] == "step":
        outs.update(hi_pool=None, lo_pool=None, hi_tok=None, lo_tok=None)
    return outs
