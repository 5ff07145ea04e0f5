"""Kernels launched as programmatic dependents may start while the kernel before them on the
stream still runs, so they read nothing that earlier work wrote before their wait.  On the
CPU: between a kernel's start and its pdl_wait() the source reads through no pointer of its
arguments.  On the GPU: codebooks that a kernel writes right before the call are the
ones used."""
import math
import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2608_28911_gb300", "csrc")


def _read(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def _kernels(text):
    """(name, body) of every __global__ function."""
    for m in re.finditer(r"__global__\s+void\b[^{;]*?(\w+)\s*\((?:const\s+__grid_constant__\s+)?\w+Args a[^)]*\)\s*\{", text):
        depth, i = 1, m.end()
        while depth:
            depth += {"{": 1, "}": -1}.get(text[i], 0)
            i += 1
        yield m.group(1), text[m.end():i - 1]


def _before_wait(body):
    """The text that runs before the kernel's wait: up to the first pdl_wait() outside any
    nested block, without the blocks that wait for themselves."""
    out, i, depth, start = "", 0, 0, 0
    while i < len(body):
        if depth == 0 and body.startswith("pdl_wait();", i):
            return out
        if body[i] == "{":
            if depth == 0:
                start = i
            depth += 1
        elif body[i] == "}":
            depth -= 1
            if depth == 0:
                block = body[start:i + 1]
                out += block[:block.index("pdl_wait();")] if "pdl_wait();" in block else block
        elif depth == 0:
            out += body[i]
        i += 1
    return out


def _pointer_fields():
    return set(re.findall(r"^\s*(?:const\s+)?\w+\s*\*\s*(\w+)\s*(?:=\s*nullptr)?;", _read("kernels.h"), re.M))


def _reads(text, fields):
    """Pointers of the arguments, or aliases of them, that the text indexes or dereferences."""
    names = {rf"a\.{f}": f for f in fields}
    for alias, f in re.findall(r"\*\s*(\w+)\s*=\s*a\.(\w+)", text):
        if f in fields:
            names[alias] = f
    return {f for n, f in names.items()
            if re.search(rf"\b{n}\b\s*\)?\s*\[", text) or re.search(rf"(?:[=(,?:!]\s*\*|__ldg\()\s*\(?{n}\b", text)}


def test_nothing_is_read_before_the_wait():
    fields = _pointer_fields()
    assert {"cb_hi", "thr_lo", "signs", "q", "scores", "hi_tok"} <= fields
    seen, early = set(), {}
    for name in sorted(f for f in os.listdir(CSRC) if f.endswith(".cu")):
        for kernel, body in _kernels(_read(name)):
            if "pdl_wait();" not in body:
                continue
            seen.add(kernel)
            used = _reads(_before_wait(body), fields)
            if used:
                early[kernel] = sorted(used)
    assert not early
    assert {"decode_affine_kernel", "decode_affine_fast_kernel", "decode_tq_kernel", "scatter_tok_kernel",
            "quantize_affine_kernel", "quantize_rows_kernel", "rank_small_kernel",
            "rank_cluster_kernel", "score_kv_norm_kernel"} <= seen


@pytest.mark.gpu
@pytest.mark.parametrize("levels", [(4, 3), (5, 2)])
def test_codebooks_written_right_before_the_call(levels):
    import torch
    from paper_2608_28911_gb300 import synthetic
    from parity import Pair
    p = Pair(1, levels[0], levels[1], 1, 1, 2, 8, 3000, 1, 2, seed=950)
    tables = p.desc._keep[1:]
    good = [t.clone() for t in tables]
    p.quantize()
    p.assert_records_equal()
    ref, _ = p.decode(0)
    pools = [p.cache.hi_pool.clone(), p.cache.lo_pool.clone()]
    k, v = torch.from_numpy(p.k).to(p.dev), torch.from_numpy(p.v).to(p.dev)
    q = torch.from_numpy(synthetic.queries(p.seed, 1, 8)).to(p.dev)
    out = torch.empty((1, 8, 128), dtype=torch.float32, device=p.dev)
    ws = p.cache.workspace()
    for _ in range(5):
        for t, g in zip(tables, good):
            t.zero_()
            torch.add(g, 0.0, out=t)
        p.semkv.semkv_quantize_pack(p.desc, k, v, p.is_high, p.slot, p.n_high, p.cache)
        for t, g in zip(tables, good):
            t.zero_()
            torch.add(g, 0.0, out=t)
        p.semkv.semkv_decode_attention(p.desc, p.cache, 0, q, out, 1.0 / math.sqrt(128), ws)
        torch.cuda.synchronize()
        assert torch.equal(p.cache.hi_pool, pools[0]) and torch.equal(p.cache.lo_pool, pools[1])
        assert (out.cpu().numpy() == ref).all()
