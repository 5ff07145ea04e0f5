"""Which instance of the clustered top-r selection a call takes (host logic of rank.cu):
tests/rank_rule_check.cu includes rank.cu and checks the rule on the CPU.  On the GPU, both
instances on the two sides of the rule, against the oracle."""
import os
import shutil
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


def test_two_ctas_per_sm_only_where_they_fit(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    exe = str(tmp_path / "rank_rule_check")
    cmd = [nvcc, "-std=c++17", "-O1", "--expt-relaxed-constexpr",
           "-gencode", "arch=compute_103a,code=sm_103a",
           "-I", os.path.join(ROOT, "include"),
           "-I", os.path.join(ROOT, "paper_2608_28911_gb300", "csrc"),
           os.path.join(HERE, "rank_rule_check.cu"), "-o", exe]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "rule ok" in r.stdout, r.stdout


@pytest.mark.gpu
@pytest.mark.parametrize("B,T", [
    (17, 132576),   # the longest keys with which two CTAs fit an SM
    (17, 132584),   # eight tokens more: one CTA per SM
    (16, 9000),
])
def test_both_instances(B, T):
    import torch

    import oracle
    from paper_2608_28911_gb300 import semkv, synthetic
    s = synthetic.scores_zipf(60, B, T)
    h = torch.full((B, T), 7, dtype=torch.uint8, device="cuda")
    slot = torch.full((B, T), -1, dtype=torch.int32, device="cuda")
    semkv.semkv_rank_assign(torch.from_numpy(s).cuda(), T // 4, h, slot)
    torch.cuda.synchronize()
    want_h, want_slot = oracle.rank_assign(s, T // 4)[:2]
    assert np.array_equal(h.cpu().numpy(), want_h)
    assert np.array_equal(slot.cpu().numpy().astype(np.int64), np.asarray(want_slot, np.int64))
