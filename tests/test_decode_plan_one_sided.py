"""The decode work plan (host logic of decode.cu) over caches whose tokens are all in one
pool, from one (sequence, KV head) pair up: tests/plan_one_sided.cu includes decode.cu and
checks make_decode_plan on the CPU; no GPU is used.
"""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


def test_one_sided_plans_cover_every_tile_inside_the_stride(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    exe = str(tmp_path / "plan_one_sided")
    cmd = [nvcc, "-std=c++17", "-O1", "--expt-relaxed-constexpr",
           "-gencode", "arch=compute_103a,code=sm_103a",
           "-I", os.path.join(ROOT, "include"),
           "-I", os.path.join(ROOT, "paper_2608_28911_gb300", "csrc"),
           os.path.join(HERE, "plan_one_sided.cu"), "-o", exe]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    r = subprocess.run([exe], capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stdout[-3000:]
    assert "all plans ok" in r.stdout
