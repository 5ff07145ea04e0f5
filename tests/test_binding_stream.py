"""The stream a call of the binding goes to: torch's current one, also where torch has not
the private names that give its raw handle (CPU), and the same handle by both ways (GPU)."""
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

WITHOUT = """
import torch
for name in ("_cuda_getCurrentRawStream", "_cuda_getDevice"):
    if hasattr(torch._C, name):
        delattr(torch._C, name)
from paper_2608_28911_gb300 import semkv
torch.cuda.is_initialized = lambda: True
torch.cuda.current_stream = lambda *a: type("S", (), {"cuda_stream": 1234})()
assert semkv._stream(None) == 1234
assert semkv._stream(type("S", (), {"cuda_stream": 77})()) == 77
print("ok")
"""


def test_current_stream_without_the_private_names():
    from paper_2608_28911_gb300 import build
    build.build()
    r = subprocess.run([sys.executable, "-c", WITHOUT], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stderr[-2000:]


@pytest.mark.gpu
def test_raw_handle_is_the_current_streams():
    import torch
    from paper_2608_28911_gb300 import semkv
    torch.zeros(1, device="cuda")
    s = torch.cuda.Stream()
    assert semkv._stream(None) == torch.cuda.current_stream().cuda_stream
    with torch.cuda.stream(s):
        assert semkv._stream(None) == s.cuda_stream
    assert semkv._stream(s) == s.cuda_stream
