"""The projection's wait limit bounds single waits, not the run of the whole persistent kernel."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def test_a_call_longer_than_the_wait_limit_reports_no_timeout():
    """65536 tokens of 4096 features to 12288 columns: 3.4 ms at least, in tiles of some 20 us each.  With a
    limit of 1 ms a wait no wait runs out."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    code = (
        "import torch, paper_2606_07713_gb300 as p\n"
        "x = torch.randn(1, 65536, 4096, device='cuda', dtype=torch.bfloat16)\n"
        "w = torch.randn(4096, 12288, device='cuda', dtype=torch.bfloat16) / 64\n"
        "p.qkv_proj(x, w, 32, 128, 128)\n"
        "a = p.get_device_status()\n"
        "e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]\n"
        "e[0].record(); p.qkv_proj(x, w, 32, 128, 128); e[1].record()\n"
        "b = p.get_device_status()\n"
        "print('status', a, b, 'long' if e[0].elapsed_time(e[1]) > 2.0 else 'short')\n")
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    env = dict(os.environ, MOA_WAIT_LIMIT_NS="1000000", PYTHONPATH=root)
    r = subprocess.run([sys.executable, "-c", code], env=env, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    assert "status 0 0 long" in r.stdout, r.stdout
