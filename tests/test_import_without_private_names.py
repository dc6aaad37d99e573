"""The package imports on a build of torch without the private queries behind
torch.cuda's wrappers (a CPU-only build has none), and then uses the wrappers."""
import os
import subprocess
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

BODY = """
import torch
for name in ("_cuda_getDevice", "_cuda_getCurrentRawStream"):
    if hasattr(torch._C, name):
        delattr(torch._C, name)
import paper_2203_09384_gb300 as gb


class Stream:
    cuda_stream = 77


torch.cuda.current_stream = lambda index: Stream if index == 3 else None
gb._current_device = lambda: 3
gb._enqueue(3, None, lambda *a: print(*a), 5)
assert gb.fft_validate(64, 1) == 0
"""


def test_import_and_enqueue():
    r = subprocess.run([sys.executable, "-c", BODY], cwd=ROOT, capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr[-2000:]
    assert r.stdout.split() == ["5", "77"]
