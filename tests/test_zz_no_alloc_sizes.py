"""fft_execute_noalloc picks its kernel by the size of the call; the first call
of a length and direction sets up the kernels of every size, so a later call of
another batch takes no device memory (the code of a kernel is loaded on first
use) and needs no query under capture.  In a fresh process: nothing loaded."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

BODY = """
import torch
from paper_2203_09384_gb300 import _abi

elems = 1 << 24
x = torch.zeros(elems, dtype=torch.complex64, device="cuda")
y = torch.empty_like(x)
s = torch.cuda.Stream()
g = torch.cuda.CUDAGraph()


def call(n, batch, inverse):
    _abi.fft_execute_noalloc(n, batch, inverse, 0, x.data_ptr(), y.data_ptr(), s.cuda_stream)


lengths = [2 ** k for k in range(1, 12)]
for inverse in (0, 1):
    for n in lengths:
        call(n, 3, inverse)
torch.cuda.synchronize()
before = torch.cuda.mem_get_info()[0]
for inverse in (0, 1):
    for n in lengths:
        for le in (15, 16, 17, 18, 20, 20.7, 21.4, 22, 22.6, 23.2, 24):
            call(n, int(2 ** le) // n, inverse)
torch.cuda.synchronize()
taken = before - torch.cuda.mem_get_info()[0]
with torch.cuda.graph(g, stream=s):
    call(1024, elems // 1024, 0)
g.replay()
torch.cuda.synchronize()
print("taken", taken)
"""


def test_other_batch_sizes_take_no_device_memory():
    r = subprocess.run([sys.executable, "-c", BODY], cwd=ROOT, capture_output=True, text=True, timeout=600,
                       env={**os.environ, "GBFFT_TUNE_CACHE": "off"})
    assert r.returncode == 0, r.stderr[-2000:]
    assert r.stdout.split() == ["taken", "0"], r.stdout
