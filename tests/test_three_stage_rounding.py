"""Rounding of the FP32 three-stage schedules (N = 512, 1024, 2048).

With radix 16 first and last they run two radix-16 butterflies, whose constant
cos(pi/8) is off by half a unit in the last place; the butterfly with the
factored constants keeps their error below that of the radices [8,8,8],
[8,16,8] and [8,16,16], which took fewer radix-16 stages.
"""
import math
import os
import re

import numpy as np
import pytest
import torch

import oracle
import synth
from tests.helpers import to_np
from tests.test_bounded_waits import CSRC

# relative L2 error of those radices over 2^24 elements of uniform signals
LEAST = {512: 9.82e-8, 1024: 1.048e-7, 2048: 1.127e-7}


def test_the_factored_constants_are_exact_to_1e_10():
    with open(os.path.join(CSRC, "fft_device.cuh")) as f:
        text = f.read()
    g, a, b = (float(np.float32(re.search(rf"constexpr float {k} = ([\d.]+)f;", text).group(1)))
               for k in ("kG8", "kA8", "kB8"))
    assert abs(g * a / math.cos(math.pi / 8) - 1) < 1e-10
    assert abs(g * b / math.sin(math.pi / 8) - 1) < 1e-10


@pytest.mark.gpu
@pytest.mark.parametrize("ragged", [False, True])
@pytest.mark.parametrize("inverse", [False, True])
@pytest.mark.parametrize("n", sorted(LEAST))
def test_no_further_off_than_the_radices_replaced(n, inverse, ragged):
    import paper_2203_09384_gb300 as gb

    batch = (1 << 20) // n
    x = synth.uniform(batch, n, seed=n)
    if ragged:
        plan = gb.RaggedPlan([i * n for i in range(batch + 1)], inverse=inverse)
        y = plan.execute(x.cuda().view(-1)).view(batch, n)
        torch.cuda.synchronize()
        plan.close()
    else:
        y = gb.ifft(x.cuda()) if inverse else gb.fft(x.cuda())
    want = oracle.reference(x.numpy(), inverse, True, threads=8)
    assert np.linalg.norm(to_np(y) - want) / np.linalg.norm(want) <= LEAST[n]
