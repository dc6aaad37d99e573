"""The one-thread-per-signal kernels that take the tiles of unstarted blocks
wait on the device for each answer, so the stall test mode applies to them: the
wait runs out, the error word says so, nothing is stored, the whole grid ends
after one wait, and the device goes on working."""
import time

import pytest
import torch

import oracle
import synth
from tests.helpers import FP32_TOL, max_rel_l2, to_np
from tests.test_bank_model import _rows

pytestmark = pytest.mark.gpu

import paper_2203_09384_gb300 as gb  # noqa: E402
from paper_2203_09384_gb300 import _abi  # noqa: E402

TIMEOUT = _abi.STATUS_CODE["FFT_ERR_TIMEOUT"]


@pytest.mark.parametrize("n,variant", [(1 << r[0], r[1]) for r in _rows("GBFFT_SMALL_SCHEDULES", 5) if r[4] & 4])
def test_complex64(n, variant):
    batch = (1 << 25) // n + 1  # many tiles per resident block
    x = synth.uniform(batch, n, seed=n, device="cuda")
    out = torch.zeros_like(x)
    plan = gb.Plan(n, batch, variant=variant, extra_flags=gb.FFT_FLAG_TEST_STALL)
    plan.set_wait_limit(100_000_000)  # 0.1 s
    t0 = time.perf_counter()
    plan.execute(x, out)
    assert plan.error() == TIMEOUT
    assert time.perf_counter() - t0 < 3.0
    assert plan.error() == 0
    assert torch.count_nonzero(out) == 0
    plan.close()
    plan = gb.Plan(n, batch, variant=variant)
    plan.execute(x, out)
    assert plan.error() == 0
    assert max_rel_l2(to_np(out[:64]), oracle.reference(x[:64].cpu().numpy())) <= FP32_TOL
    plan.close()


@pytest.mark.parametrize("n,variant", [(1 << r[0], r[1]) for r in _rows("GBFFT_C32_SMALL_SCHEDULES", 5) if r[4] & 4])
def test_complex32(n, variant):
    batch = (1 << 26) // n + 1
    x = torch.ones(batch, 2 * n, dtype=torch.float16, device="cuda").view(torch.complex32)
    e = torch.zeros(batch, dtype=torch.int8, device="cuda")
    y, f = torch.full_like(x.view(torch.float16), 3.0), torch.full_like(e, 77)
    plan = gb.Plan(n, batch, dtype="c32", variant=variant, extra_flags=gb.FFT_FLAG_TEST_STALL)
    plan.set_wait_limit(100_000_000)
    t0 = time.perf_counter()
    plan.execute_c32(x, e, y.view(torch.complex32), f)
    assert plan.error() == TIMEOUT
    assert time.perf_counter() - t0 < 3.0
    assert torch.all(y == 3.0) and torch.all(f == 77)
    plan.close()
    plan = gb.Plan(n, batch, dtype="c32", variant=variant)
    plan.execute_c32(x, e, y.view(torch.complex32), f)
    assert plan.error() == 0
    # a constant signal 1 + i: n (1 + i) in bin 0, zeros elsewhere
    assert torch.all(y[:, :2] == 2.0 ** 14) and torch.count_nonzero(y[:, 2:]) == 0
    assert torch.all(f == n.bit_length() - 1 - 14)
    plan.close()
