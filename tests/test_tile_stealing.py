"""Schedules whose blocks take the tiles of unstarted blocks (CH bit 2): every
tile is transformed exactly once whatever the number of tiles per resident
block, a launch keeps no state another could meet, programmatic launches stay
in order, and a wait that gives up ends the whole grid at once."""
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

ROWS = [(1 << r[0], r[1]) for r in _rows("GBFFT_GENERIC_SCHEDULES", 13) if r[12] & 4] + \
       [(1 << r[0], r[1]) for r in _rows("GBFFT_SMALL_SCHEDULES", 5) if r[4] & 4]


def _plan(n, batch, v, **kw):
    return gb.Plan(n, batch, variant=v, dtype=gb.DTYPE_NAMES[gb.fft_variant_dtype(n, v)], **kw)


@pytest.mark.parametrize("n,variant", ROWS)
def test_every_tile_once(n, variant):
    probe = _plan(n, 1 << 22, variant)
    resident, s = probe.info().grid, probe.info().signals_per_block  # capped at the resident blocks
    probe.close()
    tol = FP32_TOL if gb.fft_variant_dtype(n, variant) == _abi.FFT_C64 else 5e-3
    for batch in sorted({1, s, s + 1, (resident - 1) * s + 1, resident * s + 1, 2 * resident * s,
                         3 * resident * s + s // 2 + 1}):
        x = synth.uniform(batch, n, seed=variant, device="cuda")
        guard = torch.full((batch + 3, n), 5.0, dtype=torch.complex64, device="cuda")
        p = _plan(n, batch, variant)
        p.execute(x, guard[:batch])
        torch.cuda.synchronize()
        assert p.error() == 0
        assert torch.all(guard[batch:] == 5.0)
        # every signal against the one-call FP32 schedule, sampled ones against the oracle
        ref = gb.Plan(n, batch, variant=1 if n <= 32 else None)
        y = ref.execute(x)
        far = (guard[:batch] - y).norm(dim=1) / y.norm(dim=1)
        assert float(far.max()) <= 2 * tol, (batch, int(far.argmax()))
        idx = torch.unique(torch.cat([torch.arange(min(batch, 16)), torch.arange(max(0, batch - 16), batch)]))
        assert max_rel_l2(to_np(guard[idx.cuda()]), oracle.reference(x[idx.cuda()].cpu().numpy())) <= tol
        p.close()
        ref.close()


C32_ROWS = [(1 << r[0], r[1]) for r in _rows("GBFFT_C32_SCHEDULES", 11) if r[10] & 15 == 14] + \
           [(1 << r[0], r[1]) for r in _rows("GBFFT_C32_SMALL_SCHEDULES", 5) if r[4] & 4]
C32_FIXED = {1 << r[0]: r[1] for r in _rows("GBFFT_C32_SCHEDULES", 11) if r[10] in (0, 6)}


@pytest.mark.parametrize("inverse", [False, True])
@pytest.mark.parametrize("n,variant", C32_ROWS)
def test_complex32_tiles_bit_for_bit(n, variant, inverse):
    """Against a fixed-stride row of the same arithmetic (N <= 32: the direct
    kernel splits the length, so there the results agree to one stored ulp)."""
    probe = _plan(n, 1 << 22, variant)
    resident, s = probe.info().grid, probe.info().signals_per_block
    probe.close()
    for batch in (1, s + 1, resident * s - 1, 2 * resident * s + 3, 5 * resident * s + s // 2):
        g = torch.Generator(device="cuda").manual_seed(batch)
        x = (torch.randn(batch, n, 2, generator=g, device="cuda") * 700).half()
        e = torch.randint(-20, 20, (batch,), generator=g, device="cuda").to(torch.int8)
        got = []
        for v in (variant, C32_FIXED[n]):
            y, f = torch.full_like(x, 3.0), torch.full_like(e, 77)
            p = _plan(n, batch, v, inverse=inverse)
            p.execute_c32(torch.view_as_complex(x), e, torch.view_as_complex(y), f)
            assert p.error() == 0
            p.close()
            got.append((y, f))
        if n > 32:
            assert torch.equal(got[0][0].view(torch.int16), got[1][0].view(torch.int16))
            assert torch.equal(got[0][1], got[1][1])
        else:
            d = [y.double() * torch.pow(2.0, f.double())[:, None, None] for y, f in got]
            top = d[1].abs().amax(dim=(1, 2), keepdim=True)
            assert float(((d[0] - d[1]).abs() / top).max()) <= 2.0 ** -10


@pytest.mark.parametrize("n,variant", [(8, 0), (64, 0), (512, 0), (2048, 0), (2048, 22)])
def test_launches_share_nothing_and_stay_in_order(n, variant):
    batch = (1 << 23) // n + 7
    x = synth.uniform(batch, n, seed=3, device="cuda")
    fwd, inv = _plan(n, batch, variant), _plan(n, batch, variant, inverse=True)
    want = fwd.execute(x)
    a, b, c = x.clone(), torch.empty_like(x), torch.empty_like(x)
    s1, s2 = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    for _ in range(4):  # the same plan on two streams at once
        fwd.execute(x, b, stream=s1)
        fwd.execute(x, c, stream=s2)
    for _ in range(6):  # in place, each launch reading the one before it
        fwd.execute(a, a)
        inv.execute(a, a)
    torch.cuda.synchronize()
    assert fwd.error() == 0 and inv.error() == 0
    assert torch.equal(b, want) and torch.equal(c, want)
    tol = 12 * (FP32_TOL if gb.fft_variant_dtype(n, variant) == _abi.FFT_C64 else 5e-3)
    assert float(((a - x).norm(dim=1) / x.norm(dim=1)).max()) <= tol
    fwd.close()
    inv.close()


@pytest.mark.parametrize("n,variant", [(64, 7), (256, 24), (2048, 23)])
def test_a_stalled_complex32_grid_ends_after_one_wait(n, variant):
    batch = (1 << 26) // n
    x = torch.zeros(batch, n, 2, dtype=torch.float16, device="cuda")
    e = torch.zeros(batch, dtype=torch.int8, device="cuda")
    y, f = torch.full_like(x, 3.0), torch.full_like(e, 77)
    plan = _plan(n, batch, variant, extra_flags=gb.FFT_FLAG_TEST_STALL)
    plan.set_wait_limit(100_000_000)
    t0 = time.perf_counter()
    plan.execute_c32(torch.view_as_complex(x), e, torch.view_as_complex(y), f)
    assert plan.error() == _abi.STATUS_CODE["FFT_ERR_TIMEOUT"]
    assert time.perf_counter() - t0 < 3.0
    assert torch.all(y == 3.0) and torch.all(f == 77)
    plan.close()


@pytest.mark.parametrize("n,variant", [(64, 0), (512, 0), (2048, 0), (256, 20), (1024, 18)])
def test_a_stalled_grid_ends_after_one_wait(n, variant):
    batch = (1 << 26) // n  # many tiles per resident block
    x = synth.uniform(batch, n, seed=1, device="cuda")
    out = torch.zeros_like(x)
    plan = _plan(n, batch, variant, extra_flags=gb.FFT_FLAG_TEST_STALL)
    plan.set_wait_limit(100_000_000)  # 0.1 s: with one wait per tile this would take tens of seconds
    t0 = time.perf_counter()
    plan.execute(x, out)
    assert plan.error() == _abi.STATUS_CODE["FFT_ERR_TIMEOUT"]
    assert time.perf_counter() - t0 < 3.0
    assert plan.error() == 0
    assert torch.count_nonzero(out) == 0
    plan.close()
    good = _plan(n, 999, variant)
    y = good.execute(x[:999])
    assert good.error() == 0
    tol = FP32_TOL if gb.fft_variant_dtype(n, variant) == _abi.FFT_C64 else 5e-3
    assert max_rel_l2(to_np(y[:64]), oracle.reference(x[:64].cpu().numpy())) <= tol
    good.close()
