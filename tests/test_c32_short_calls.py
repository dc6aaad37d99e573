"""complex32 short calls run one signal per thread group (N = 256, 1024, 2048):
the two-signals-per-thread kernels have a longer chain and had made them slower.
Both store the same bits."""
import pytest
import torch

pytestmark = pytest.mark.gpu

import paper_2203_09384_gb300 as gb  # noqa: E402

# n: the one-signal row, a two-signal row, elements up to which the first is the default
ROWS = {256: (6, 5, 5 << 19), 1024: (9, 8, 19 << 15), 2048: (9, 8, 7 << 16)}


@pytest.mark.parametrize("n", sorted(ROWS))
def test_default_by_size(n):
    direct, _, most = ROWS[n]
    for batch, short in ((1, True), (most // n, True), (most // n + 1, False)):
        plan = gb.Plan(n, batch, dtype="c32")
        assert (plan.info().variant == direct) == short
        assert (plan.info().pipeline == 0) == short
        plan.close()


@pytest.mark.parametrize("inverse", [False, True])
@pytest.mark.parametrize("n", sorted(ROWS))
def test_bit_for_bit_the_two_signal_kernels(n, inverse):
    direct, pair, most = ROWS[n]
    for batch in (1, 2, 3, 5, 152 * 4 + 3, most // n):
        g = torch.Generator(device="cuda").manual_seed(batch)
        h = (torch.randn(batch, n, 2, generator=g, device="cuda") * 900).half()
        h[0] = 0  # a zero signal
        if batch > 4:
            h[1] = torch.randint(-1, 2, (n, 2), generator=g, device="cuda").half() * 32768  # sums at powers of two
            h[2] *= 2.0 ** -18  # subnormal
            h[3, 5, 0], h[4, 7, 1] = float("inf"), float("nan")
        e = torch.randint(-128, 128, (batch,), generator=g, device="cuda").to(torch.int8)
        got = []
        for v in (direct, pair):
            plan = gb.Plan(n, batch, inverse=inverse, dtype="c32", variant=v)
            y, f = plan.execute_c32(torch.view_as_complex(h), e)
            assert plan.error() == 0
            plan.close()
            got.append((torch.view_as_real(y).clone(), f))
        bits = [y.view(torch.int16) for y, _ in got]
        same = (bits[0] == bits[1]) | (torch.isnan(got[0][0]) & torch.isnan(got[1][0]))  # a NaN's payload is free
        assert bool(same.all()), (n, batch, torch.nonzero(~same)[:4].tolist())
        assert torch.equal(got[0][1], got[1][1])
