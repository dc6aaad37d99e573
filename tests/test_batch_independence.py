"""A signal's transform does not depend on how many others share its call: the
schedule follows the size of the call, but all defaults of a length take its
radices in one order and round alike, so the bits stay the same."""
import re

import pytest
import torch

import synth
from tests.test_bank_model import SCHEDULES, _rows

import paper_2203_09384_gb300 as gb

SIZES = [10, 16, 17.5, 19, 19.4, 20.2, 20.7, 21.2, 22.4, 22.8, 23.7]  # log2 of the elements: every line of the table


def test_default_rows_of_a_length_share_their_radix_order():
    """CPU: the FP32 rows that plans take by size, from the compiled table."""
    radices = {(r[0], r[1]): [x for x in r[4:8] if x] for r in _rows("GBFFT_GENERIC_SCHEDULES", 13)}
    with open(SCHEDULES) as f:
        lines = re.findall(r"\bDX\((\d+), 0, [^,]+, (\d+)\)", f.read())
    for log2n in range(6, 12):
        used = {0} | {int(v) for k, v in lines if int(k) == log2n}
        assert len(used) > 1
        assert len({tuple(radices[(log2n, v)]) for v in used}) == 1, (1 << log2n, {v: radices[(log2n, v)] for v in used})


@pytest.mark.gpu
@pytest.mark.parametrize("inverse", [False, True])
@pytest.mark.parametrize("n", [2 ** k for k in range(1, 12)])
def test_first_signals_of_every_batch_size(n, inverse):
    few = (1 << 10) // n + 1 if n <= 1024 else 2
    x = synth.uniform(int(2 ** SIZES[-1]) // n, n, seed=n, device="cuda")
    want = None
    for le in SIZES:
        batch = max(few, int(2 ** le) // n)
        plan = gb.Plan(n, batch, inverse=inverse)
        y = plan.execute(x[:batch])[:few]
        assert plan.error() == 0
        want = y if want is None else want
        assert torch.equal(y, want), (n, le, plan.info().variant)
        plan.close()


@pytest.mark.gpu
@pytest.mark.parametrize("n", [2 ** k for k in range(1, 12)])
def test_first_complex32_signals_of_every_batch_size(n):
    few = (1 << 10) // n + 1 if n <= 1024 else 2
    most = int(2 ** 24.6) // n
    g = torch.Generator(device="cuda").manual_seed(n)
    x = torch.view_as_complex((torch.randn(most, n, 2, generator=g, device="cuda") * 700).half())
    e = torch.randint(-12, 13, (most,), generator=g, device="cuda").to(torch.int8)
    want = None
    for le in SIZES + [21.8, 22.1, 24.6]:
        batch = max(few, int(2 ** le) // n)
        plan = gb.Plan(n, batch, dtype="c32")
        y, f = plan.execute_c32(x[:batch], e[:batch])
        assert plan.error() == 0
        got = (y[:few].view(torch.int16).clone(), f[:few].clone())
        want = got if want is None else want
        assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1]), (n, le, plan.info().variant)
        plan.close()
