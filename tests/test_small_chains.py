"""Small dependent calls back to back: each kernel is launched programmatically
and waits for its predecessor itself, so chains in place, across kernel
families and behind other kernels of the stream read finished results."""
import pytest
import torch

import synth
from tests.helpers import FP32_TOL, c32_encode, c32_to

pytestmark = pytest.mark.gpu

import paper_2203_09384_gb300 as gb  # noqa: E402


@pytest.mark.parametrize("capture", [False, True])
@pytest.mark.parametrize("n,batch", [(2, 5), (8, 3001), (64, 16), (256, 77), (512, 1000), (1024, 3), (2048, 301)])
def test_in_place_round_trips(n, batch, capture):
    x = synth.uniform(batch, n, seed=n, device="cuda")
    fwd, inv = gb.Plan(n, batch), gb.Plan(n, batch, inverse=True)
    a = x.clone()

    def chain():
        for _ in range(8):
            fwd.execute(a, a)
            inv.execute(a, a)
            a.mul_(2.0)  # another library's kernel in between
            fwd.execute(a, a)
            a.mul_(0.5)
            inv.execute(a, a)

    if capture:
        chain()
        a.copy_(x)
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            chain()
        g.replay()
    else:
        chain()
    torch.cuda.synchronize()
    assert fwd.error() == 0 and inv.error() == 0
    assert float(((a - x).norm(dim=1) / x.norm(dim=1)).max()) <= 32 * FP32_TOL
    fwd.close()
    inv.close()


def test_ragged_and_complex32_between_plain_calls():
    n, batch = 128, 40
    x = synth.uniform(batch, n, seed=4, device="cuda")
    plain, back = gb.Plan(n, batch), gb.Plan(n, batch, inverse=True)
    offs = [i * n for i in range(batch + 1)]
    for variant in (0, 3, 4, 9):
        ragged = gb.RaggedPlan(offs, inverse=True, variant=variant)
        a = x.clone()
        for _ in range(8):
            plain.execute(a, a)
            ragged.execute(a.view(-1), a.view(-1))
        torch.cuda.synchronize()
        assert ragged.error() == 0
        assert float(((a - x).norm(dim=1) / x.norm(dim=1)).max()) <= 16 * FP32_TOL
        ragged.close()
    xs, xe = c32_encode(x.cpu().numpy())
    xs, xe = c32_to(xs, "cuda"), xe.cuda()
    f, b = gb.Plan(n, batch, dtype="c32"), gb.Plan(n, batch, dtype="c32", inverse=True)
    y, e = f.execute_c32(xs, xe)
    want, we = b.execute_c32(y, e)
    torch.cuda.synchronize()
    for _ in range(8):  # the same two calls in place, launched without a gap
        d, de = xs.clone(), xe.clone()
        f.execute_c32(d, de, d, de)
        b.execute_c32(d, de, d, de)
    torch.cuda.synchronize()
    assert torch.equal(d.view(torch.int16), want.view(torch.int16)) and torch.equal(de, we)
    for p in (plain, back, f, b):
        p.close()
