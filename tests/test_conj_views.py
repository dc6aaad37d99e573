"""Lazily conjugated tensors (x.conj() keeps x's storage and sets a flag): the
library reads storage, so every entry point has to hand it the conjugated
values, and refuses a conjugated view as an output."""
import pytest
import torch

import synth

import paper_2203_09384_gb300 as gb


def _fake(cls, monkeypatch, **attrs):
    """A plan on the CPU whose launch copies `in` to `out`, bytes as stored."""
    import ctypes

    plan = cls.__new__(cls)
    plan.handle, plan.device = None, torch.device("cpu")
    for k, v in attrs.items():
        setattr(plan, k, v)

    def enqueue(index, stream, call, handle, src, *rest):
        ctypes.memmove(rest[0] if len(rest) < 3 else rest[1], src, plan.nbytes)

    monkeypatch.setattr(gb, "_enqueue", enqueue)
    return plan


def test_plans_read_the_conjugated_values(monkeypatch):
    x = torch.complex(torch.arange(8.0), torch.arange(8.0) + 0.5)
    plan = _fake(gb.Plan, monkeypatch, n=4, batch=2, nbytes=64)
    assert torch.equal(plan.execute(x.conj()), x.conj().resolve_conj())
    ragged = _fake(gb.RaggedPlan, monkeypatch, total=8, nbytes=64)
    assert torch.equal(ragged.execute(x.conj()), x.conj().resolve_conj())
    c32 = _fake(gb.Plan, monkeypatch, n=4, batch=2, nbytes=32)
    h, e = x.to(torch.complex32), torch.zeros(2, dtype=torch.int8)
    got, _ = c32.execute_c32(h.conj(), e)
    assert torch.equal(torch.view_as_real(got), torch.view_as_real(h) * torch.tensor([1.0, -1.0]).half())


def test_conjugated_outputs_are_refused(monkeypatch):
    x = torch.zeros(8, dtype=torch.complex64)
    with pytest.raises(ValueError, match="conjugated"):
        _fake(gb.Plan, monkeypatch, n=4, batch=2, nbytes=64).execute(x, torch.zeros_like(x).conj())
    with pytest.raises(ValueError, match="conjugated"):
        _fake(gb.RaggedPlan, monkeypatch, total=8, nbytes=64).execute(x, torch.zeros_like(x).conj())


@pytest.mark.gpu
def test_every_entry_point_against_the_materialised_conjugate():
    n, batch = 64, 33
    x = synth.uniform(batch, n, seed=8, device="cuda")
    c = x.conj()
    m = c.resolve_conj()
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    for inverse in (False, True):
        one = gb.ifft if inverse else gb.fft
        assert torch.equal(one(c), one(m))
        assert torch.equal(one(c.t().contiguous().t()), one(m))  # copied by .contiguous(), the flag kept
        plan = gb.Plan(n, batch, inverse=inverse, host_staging=True)
        want = plan.execute(m)
        assert torch.equal(plan.execute(c), want)
        got = plan.execute(c, stream=side)
        side.synchronize()
        assert torch.equal(got, want)
        assert torch.equal(plan.execute_host(x.cpu().conj()), want.cpu())
        plan.close()
    ragged = gb.RaggedPlan([i * n for i in range(batch + 1)])
    assert torch.equal(ragged.execute(c.view(-1)), ragged.execute(m.view(-1)))
    ragged.close()
    h = torch.view_as_complex((torch.view_as_real(x) * 100).half())
    e = torch.zeros(batch, dtype=torch.int8, device="cuda")
    hm = torch.view_as_complex(torch.view_as_real(h) * torch.tensor([1.0, -1.0], device="cuda").half())
    c32 = gb.Plan(n, batch, dtype="c32")
    (got, ge), (want, we) = c32.execute_c32(h.conj(), e), c32.execute_c32(hm, e)
    assert torch.equal(got.view(torch.int16), want.view(torch.int16)) and torch.equal(ge, we)
    c32.close()
    g = synth.uniform(batch, n, seed=9, device="cuda")
    a = x.clone().requires_grad_(True)
    for f in (gb.FFTFunction, gb.IFFTFunction):
        (lazy,) = torch.autograd.grad(f.apply(a), a, g.conj())
        (plain,) = torch.autograd.grad(f.apply(a), a, g.conj().resolve_conj())
        assert torch.equal(lazy, plain)
