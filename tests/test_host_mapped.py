"""fft_execute_host on page-locked buffers runs one kernel over the mapped host
memory; anything else goes through the staging copies.  Both give what a
device-buffer execute of the same plan gives, bit for bit, and touch nothing
outside the range."""
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu

import paper_2203_09384_gb300 as gb  # noqa: E402


def _buffers(batch, n, kind):
    """(owner, view) of a [batch, n] complex64 host buffer with 64 guard
    elements on either side; kind: pinned, registered, or pageable."""
    total = batch * n + 128
    if kind == "pinned":
        own = torch.zeros(total, dtype=torch.complex64, pin_memory=True)
    else:
        own = torch.zeros(total, dtype=torch.complex64)
        if kind == "registered":
            assert int(torch.cuda.cudart().cudaHostRegister(own.data_ptr(), total * 8, 0)) == 0
    return own, own[64:64 + batch * n].view(batch, n)


@pytest.mark.parametrize("kinds", [("pinned", "pinned"), ("registered", "pinned"), ("pinned", "pageable"),
                                   ("pageable", "pinned")])
@pytest.mark.parametrize("n,batch,dtype", [(2, 1, "c64"), (8, 100003, "c64"), (64, 3001, "c64"), (256, 77, "c64"),
                                           (512, 40001, "c64"), (1024, 513, "c64"), (2048, 3, "c64"),
                                           (2048, 9001, "c64"), (256, 1001, "tc_f16")])
def test_host_execute_matches_device_execute(n, batch, dtype, kinds):
    x = synth.uniform(batch, n, seed=n)
    for inverse in (False, True):
        plan = gb.Plan(n, batch, inverse=inverse, dtype=dtype, host_staging=True)
        want = plan.execute(x.cuda()).cpu()
        (own_in, hin), (own_out, hout) = _buffers(batch, n, kinds[0]), _buffers(batch, n, kinds[1])
        try:
            hin.copy_(x)
            own_out.fill_(7.0)
            plan.execute_host(hin, hout)
            assert plan.error() == 0
            assert torch.equal(hout, want) and torch.equal(hin, x)
            assert torch.all(own_out[:64] == 7.0) and torch.all(own_out[64 + batch * n:] == 7.0)
            plan.execute_host(hin, hin)  # in place
            assert torch.equal(hin, want)
            assert torch.count_nonzero(own_in[:64]) == 0 and torch.count_nonzero(own_in[64 + batch * n:]) == 0
        finally:
            for own, kind in ((own_in, kinds[0]), (own_out, kinds[1])):
                if kind == "registered":
                    torch.cuda.cudart().cudaHostUnregister(own.data_ptr())
            plan.close()


def test_mapped_execute_is_ordered_on_the_callers_stream_and_capturable():
    n, batch = 256, 2000
    x = synth.uniform(batch, n, seed=5)
    plan = gb.Plan(n, batch, host_staging=True)
    want = plan.execute(x.cuda()).cpu()
    hin, hout = torch.zeros(batch, n, dtype=torch.complex64, pin_memory=True), \
        torch.zeros(batch, n, dtype=torch.complex64, pin_memory=True)
    xd, yd = x.cuda(), torch.empty(batch, n, dtype=torch.complex64, device="cuda")
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        hin.copy_(xd, non_blocking=True)  # the transform has to see this copy
        gb.fft_execute_host(plan.handle, hin.data_ptr(), hout.data_ptr(), s.cuda_stream)
        yd.copy_(hout, non_blocking=True)  # and this copy the transform
    s.synchronize()
    assert torch.equal(yd.cpu(), want)
    hout.zero_()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        gb.fft_execute_host(plan.handle, hin.data_ptr(), hout.data_ptr(), s.cuda_stream)
    assert torch.count_nonzero(hout) == 0
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(hout, want)
    plan.close()
