"""complex32 kernels with two signals per thread (csrc/fft_pair.cuh).

CPU: the exchange swizzle and the grouped tile layout are replayed from the
schedule rows: the swizzle is linear over XOR (the kernels split an address
into the thread's base and a compile-time offset), a permutation of each tile,
and every 128-bit exchange access and every tile access is free of bank
conflicts (128-bit accesses resolve per quarter-warp, 64-bit ones per
half-warp).  GPU: odd and partial tiles, in place, every row, against the
oracle; the stall test mode of the per-warp ring.
"""
import numpy as np
import pytest
import torch

import oracle
import synth
from tests.helpers import FP32_TOL, c32_decode, c32_encode, c32_to, rel_l2_per_signal
from tests.test_bank_model import _rows, wavefronts

PAIR_ROWS = [dict(L=r[0], variant=r[1], E=r[2], S=r[3], radix=[x for x in r[4:8] if x], D=r[9])
             for r in _rows("GBFFT_C32_SCHEDULES", 11) if r[10] & 7 == 6]
IDS = [f"N{1 << r['L']}-v{r['variant']}" for r in PAIR_ROWS]
# binary16 storage of every output component, plus the FP32 arithmetic
C32_TOL = 2.0 ** -11 + FP32_TOL


def swz(a):
    return a ^ (((a >> 3) ^ (a >> 6)) & 7)


def geometry(row):
    N = 1 << row["L"]
    T = N // row["E"]
    NT = row["S"] // 2 * T
    SU = row["S"] // (NT // 32) if T <= 32 else row["S"]

    def bfly(s, t, c):
        K = row["E"] // row["radix"][s]
        return K * t + c if s in (0, len(row["radix"]) - 1) else t + T * c

    def groups(s):
        if T > 32:
            return 1
        return max(1, (16 if row["E"] // row["radix"][s] >= 2 else 32) // T)

    return N, T, NT, SU, bfly, groups


@pytest.mark.parametrize("row", PAIR_ROWS, ids=IDS)
def test_exchanges_write_every_slot_once_without_conflicts(row):
    N, T, NT, _, bfly, _ = geometry(row)
    E, radix = row["E"], row["radix"]
    ns = [int(np.prod(radix[:s])) for s in range(len(radix))]
    for s in range(len(radix) - 1):
        R, Ns, R1 = radix[s], ns[s], radix[s + 1]
        stored = {}
        for w in range(0, NT, 32):
            for c in range(E // R):
                for q in range(R):
                    at = []
                    for tid in range(w, w + 32):
                        p, t = divmod(tid, T)
                        j = bfly(s, t, c)
                        base, k = p * N + j // Ns * Ns * R + j % Ns, q * Ns
                        a = (swz(base) ^ (swz(k) & 7)) + (swz(k) & ~7)  # pair_slot
                        assert a == swz(base + k)
                        assert a not in stored
                        stored[a] = (p, base + k)
                        at.append(a)
                    assert wavefronts(at, 8, 8) == 4
        assert sorted(stored) == list(range(NT // T * N))
        for w in range(0, NT, 32):
            for c in range(E // R1):
                for r in range(R1):
                    at = []
                    for tid in range(w, w + 32):
                        p, t = divmod(tid, T)
                        base, k = p * N + bfly(s + 1, t, c), r * (N // R1)
                        a = (swz(base) ^ (swz(k) & 7)) + (swz(k) & ~7)
                        assert stored[a] == (p, base + k)
                        at.append(a)
                    assert wavefronts(at, 8, 8) == 4


@pytest.mark.parametrize("row", [r for r in PAIR_ROWS if r["L"] <= 9],
                         ids=[i for r, i in zip(PAIR_ROWS, IDS) if r["L"] <= 9])
def test_tiles_hold_every_signal_apart_and_are_read_without_conflicts(row):
    N, T, _, SU, bfly, groups = geometry(row)
    E, radix = row["E"], row["radix"]
    gin = groups(0)
    own = [(p % gin) * (SU // gin) + p // gin * 2 for p in range(32 // T)]  # pair_signal
    assert sorted(own + [o + 1 for o in own]) == list(range(SU))
    for s in (0, len(radix) - 1):
        g = groups(s)
        place = [sig * N + (sig // (SU // g) * (32 // g) if g > 1 else 0) for sig in range(SU)]  # pair_place
        assert all(b - a >= N for a, b in zip(place, place[1:]))
        assert place[-1] + N <= SU * N + 32  # the slot's gap bytes; 4-byte elements
        K = E // radix[s]
        for q in range(radix[s]):
            first = [place[own[lane // T]] + bfly(s, lane % T, 0) + q * (N // radix[s]) for lane in range(32)]
            if K >= 2:
                assert all(a % 2 == 0 for a in first)
                assert wavefronts([a // 2 for a in first], 16, 16) == 2
            else:
                assert wavefronts(first, 32, 32) == 1


@pytest.mark.gpu
@pytest.mark.parametrize("inverse", [False, True])
@pytest.mark.parametrize("row", PAIR_ROWS, ids=IDS)
def test_partial_tiles_and_in_place(row, inverse):
    import paper_2203_09384_gb300 as gb

    n, S = 1 << row["L"], row["S"]
    for batch in sorted({1, 2, 3, S - 1, S, S + 1, 5 * S + 3, 2500 * S // 2 + 1}):
        if batch < 1:
            continue
        x, _ = synth.scaled_normal(batch, n, seed=batch)
        xs, xe = c32_encode(x.numpy())
        want = oracle.reference(c32_decode(xs, xe), inverse, True, threads=8)
        plan = gb.Plan(n, batch, inverse=inverse, dtype="c32", variant=row["variant"])
        try:
            guard = 8  # signals past the batch that must stay as they are
            buf = torch.full((batch + guard, 2 * n), 3.0, dtype=torch.float16, device="cuda")
            exp = torch.full((batch + guard,), 9, dtype=torch.int8, device="cuda")
            d, e = buf[:batch].view(torch.complex32), exp[:batch]
            buf[:batch] = c32_to(xs, "cuda").view(torch.float16)
            e.copy_(xe)
            plan.execute_c32(d, e, d, e)
            torch.cuda.synchronize()
            assert plan.error() == 0
        finally:
            plan.close()
        assert torch.all(buf[batch:] == 3.0) and torch.all(exp[batch:] == 9)
        assert rel_l2_per_signal(c32_decode(c32_to(d, "cpu"), e.cpu()), want).max() <= C32_TOL, (n, batch)


@pytest.mark.gpu
@pytest.mark.parametrize("n", [64, 512])
def test_per_warp_ring_reports_timeout(n):
    import paper_2203_09384_gb300 as gb
    from paper_2203_09384_gb300 import _abi

    batch = 5000
    xs = torch.zeros(batch, 2 * n, dtype=torch.float16, device="cuda").view(torch.complex32)
    xe = torch.zeros(batch, dtype=torch.int8, device="cuda")
    ys = torch.full((batch, 2 * n), 1.0, dtype=torch.float16, device="cuda").view(torch.complex32)
    ye = torch.full((batch,), 5, dtype=torch.int8, device="cuda")
    plan = gb.Plan(n, batch, dtype="c32", extra_flags=gb.FFT_FLAG_TEST_STALL)
    plan.set_wait_limit(1_000_000)  # 1 ms
    plan.execute_c32(xs, xe, ys, ye)
    torch.cuda.synchronize()
    assert plan.error() == _abi.STATUS_CODE["FFT_ERR_TIMEOUT"]
    assert torch.all(ys.view(torch.float16) == 1.0) and torch.all(ye == 5)  # nothing stored
    plan.close()
