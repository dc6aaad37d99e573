"""Every thread decides a bounded wait for itself, so some threads of a block may
give up where others do not.  Whatever a warp or a block does together
(barriers, shuffles, votes, the aligned tensor-core instructions) must then not
sit under a condition on the thread's own outcome.

CPU: a lint of the kernels that take the tiles of unstarted blocks, where a
thread that gave up has no tile.  GPU: the stall test mode of every schedule
whose first stage holds such steps (all threads give up together there)."""
import os
import re
import time

import pytest
import torch

import synth
from tests.helpers import oracle_max_rel_l2
from tests.test_bank_model import _rows
from tests.test_bounded_waits import CSRC, blank, function_spans

KERNELS = [("fft_device.cuh", "fft_stockham_slot_ring_kernel"), ("fft_device.cuh", "fft_small_steal_kernel"),
           ("fft_device.cuh", "fft_small_c32_steal_kernel"), ("fft_pair.cuh", "fft_pair_c32_warp_kernel"),
           ("fft_pair.cuh", "fft_pair_c32_ring_kernel")]
TOGETHER = r"__sync\w+|__shfl\w+|__any_sync|__reduce_\w+|\bpair_stages\b|\btwist_and_dft\b|\btc_norm_\w+\b"
UNIFORM = r"__any_sync|__syncthreads_or|C::kStage0Together"  # conditions all threads of a warp or block share


def _closing(code, at, pair):
    depth = 0
    for k in range(at, len(code)):
        depth += {pair[0]: 1, pair[1]: -1}.get(code[k], 0)
        if depth == 0:
            return k
    raise AssertionError("unbalanced")


def steps_under_a_threads_own_outcome(body):
    """(condition, step) for every step taken together inside an if whose
    condition is one thread's (its `tile` or `dead`)."""
    out = []
    for m in re.finditer(r"\bif\s*\(", body):
        close = _closing(body, m.end() - 1, "()")
        cond = body[m.end():close]
        if not re.search(r"\b(tile|dead)\b", cond) or re.search(UNIFORM, cond):
            continue
        rest = body[close + 1:]
        start = close + 1 + len(rest) - len(rest.lstrip())
        end = _closing(body, start, "{}") if body[start] == "{" else body.index(";", start)
        out += [(cond.strip(), s) for s in re.findall(TOGETHER, body[start:end])]
    return out


def _body(source, kernel):
    with open(os.path.join(CSRC, source)) as f:
        code = blank(f.read())
    (span,) = [(b, e) for name, b, e in function_spans(code) if name == kernel]
    return code[span[0]:span[1]]


@pytest.mark.parametrize("source,kernel", KERNELS)
def test_no_common_step_depends_on_one_threads_wait(source, kernel):
    assert steps_under_a_threads_own_outcome(_body(source, kernel)) == []


def test_the_lint_sees_planted_steps():
    planted = "if (!C::kSteal || tile >= 0) { gather(); twist_and_dft<C, 0>(v); } if (dead) __syncwarp(); if (a) __syncwarp();"
    assert [s for _, s in steps_under_a_threads_own_outcome(planted)] == ["twist_and_dft", "__syncwarp"]


ROWS = [(1 << r[0], r[1]) for r in _rows("GBFFT_GENERIC_SCHEDULES", 13) if r[10] and r[12] & 4]


@pytest.mark.gpu
@pytest.mark.parametrize("n,variant", ROWS)
def test_a_stalled_tensor_core_grid_ends(n, variant):
    import paper_2203_09384_gb300 as gb
    from paper_2203_09384_gb300 import _abi

    batch = (1 << 25) // n
    x = synth.uniform(batch, n, seed=1, device="cuda")
    out = torch.zeros_like(x)
    dtype = gb.DTYPE_NAMES[gb.fft_variant_dtype(n, variant)]
    plan = gb.Plan(n, batch, variant=variant, dtype=dtype, extra_flags=gb.FFT_FLAG_TEST_STALL)
    plan.set_wait_limit(100_000_000)
    t0 = time.perf_counter()
    plan.execute(x, out)
    assert plan.error() == _abi.STATUS_CODE["FFT_ERR_TIMEOUT"]
    assert time.perf_counter() - t0 < 3.0
    assert torch.count_nonzero(out) == 0
    plan.close()
    plan = gb.Plan(n, batch, variant=variant, dtype=dtype)  # one tile a block or more, its end included
    plan.execute(x, out)
    assert plan.error() == 0
    assert oracle_max_rel_l2(x, out)[0] <= 5e-3
    plan.close()
