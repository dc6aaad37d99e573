"""Ragged calls of few blocks are launched plainly, larger ones with programmatic
stream serialization: chains that mix both kinds, each reading what the one
before wrote, must be ordered.  Tolerance: a forward and an inverse transform,
each within FP32_TOL, of an input with relative norm 1, so 2 * FP32_TOL a pair."""
import pytest
import torch

import synth
from tests.helpers import FP32_TOL, max_rel_l2, to_np

pytestmark = pytest.mark.gpu

import paper_2203_09384_gb300 as gb  # noqa: E402


@pytest.mark.parametrize("blocks", [1, 63, 64, 65])
def test_chain_across_the_launch_rule(blocks):
    n = 2048  # one signal per work item
    offsets = torch.arange(blocks + 1, dtype=torch.int64) * n
    x = synth.uniform(blocks, n, seed=blocks).cuda()
    fwd = gb.RaggedPlan(offsets)
    inv = gb.Plan(n, blocks, inverse=True)  # always overlapped
    assert fwd.info().grid == blocks
    y, z = torch.empty_like(x), x.clone()
    pairs = 8
    for _ in range(pairs):
        fwd.execute(z.reshape(-1), y.reshape(-1))
        inv.execute(y, z)
    assert max_rel_l2(to_np(z), to_np(x)) <= pairs * 2 * FP32_TOL
    assert fwd.error() == 0 and inv.error() == 0
    fwd.close()
    inv.close()
