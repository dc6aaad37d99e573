"""Ragged work items at the edges of a ring slot (default and 3-slot forms).

A slot's item is at most one tile of a length: one signal, a whole tile, one
more than a tile; its signals back to back or scattered among other lengths.
The producer warp passes every item's length, count and offsets to the compute
threads through shared memory, so a wrong one shows as signals at the wrong
place.  Tolerance: FP32_TOL, the FP32 kernels' bound against the FP64 oracle.
"""
import numpy as np
import pytest

import oracle
import synth
from tests.helpers import FP32_TOL, max_rel_l2

pytestmark = pytest.mark.gpu

import paper_2203_09384_gb300 as gb  # noqa: E402


def _lengths(log2n, contig, variant):
    """One signal less than a tile, a tile, one more, and three of a tile and one."""
    n = 2 ** log2n
    tile = {1: 256, 2: 128, 3: 128, 4: 128, 5: 128}.get(log2n, 4096 >> log2n) // (1 if variant == 5 else 2)
    other = 2 if n > 2 else 8
    counts = [max(tile - 1, 1), tile, tile + 1, 3 * tile + 1]
    if contig:
        return np.concatenate([np.concatenate([np.full(c, n), [other]]) for c in counts])
    return np.concatenate([np.stack([np.full(c, n), np.full(c, other)], 1).reshape(-1) for c in counts])


@pytest.mark.parametrize("variant", [None, 5, 7])
@pytest.mark.parametrize("contig", [True, False])
@pytest.mark.parametrize("log2n", range(1, 12))
def test_items_at_the_edges_of_a_slot(log2n, contig, variant):
    lengths = _lengths(log2n, contig, variant)
    offsets = np.concatenate([[4], 4 + np.cumsum(lengths)])
    x = synth.uniform(1, int(offsets[-1]), seed=100 + log2n).reshape(-1)
    inverse = bool(log2n % 2)
    plan = gb.RaggedPlan(offsets, inverse=inverse, variant=variant)
    y = plan.execute(x.cuda()).cpu().numpy()
    assert plan.error() == 0
    plan.close()
    for n in np.unique(lengths):
        at = offsets[:-1][lengths == n][:, None] + np.arange(n)
        want = oracle.reference(x.numpy()[at], inverse)
        assert max_rel_l2(y[at].astype(np.complex128), want) <= FP32_TOL, n
