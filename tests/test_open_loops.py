"""Loops of the kernels that do not count up to a bound (CPU lint).

tests/test_bounded_waits.py finds loops without any condition.  This finds the
rest: loops with an empty or compound condition, loops that run while a tile is
at hand, and every while.  Each is listed with the reason why it ends; a new one
has to be reviewed and listed before this test passes.
"""
import re

from tests.test_bounded_waits import blank, enclosing_function, sources

ENDS = {
    "mbar_wait_bounded": "returns on completion or once the wall-time limit has passed",
    "drain": "RingInFlight: a fixed number of slots.  TileTaker: each pass waits (bounded) for one answer; it goes "
             "on only after an answer with a tile, and a grid has finitely many blocks to take",
    "fft_stockham_slot_ring_kernel": "a fixed stride counts up to the tiles; taken tiles end with the first answer "
                                     "without one or a wait that gave up, marked in the slot every thread reads",
    "fft_pair_c32_ring_kernel": "as fft_stockham_slot_ring_kernel",
    "fft_pair_c32_warp_kernel": "a fixed stride counts up to the tiles; taken tiles end with the first answer "
                                "without one, or at once when a lane's wait gave up",
    "fft_small_steal_kernel": "ends with the first answer without a tile, or when the wait for one gave up",
    "fft_small_c32_steal_kernel": "as fft_small_steal_kernel",
    "fft_ragged_kernel": "the item index only grows and the loop ends past n_items",
    "slot_produce": "the item index only grows and the loop ends past n_items; a wait that gave up ends it too",
    "noalloc_prepare": "at most four stages",
}
HOST = {"small_c32_entry", "small_entry", "ilog2", "ilog2_exact", "ragged_create", "default_variant",
        "fft_plan_get_info"}
COUNTS = re.compile(r"[^<>=!&|]+(<|>|<=|>=|!=)[^<>=!&|]+")


def loops_not_counting(text):
    """The functions of every loop that is not `for (...; a < b; ...)`, and of
    those that run while a tile is at hand."""
    code = blank(text)
    out = []
    for m in re.finditer(r"\bfor\s*\(", code):
        depth, clauses = 0, [""]
        for c in code[m.end() - 1:]:
            depth += {"(": 1, ")": -1}.get(c, 0)
            if depth == 0:
                break
            if c == ";" and depth == 1:
                clauses.append("")
            elif not (c == "(" and depth == 1):
                clauses[-1] += c
        if len(clauses) != 3:
            continue  # range for
        cond = re.sub(r"\w+<[\w:, ]*>|->", "", clauses[1]).strip()
        if not COUNTS.fullmatch(cond) or "kSteal" in cond or re.search(r"\btile\s*>=", cond):
            out.append(enclosing_function(code, m.start()))
    out += [enclosing_function(code, m.start()) for m in re.finditer(r"\bwhile\s*\(", code)]
    return out


def test_every_loop_that_does_not_count_is_reviewed():
    seen = set()
    for name, text in sources():
        for fn in loops_not_counting(text):
            assert fn in ENDS or fn in HOST, (name, fn)
            seen.add(fn)
    assert {"drain", "fft_stockham_slot_ring_kernel", "fft_pair_c32_ring_kernel", "fft_small_steal_kernel"} <= seen


def test_the_lint_sees_planted_loops():
    planted = """
    void a() { for (int i = 0; i < n; ++i) { } }
    void b() { for (int t = x;; t += 1) { } }
    void c() { for (long t = x; C::kSteal || t < n; t += 1) { } }
    void d() { for (long tile = x; tile >= 0;) { } }
    void e() { while (!done) { } }
    """
    assert loops_not_counting(planted) == ["b", "c", "d", "e"]
