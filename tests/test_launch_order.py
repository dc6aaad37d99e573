"""A kernel lets its successor launch only after its own wait for its
predecessor: otherwise every grid of a chain lets the next one in at once, and
waiting blocks crowd the running ones onto few SMs (CPU lint)."""
import re

from tests.test_bounded_waits import blank, function_spans, sources
from tests.test_launch_lint import PLAIN_ONLY


def test_the_wait_comes_before_the_release():
    kernels = 0
    for name, text in sources():
        code = blank(text)
        spans = {fn: code[b:e] for fn, b, e in function_spans(code)}
        if "pdl_enter" in spans:
            raw = {fn: text[b:e] for fn, b, e in function_spans(code)}
            assert "griddepcontrol.wait" in raw["pdl_enter"] and "launch_dependents" not in raw["pdl_enter"]
            assert text.count('"griddepcontrol.launch_dependents') == 1 and "launch_dependents" in raw["pdl_release"]
        for m in re.finditer(r"__global__\b[^{;]*?(\w+)\s*\((?:const|RaggedArgs)", code):
            if m.group(1) in PLAIN_ONLY:
                continue
            body = spans[m.group(1)]
            assert body.count("pdl_enter()") == body.count("pdl_release()") == 1, (name, m.group(1))
            assert body.index("pdl_enter()") < body.index("pdl_release()"), (name, m.group(1))
            kernels += 1
    assert kernels >= 14
