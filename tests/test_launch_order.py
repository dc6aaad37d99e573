"""A kernel lets its successor launch only after its own wait for its
predecessor: otherwise every grid of a chain lets the next one in at once, and
waiting blocks crowd the running ones onto few SMs (CPU lint)."""
import os

from tests.test_bounded_waits import CSRC, function_spans, blank


def test_the_wait_comes_before_the_release():
    with open(os.path.join(CSRC, "fft_device.cuh")) as f:
        text = f.read()
    (body,) = [text[b:e] for name, b, e in function_spans(blank(text)) if name == "pdl_enter"]
    assert 0 <= body.find("griddepcontrol.wait") < body.find("griddepcontrol.launch_dependents")
    assert text.count("griddepcontrol.launch_dependents") == 1
