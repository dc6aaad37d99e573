"""The tuner's number 0 is the schedule by size of the call, which is what a
default of 0 gives later plans: it is timed as a plan that names no variant, and
the default in force meanwhile is put back.  (CPU: plans and times are stand-ins.)"""
import pytest

import paper_2203_09384_gb300 as gb
from paper_2203_09384_gb300 import _abi, autotune

N = 256
FP32 = [v for v in range(_abi.fft_variant_count(N)) if _abi.fft_variant_dtype(N, v) == _abi.FFT_C64]
OTHER = FP32[1]


@pytest.fixture
def made(monkeypatch):
    plans = []

    class FakePlan:
        def __init__(self, n, batch, variant=None, device=None):
            plans.append((variant, _abi.fft_get_default_variant(n)))

        def execute(self, x, out):
            pass

        def error(self):
            return 0

        def close(self):
            pass

    monkeypatch.setattr(gb, "Plan", FakePlan)
    monkeypatch.setattr(autotune, "_time", lambda fn, reps: len(plans))  # the first candidate is the fastest
    before = _abi.fft_get_default_variant(N)
    yield plans
    _abi.fft_set_default_variant(N, before)


def test_zero_is_timed_by_size(made):
    _abi.fft_set_default_variant(N, OTHER)
    result = autotune.tune_lengths([N], elems=1 << 12, apply=False, device="cpu")
    assert made[0] == (None, 0)
    assert [v for v, _ in made[1:]] == FP32[1:] and all(d == OTHER for _, d in made[1:])
    assert result[N]["best"] == 0 and sorted(result[N]["ms"]) == FP32
    assert _abi.fft_get_default_variant(N) == OTHER
    autotune.tune_lengths([N], elems=1 << 12, device="cpu")
    assert _abi.fft_get_default_variant(N) == 0


def test_a_plan_that_cannot_be_made_leaves_the_default(made, monkeypatch):
    def broken(*a, **k):
        raise RuntimeError

    monkeypatch.setattr(gb, "Plan", broken)
    _abi.fft_set_default_variant(N, OTHER)
    with pytest.raises(RuntimeError):
        autotune.tune_lengths([N], elems=1 << 12, device="cpu")
    assert _abi.fft_get_default_variant(N) == OTHER
