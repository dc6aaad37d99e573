"""Performance cases: the calls a program that uses this package makes, over
the range of lengths, batches, storage types and entry points it offers.

A case is a dict of plain values.  ``kind`` names the entry point:

  pair    fft() then ifft() of its result: a spectrum edited in between is
          the usual reason to call both
  func    fft() or ifft() on a tensor [batch, n], the output allocated by the call
  plan    Plan.execute into a kept output buffer; ``dtype`` is the plan's
          (complex64 in and out: c64, tc_f16, tc_bf16)
  grad    FFTFunction forward and its backward for a given output gradient
  ragged  RaggedPlan over signals of mixed lengths packed in a random order
          (or sorted by length), as a captured graph or a plain execute
  c32     Plan.execute_c32: binary16 pairs with one exponent per signal
  host    Plan.execute_host on pinned host buffers
"""
from __future__ import annotations

import math

import torch

import paper_2203_09384_gb300 as gb


def listed():
    return [
        # a small interactive call: 16 short signals there and back
        {"name": "pair_n64_b16", "kind": "pair", "n": 64, "batch": 16},
        # one chunk of a stream of frames: about a million samples, odd batch
        {"name": "plan_n256_b5001", "kind": "plan", "n": 256, "batch": 5001, "inverse": False, "dtype": "c64"},
        # an ordinary inverse transform through the functional interface
        {"name": "ifft_n1024_b3001", "kind": "func", "n": 1024, "batch": 3001, "inverse": True},
        # a great many tiny signals (per-sample sensor windows), odd batch
        {"name": "plan_n8_b1000003", "kind": "plan", "n": 8, "batch": 1000003, "inverse": False, "dtype": "c64"},
        # the length sweep's batch of 2^28 elements, at a middle length
        {"name": "plan_n512_2p28", "kind": "plan", "n": 512, "batch": 1 << 19, "inverse": False, "dtype": "c64"},
        # a training step's transform and its adjoint
        {"name": "grad_n1024_b65536", "kind": "grad", "n": 1024, "batch": 65536},
        # mixed lengths 2^4..2^11 in one graph-captured launch
        {"name": "ragged_20000", "kind": "ragged", "count": 20000, "lo": 4, "hi": 11, "sorted": False,
         "inverse": False, "graph": True},
        # tensor-core stages on signals of widely different scale
        {"name": "tc_f16_n256_2p17", "kind": "plan", "n": 256, "batch": 1 << 17, "inverse": False, "dtype": "tc_f16"},
        {"name": "tc_bf16_n2048_2p17", "kind": "plan", "n": 2048, "batch": 1 << 17, "inverse": False,
         "dtype": "tc_bf16"},
        # half-size storage: a large batch of the longest signals ...
        {"name": "c32_n2048_b65536", "kind": "c32", "n": 2048, "batch": 65536, "inverse": False},
        # ... and an ordinary one of short signals, odd batch, inverse
        {"name": "c32_n128_b100003", "kind": "c32", "n": 128, "batch": 100003, "inverse": True},
        # data that lives on the host: in, transform, out
        {"name": "host_n1024_b16384", "kind": "host", "n": 1024, "batch": 16384, "inverse": False},
    ]


def _batch(rng, n, lo, hi):
    """A batch of n-point signals of 2^lo..2^hi elements, spread over the logarithm."""
    return max(1, int(2.0 ** rng.uniform(lo, hi)) // n)


def draw(rng):
    kind = rng.choice(["pair", "func", "plan", "plan", "grad", "ragged", "tc", "c32", "c32", "host"])
    inverse = rng.random() < 0.5
    n = 1 << rng.randint(1, 11)
    if kind == "pair":
        return {"kind": "pair", "n": n, "batch": _batch(rng, n, 10, 20)}
    if kind == "func":
        return {"kind": "func", "n": n, "batch": _batch(rng, n, 12, 26), "inverse": inverse}
    if kind == "plan":
        return {"kind": "plan", "n": n, "batch": _batch(rng, n, 14, 28), "inverse": inverse, "dtype": "c64"}
    if kind == "grad":
        return {"kind": "grad", "n": n, "batch": _batch(rng, n, 16, 26)}
    if kind == "ragged":
        lo = rng.randint(1, 9)
        hi = rng.randint(lo + 1, 11)
        mean = sum(1 << k for k in range(lo, hi + 1)) / (hi - lo + 1)
        most = min(40000, int(10.2e6 / mean))
        return {"kind": "ragged", "count": int(math.exp(rng.uniform(math.log(200), math.log(most)))), "lo": lo,
                "hi": hi, "sorted": rng.random() < 0.25, "inverse": inverse, "graph": rng.random() < 0.5}
    if kind == "tc":
        n = 1 << rng.randint(7, 11)
        return {"kind": "plan", "n": n, "batch": _batch(rng, n, 18, 28), "inverse": inverse,
                "dtype": rng.choice(["tc_f16", "tc_bf16"])}
    if kind == "c32":
        return {"kind": "c32", "n": n, "batch": _batch(rng, n, 16, 27), "inverse": inverse}
    return {"kind": "host", "n": n, "batch": _batch(rng, n, 16, 24), "inverse": inverse}


# ---------------------------------------------------------------------------
# inputs, from the seed alone
# ---------------------------------------------------------------------------
def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _uniform(shape, g):
    """complex64, real and imaginary parts uniform on [-1, 1]."""
    r = torch.rand(*shape, 2, generator=g, device="cuda", dtype=torch.float32)
    return torch.view_as_complex(r.mul_(2.0).sub_(1.0))


def _normal(shape, g):
    return torch.view_as_complex(torch.randn(*shape, 2, generator=g, device="cuda", dtype=torch.float32))


def _scaled_normal(batch, n, g):
    """Normal signals, each scaled by 10^u, u uniform on [-3, 3]."""
    x = _normal((batch, n), g)
    u = torch.rand(batch, generator=g, device="cuda", dtype=torch.float32) * 6.0 - 3.0
    return torch.view_as_complex(torch.view_as_real(x).mul_(torch.pow(10.0, u)[:, None, None]))


def _c32(batch, n, g):
    """binary16 pairs [batch, n, 2] and one exponent per signal (value = stored * 2^exp)."""
    x = torch.randn(batch, n, 2, generator=g, device="cuda", dtype=torch.float32).mul_(1024.0)
    e = torch.randint(-12, 13, (batch,), generator=g, device="cuda", dtype=torch.int64)
    return x.to(torch.float16), e.to(torch.int8)


def _offsets(case, seed):
    """Lengths (each power of two equally often, in an order drawn from the
    seed) and the start of every signal in the packed buffer, the total last."""
    lengths = 1 << (case["lo"] + torch.arange(case["count"]) % (case["hi"] + 1 - case["lo"]))
    if case["sorted"]:
        lengths = lengths.sort().values
    else:
        lengths = lengths[torch.randperm(case["count"], generator=torch.Generator().manual_seed(seed))]
    off = torch.zeros(case["count"] + 1, dtype=torch.int64)
    off[1:] = lengths.cumsum(0)
    return lengths, off


def _inputs(case, seed):
    g = _generator(seed)
    kind = case["kind"]
    if kind == "ragged":
        lengths, off = _offsets(case, seed)
        return {"lengths": lengths, "offsets": off, "x": _uniform((int(off[-1]),), g)}
    shape = (case["batch"], case["n"])
    if kind == "grad":
        return {"x": _normal(shape, g), "g": _normal(shape, g)}
    if kind == "c32":
        x, e = _c32(*shape, g)
        return {"x": x, "e": e}
    if case.get("dtype", "c64") != "c64":
        return {"x": _scaled_normal(*shape, g)}
    return {"x": _uniform(shape, g)}


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def prepare(case, seed):
    kind = case["kind"]
    s = dict(_inputs(case, seed), kind=kind, inverse=case.get("inverse", False))
    if kind == "plan":
        s["plan"] = gb.Plan(case["n"], case["batch"], inverse=case["inverse"], dtype=case["dtype"])
        s["out"] = torch.empty_like(s["x"])
    elif kind == "grad":
        s["x"].requires_grad_(True)
    elif kind == "ragged":
        s["plan"] = gb.RaggedPlan(s["offsets"], inverse=case["inverse"])
        s["out"] = torch.empty_like(s["x"])
        s["graph"] = s["plan"].capture(s["x"], s["out"]) if case["graph"] else None
    elif kind == "c32":
        s["plan"] = gb.Plan(case["n"], case["batch"], inverse=case["inverse"], dtype="c32")
        s["x"] = torch.view_as_complex(s["x"])
        s["out"] = torch.empty_like(s["x"])
        s["out_exp"] = torch.empty_like(s["e"])
    elif kind == "host":
        s["plan"] = gb.Plan(case["n"], case["batch"], inverse=case["inverse"], host_staging=True)
        host = torch.empty(s["x"].shape, dtype=s["x"].dtype, pin_memory=True)
        s["x"] = host.copy_(s["x"])
        s["out"] = torch.empty(host.shape, dtype=host.dtype, pin_memory=True)
    return s


def run(state):
    kind, x = state["kind"], state["x"]
    if kind == "pair":
        spectrum = gb.fft(x)
        return spectrum, gb.ifft(spectrum)
    if kind == "func":
        return gb.ifft(x) if state["inverse"] else gb.fft(x)
    if kind == "plan":
        return state["plan"].execute(x, state["out"])
    if kind == "grad":
        y = gb.FFTFunction.apply(x)
        return y, torch.autograd.grad(y, x, state["g"])[0]
    if kind == "ragged":
        if state["graph"] is not None:
            state["graph"].replay()
            return state["out"]
        return state["plan"].execute(x, state["out"])
    if kind == "c32":
        out, exp = state["plan"].execute_c32(x, state["e"], state["out"], state["out_exp"])
        return torch.view_as_real(out), exp
    return state["plan"].execute_host(x, state["out"])


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def work(case):
    """Each input read once, each output written once; 5 N log2 N operations a transform."""
    if case["kind"] == "ragged":
        logs = [case["lo"] + k % (case["hi"] + 1 - case["lo"]) for k in range(case["count"])]
        return {"bytes": sum(16 << k for k in logs), "flops": sum((5 * k) << k for k in logs)}
    n, batch = case["n"], case["batch"]
    passes = 2 if case["kind"] in ("pair", "grad") else 1
    per_signal = 8 * n + 2 if case["kind"] == "c32" else 16 * n
    return {"bytes": passes * batch * per_signal, "flops": passes * batch * 5 * n * (n.bit_length() - 1)}


# ---------------------------------------------------------------------------
# the same outputs in 64 bits, from torch alone
# ---------------------------------------------------------------------------
def _dft(x, inverse=False, norm="backward"):
    x = x.to(torch.complex128)
    return torch.fft.ifft(x, norm=norm) if inverse else torch.fft.fft(x, norm=norm)


def exact(case, seed):
    kind, s = case["kind"], _inputs(case, seed)
    if kind == "pair":
        return _dft(s["x"]), s["x"].to(torch.complex128)
    if kind == "grad":
        return _dft(s["x"]), _dft(s["g"], True, "forward")  # the adjoint: not normalised
    if kind == "ragged":
        start, lengths = s["offsets"][:-1].cuda(), s["lengths"].cuda()
        out = torch.empty(s["x"].shape, dtype=torch.complex128, device="cuda")
        for n in lengths.unique().tolist():
            at = start[lengths == n][:, None] + torch.arange(n, device="cuda")
            out[at] = _dft(s["x"][at], case["inverse"])
        return out
    if kind == "c32":
        # stored numbers: the exponent that puts a signal's largest component in [2^14, 2^15)
        y = torch.view_as_real(_dft(torch.view_as_complex(s["x"].to(torch.float64)), case["inverse"]))
        _, f = torch.frexp(y.abs().amax(dim=(1, 2)))
        return torch.ldexp(y, (15 - f)[:, None, None].to(torch.float64)), None
    return _dft(s["x"], case.get("inverse", False))
