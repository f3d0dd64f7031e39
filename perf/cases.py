"""What a user of the library has it do, as measurable cases: decoding, prefill, training passes of the selective scan
in its real and complex forms, and the short convolution in front of it.

A case is a dict of plain values:

* `op`      "step" (one decoding step), "prefill" (forward only, state out), "train" (forward that saves its checkpoint
            states, then backward) or "conv" (short convolution, forward and backward).
* `batch`, `L`, `D`, `N`, `io` ("bf16" / "f32"): the shape and the element type of the activations.
* `dt`      "given": the step size is an input; "fused": its pre-activation and bias are (softplus inside the call).
* `A`       "init": A[d, n] = -(n + 1), the S4D-Real initialisation; "trained": every entry moved off that
            progression, as after any optimizer step.
* `dt_min`, `dt_max`: the step sizes are log-uniform over the channels in this range.
* `chunk`   the prefill continues from a carried-in state.
* `complex` complex-valued state (A, B, C as (re, im) pairs, A from S4D-Lin).
* `width`   taps of the convolution.

Values: x, z, B, C, dout ~ N(0, 1); delta = softplus(0.1 N(0, 1) + b_d) with softplus(b_d) the channel's step size.
"""
from __future__ import annotations

import math

import torch

from paper_2312_00752_b200 import binding as K

_IO = {"bf16": torch.bfloat16, "f32": torch.float32}
_SCAN = {"io": "bf16", "N": 16, "dt": "given", "A": "init", "dt_min": 1e-3, "dt_max": 1e-1, "chunk": False,
         "complex": False}


def _scan(op, batch, L, D, **kw):
    return {"op": op, "batch": batch, "L": L, "D": D, **_SCAN, **kw}


def listed():
    cases = {
        # one token of 64 sequences through a layer of 2.8B width: the call that a decoding loop makes per layer
        "step_2p8b_b64": _scan("step", 64, 1, 5120, A="trained"),
        # the smallest training call (unit-test and toy-problem size): launches and host time are all of it
        "train_tiny_f32": _scan("train", 1, 256, 64, io="f32"),
        # one sequence's next prompt chunk of no round length at 130M width, continuing from a carried state
        "prompt_130m_b1": _scan("prefill", 1, 333, 1536, dt="fused", A="trained", chunk=True),
        # prefill of a batch at 2.8B width
        "prefill_2p8b": _scan("prefill", 4, 2048, 5120),
        # training of a 130M layer the way the block uses the scan: step-size activation fused, A already trained
        "train_130m_fused": _scan("train", 8, 2048, 1536, dt="fused", A="trained"),
        # the headline: training of a 2.8B layer
        "train_2p8b": _scan("train", 4, 2048, 5120),
        # half a million steps of one sequence with long memory: the time split and its carry; the largest case
        "train_long": _scan("train", 1, 524288, 1536, dt_min=1e-4, dt_max=1e-2),
        # full-precision training at an ordinary size
        "train_f32": _scan("train", 2, 2048, 1536, io="f32"),
        # nothing divides anything: odd width (no aligned rows), ragged length
        "train_odd_bf16": _scan("train", 3, 1237, 1001, A="trained"),
        # a four times larger state at 2.8B width
        "train_n64": _scan("train", 1, 2048, 5120, N=64),
        # complex state, as for continuous signals
        "train_complex": _scan("train", 2, 2048, 1536, complex=True),
        # the convolution + SiLU in front of the scan, both directions, at 2.8B width
        "conv_2p8b": {"op": "conv", "batch": 4, "L": 2048, "D": 5120, "width": 4, "io": "bf16"},
    }
    return [{"name": name, **c} for name, c in cases.items()]


def _log(rng, lo, hi, multiple=1):
    """A whole number in [lo, hi], uniform over its logarithm, rounded to a multiple."""
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return min(hi // multiple, max(-(-lo // multiple), round(v / multiple))) * multiple


def _width(rng, lo, hi):
    """A channel count: multiples of 64 as models have them, more rarely of 8, of 2 or anything."""
    return _log(rng, lo, hi, rng.choice((64, 64, 64, 8, 8, 2, 1)))


def draw(rng):
    kind = rng.choice(("step", "small", "prefill", "prefill", "train", "train", "long", "f32", "odd", "state", "complex",
                       "conv"))
    A, dt = rng.choice(("init", "trained")), rng.choice(("given", "fused"))
    if kind == "step":
        return _scan("step", _log(rng, 1, 256), 1, _width(rng, 512, 8192), N=rng.choice((8, 16, 16, 16, 64)), A=A,
                     io=rng.choice(("bf16", "bf16", "f32")))
    if kind == "small":
        return _scan("train", rng.randint(1, 2), _log(rng, 16, 512), _log(rng, 16, 256), N=rng.choice((4, 8, 16, 16)),
                     io=rng.choice(("f32", "f32", "bf16")), A=A)
    if kind == "prefill":
        batch = rng.randint(1, 8)
        return _scan("prefill", batch, _log(rng, 17, 16384 // batch), _log(rng, 768, 5120, 64), A=A, dt=dt,
                     chunk=rng.random() < 0.5)
    if kind == "train":
        batch = rng.randint(1, 8)
        return _scan("train", batch, _log(rng, 256, 16384 // batch), _log(rng, 768, 5120, 64), A=A, dt=dt,
                     N=rng.choice((16, 16, 16, 8)))
    if kind == "long":
        return _scan("train", 1, _log(rng, 32768, 524288), _log(rng, 256, 1536, 64), A=A, dt_min=1e-4, dt_max=1e-2)
    if kind == "f32":
        return _scan("train", rng.randint(1, 4), _log(rng, 128, 2048), _width(rng, 256, 2048), io="f32", A=A, dt=dt,
                     N=rng.choice((8, 16, 16, 16)))
    if kind == "odd":
        return _scan("train", rng.randint(1, 4), _log(rng, 100, 2048) | 1, _log(rng, 100, 2048) | 1, A=A, dt=dt)
    if kind == "state":
        return _scan("train", rng.randint(1, 2), _log(rng, 128, 2048), _width(rng, 256, 2560), N=rng.choice((32, 64)),
                     A=A)
    if kind == "complex":
        return _scan("train", rng.randint(1, 2), _log(rng, 128, 2048), _width(rng, 128, 1536),
                     N=rng.choice((8, 16, 16)), io=rng.choice(("bf16", "f32")), complex=True)
    return {"op": "conv", "batch": rng.randint(1, 8), "L": _log(rng, 64, 4096), "D": _width(rng, 512, 5120),
            "width": rng.choice((2, 3, 4, 4)), "io": rng.choice(("bf16", "bf16", "f32"))}


def prepare(case, seed):
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    io = _IO[case["io"]]
    batch, L, D = case["batch"], case["L"], case["D"]

    def normal(*shape, dtype=io, scale=1.0):
        return torch.randn(*shape, generator=g, device="cuda", dtype=dtype if scale == 1.0 else torch.float32).mul(scale).to(dtype)

    if case["op"] == "conv":
        return {"op": "conv", "x": normal(batch, L, D), "dy": normal(batch, L, D),
                "w": normal(D, case["width"], dtype=torch.float32, scale=case["width"] ** -0.5),
                "bias": normal(D, dtype=torch.float32, scale=0.1)}

    N, c2 = case["N"], (2,) if case["complex"] else ()
    s = {"op": case["op"], "fused": case["dt"] == "fused", "complex": case["complex"], "h0": None}
    rows = (batch, D) if case["op"] == "step" else (batch, L, D)
    s["x"], s["z"] = normal(*rows), normal(*rows)
    s["B"], s["C"] = (normal(*rows[:-1], N, *c2) for _ in range(2))
    lo, hi = math.log(case["dt_min"]), math.log(case["dt_max"])
    tau = torch.rand(D, generator=g, device="cuda").mul(hi - lo).add(lo).exp()
    bias = tau + torch.log(-torch.expm1(-tau))
    u = normal(*rows, scale=0.1)
    if s["fused"]:
        s["delta"], s["bias"] = u, bias
    else:
        s["delta"] = torch.nn.functional.softplus(u.float().add_(bias)).to(io)
    n = torch.arange(N, device="cuda", dtype=torch.float32)
    if case["complex"]:
        s["A"] = torch.stack((torch.full_like(n, -0.5), math.pi * n), -1).repeat(D, 1, 1)
    else:
        s["A"] = -(n + 1).repeat(D, 1)
        if case["A"] == "trained":
            s["A"] *= normal(D, N, dtype=torch.float32, scale=0.1).exp()
    s["D_skip"] = torch.ones(D, device="cuda")
    if case["op"] == "train":
        s["dout"] = normal(*rows)
    elif case["op"] == "step":
        s["h"] = normal(batch, D, N, *c2, dtype=torch.float32)
    elif case["chunk"]:
        s["h0"] = normal(batch, D, N, dtype=torch.float32)
    return s


def run(s):
    if s["op"] == "conv":
        y = K.ssm_conv1d_fwd(s["x"], s["w"], s["bias"])
        return {"y": y, **K.ssm_conv1d_bwd(s["x"], s["w"], s["bias"], s["dy"])}
    if s["op"] == "step":
        out = K.ssm_step(s["x"], s["delta"], s["A"], s["B"], s["C"], s["D_skip"], s["z"], s["h"])
        return {"out": out, "h": s["h"]}
    if s["op"] == "prefill":
        batch, _, D = s["x"].shape
        h_last = torch.empty(batch, D, s["A"].shape[1], device="cuda")
        if s["fused"]:
            out = K.ssm_scan_fwd_fused_dt(s["x"], s["delta"], s["bias"], s["A"], s["B"], s["C"], s["D_skip"], s["z"],
                                          h0=s["h0"], h_last=h_last)
        else:
            out = K.ssm_scan_fwd(s["x"], s["delta"], s["A"], s["B"], s["C"], s["D_skip"], s["z"], h0=s["h0"],
                                 h_last=h_last)
        return {"out": out, "h_last": h_last}
    if s["fused"]:
        args = (s["x"], s["delta"], s["bias"], s["A"], s["B"], s["C"], s["D_skip"], s["z"])
        out, saved = K.ssm_scan_fwd_fused_dt(*args, save_states=True)
        return {"out": out, **K.ssm_scan_bwd_fused_dt(*args, s["dout"], saved)}
    args = (s["x"], s["delta"], s["A"], s["B"], s["C"], s["D_skip"], s["z"])
    out, saved = K.ssm_scan_fwd(*args, save_states=True, complex_state=s["complex"])
    return {"out": out, **K.ssm_scan_bwd(*args, s["dout"], saved, complex_state=s["complex"])}


def work(case):
    """Each input read once, each output written once.  Operations: a multiply-add counts as two, an exponential as
    one; per state and step 7 forward (decay 2, input term 1, recurrence 2, readout 2) and 27 backward (the states
    rebuilt 5, the adjoint and its decay 3, the seven sums and products of the gradients); a complex state four times
    that.  The gate, the skip term and the other per-channel work are 12 forward and 24 backward."""
    e = 2 if case["io"] == "bf16" else 4
    batch, L, D = case["batch"], case["L"], case["D"]
    elements = batch * L * D
    if case["op"] == "conv":
        W = case["width"]
        return {"bytes": 4 * e * elements + 8 * D * (W + 1), "flops": elements * (8 * W + 14)}
    N, c = case["N"], 2 if case["complex"] else 1
    fwd, bwd = N * 7 * c * c + 12, N * 27 * c * c + 24
    rows, params, state = 2 * e * batch * L * N * c, 4 * D * (N * c + 1), 4 * batch * D * N * c
    if case["op"] == "train":
        return {"bytes": 8 * e * elements + 2 * rows + 2 * params, "flops": elements * (fwd + bwd)}
    states = 2 if case["op"] == "step" or case["chunk"] else 1
    return {"bytes": 4 * e * elements + rows + params + states * state, "flops": elements * fwd}


def tolerance(case):
    """bf16: one rounding of each result (2^-9), now and then the other neighbour; float32: sums in another order and
    exponentials of 2 ulp."""
    return {"rel": 5e-3, "max": 3e-2} if case["io"] == "bf16" else {"rel": 2e-5, "max": 1e-3}
