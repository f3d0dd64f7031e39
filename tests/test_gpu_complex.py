"""Complex-valued state (SSM_FLAG_COMPLEX; Section 3.6, S4D-Lin initialisation A_n = -1/2 + n i) on the GPU against
the complex oracle: forward, backward (saved and rebuilt checkpoints), the carried state, the single recurrent step
and the backward in two pieces, for both io dtypes and every supported N."""
import numpy as np
import pytest

from paper_2312_00752_b200 import synth
from tests import _gpu_util as U

pytestmark = pytest.mark.gpu


def _case(batch, L, D, N, io, dt=(1e-3, 1e-1), seed=0):
    """Real tensors from the shared generator; complex B, C drawn here (N(0,1) real and imaginary parts) and rounded
    to the io dtype like the others; A is the S4D-Lin initialisation."""
    import torch
    cfg = synth.ScanConfig("complex", 16, batch, L, D, N, io, dt[0], dt[1])
    inp = synth.make_inputs(cfg, seed=seed)
    rng = np.random.default_rng([seed, batch, L, D, N])
    def rounded(a):
        t = torch.from_numpy(a.astype(np.float32))
        return (t.to(torch.bfloat16).to(torch.float32) if io == "bf16" else t).numpy()
    for k in ("B", "C"):
        ri = rounded(rng.standard_normal((batch, L, N, 2)))
        inp[k + "_ri"] = ri
        inp[k] = ri[..., 0].astype(np.float64) + 1j * ri[..., 1].astype(np.float64)
    A_ri = np.empty((D, N, 2), dtype=np.float32)
    A_ri[..., 0] = -0.5
    A_ri[..., 1] = np.arange(N, dtype=np.float32)[None, :]
    inp["A_ri"] = A_ri
    inp["A"] = A_ri[..., 0].astype(np.float64) + 1j * A_ri[..., 1].astype(np.float64)
    return inp


def _dev(inp, io):
    import torch
    dt = torch.float32 if io == "f32" else torch.bfloat16
    d = {k: torch.from_numpy(np.ascontiguousarray(inp[k])).cuda().to(dt) for k in ("x", "delta", "z", "dout")}
    d["B"] = torch.from_numpy(inp["B_ri"]).cuda().to(dt)
    d["C"] = torch.from_numpy(inp["C_ri"]).cuda().to(dt)
    d["A"] = torch.from_numpy(inp["A_ri"]).cuda()
    d["D_skip"] = torch.from_numpy(inp["D_skip"]).cuda()
    return d


def _c(t):
    a = U.to_host(t).astype(np.float64)
    return a[..., 0] + 1j * a[..., 1]


def _cerr(got, ref):
    denom = np.abs(ref).max()
    return float(np.abs(got - ref).max() / denom) if denom > 0 else float(np.abs(got).max())


@pytest.mark.parametrize("batch,L,D,N,io", [
    (2, 100, 40, 16, "f32"),      # ragged time tail, channel tail inside a block
    (2, 100, 40, 16, "bf16"),
    (1, 257, 24, 8, "f32"),
    (2, 65, 7, 4, "bf16"),        # odd channel count
    (1, 130, 33, 2, "f32"),
    (2, 64, 70, 1, "bf16"),
    (1, 200, 20, 32, "f32"),      # 16-channel blocks
    (1, 1, 8, 16, "f32"),         # a single step
    (1, 1500, 16, 16, "f32"),     # many tiles: the phase of exp(delta A) accumulates over the sequence
])
def test_forward_backward(batch, L, D, N, io):
    from oracle import ssm_oracle_complex as OC
    from paper_2312_00752_b200 import binding as K
    inp = _case(batch, L, D, N, io)
    dev = _dev(inp, io)
    args = (dev["x"], dev["delta"], dev["A"], dev["B"], dev["C"], dev["D_skip"], dev["z"])
    ref_out = OC.scan_fwd(inp["x"], inp["delta"], inp["A"], inp["B"], inp["C"], inp["D_skip"], inp["z"])
    ref = OC.scan_bwd(inp["x"], inp["delta"], inp["A"], inp["B"], inp["C"], inp["D_skip"], inp["z"], inp["dout"])
    tol = U.TOL[io]
    out, saved = K.ssm_scan_fwd(*args, save_states=True, complex_state=True)
    assert U.rel_err(U.to_host(out), ref_out) <= tol["out"]
    for sv in (saved, None):
        g = K.ssm_scan_bwd(*args, dev["dout"], sv, complex_state=True)
        for k in ("dx", "ddelta", "dz", "dD"):
            assert U.rel_err(U.to_host(g[k]), ref[k]) <= tol["grad"], (k, sv is None)
        for k in ("dA", "dB", "dC"):
            assert _cerr(_c(g[k]), ref[k]) <= tol["grad"], (k, sv is None)
    # bitwise reproducible
    ga = K.ssm_scan_bwd(*args, dev["dout"], saved, complex_state=True)
    gb = K.ssm_scan_bwd(*args, dev["dout"], saved, complex_state=True)
    for k in ("dx", "ddelta", "dB", "dC", "dA"):
        assert np.array_equal(U.to_host(ga[k]), U.to_host(gb[k])), k


def test_without_gate_and_skip():
    from oracle import ssm_oracle_complex as OC
    from paper_2312_00752_b200 import binding as K
    inp = _case(2, 90, 24, 8, "f32")
    dev = _dev(inp, "f32")
    args = (dev["x"], dev["delta"], dev["A"], dev["B"], dev["C"], None, None)
    ref_out = OC.scan_fwd(inp["x"], inp["delta"], inp["A"], inp["B"], inp["C"])
    ref = OC.scan_bwd(inp["x"], inp["delta"], inp["A"], inp["B"], inp["C"], None, None, inp["dout"])
    out = K.ssm_scan_fwd(*args, complex_state=True)
    g = K.ssm_scan_bwd(*args, dev["dout"], None, complex_state=True)
    assert g["dz"] is None and g["dD"] is None
    assert U.rel_err(U.to_host(out), ref_out) <= 1e-5
    for k in ("dx", "ddelta"):
        assert U.rel_err(U.to_host(g[k]), ref[k]) <= 1e-4, k
    for k in ("dA", "dB", "dC"):
        assert _cerr(_c(g[k]), ref[k]) <= 1e-4, k


@pytest.mark.parametrize("N,io", [(16, "f32"), (4, "bf16")])
def test_step_by_step_equals_scan(N, io):
    import torch
    from oracle import ssm_oracle_complex as OC
    from paper_2312_00752_b200 import binding as K
    batch, T, D = 2, 24, 24
    inp = _case(batch, T, D, N, io)
    dev = _dev(inp, io)
    ref_out, ref_h = OC.scan_fwd(inp["x"], inp["delta"], inp["A"], inp["B"], inp["C"], inp["D_skip"], inp["z"],
                                 return_h_last=True)
    h = torch.zeros((batch, D, N, 2), dtype=torch.float32, device="cuda")
    outs = []
    for t in range(T):
        outs.append(K.ssm_step(dev["x"][:, t].contiguous(), dev["delta"][:, t].contiguous(), dev["A"],
                               dev["B"][:, t].contiguous(), dev["C"][:, t].contiguous(), dev["D_skip"],
                               dev["z"][:, t].contiguous(), h, complex_state=True))
    got = np.stack([U.to_host(o) for o in outs], axis=1)
    assert U.rel_err(got, ref_out) <= U.TOL[io]["out"]
    assert _cerr(_c(h), ref_h) <= 1e-5


@pytest.mark.parametrize("N,io,L,cut", [(16, "f32", 150, 70), (8, "bf16", 300, 128)])
def test_two_pieces_with_carried_state_and_adjoint(N, io, L, cut):
    import torch
    from oracle import ssm_oracle_complex as OC
    from paper_2312_00752_b200 import binding as K
    batch, D = 2, 24
    inp = _case(batch, L, D, N, io)
    dev = _dev(inp, io)
    ref_out = OC.scan_fwd(inp["x"], inp["delta"], inp["A"], inp["B"], inp["C"], inp["D_skip"], inp["z"])
    ref = OC.scan_bwd(inp["x"], inp["delta"], inp["A"], inp["B"], inp["C"], inp["D_skip"], inp["z"], inp["dout"])
    sl = lambda k, a, b: dev[k][:, a:b].contiguous()
    piece = lambda a, b: (sl("x", a, b), sl("delta", a, b), dev["A"], sl("B", a, b), sl("C", a, b), dev["D_skip"],
                          sl("z", a, b))
    h_mid = torch.empty((batch, D, N, 2), dtype=torch.float32, device="cuda")
    o1, sv1 = K.ssm_scan_fwd(*piece(0, cut), save_states=True, h_last=h_mid, complex_state=True)
    o2, sv2 = K.ssm_scan_fwd(*piece(cut, L), save_states=True, h0=h_mid, complex_state=True)
    got = np.concatenate([U.to_host(o1), U.to_host(o2)], axis=1)
    assert U.rel_err(got, ref_out) <= U.TOL[io]["out"]
    g2 = K.ssm_scan_bwd(*piece(cut, L), sl("dout", cut, L), sv2, h0=h_mid, want_dh0=True, complex_state=True)
    g1 = K.ssm_scan_bwd(*piece(0, cut), sl("dout", 0, cut), sv1, dh_last=g2["dh0"], complex_state=True)
    tol = U.TOL[io]["grad"]
    for k in ("dx", "ddelta", "dz"):
        assert U.rel_err(np.concatenate([U.to_host(g1[k]), U.to_host(g2[k])], axis=1), ref[k]) <= tol, k
    for k in ("dB", "dC"):
        assert _cerr(np.concatenate([_c(g1[k]), _c(g2[k])], axis=1), ref[k]) <= tol, k
    assert _cerr(_c(g1["dA"]) + _c(g2["dA"]), ref["dA"]) <= tol
    assert U.rel_err(U.to_host(g1["dD"]) + U.to_host(g2["dD"]), ref["dD"]) <= tol


def test_options_that_do_not_combine_are_refused():
    import torch
    from paper_2312_00752_b200 import binding as K
    inp = _case(1, 16, 8, 4, "f32")
    dev = _dev(inp, "f32")
    args = (dev["x"], dev["delta"], dev["A"], dev["B"], dev["C"], dev["D_skip"], dev["z"])
    with pytest.raises(K.SsmScanError):
        K.ssm_scan_fwd(*args, zoh=True, complex_state=True)


@pytest.mark.parametrize("batch,L,D,im,split", [
    (8, 512, 2400, 5000.0, False),   # 600 chains: the forward does not split time; a step turns the state up to 90 times
    (1, 2048, 64, 50.0, True),       # two chains of 32 pieces of 64 steps: the fold turns it by whole pieces
])
def test_the_phase_of_an_undamped_state(batch, L, D, im, split):
    """Re A = 0, no input: h_last = exp(A sum delta) h0 and dh0 = exp(conj(A) sum delta) dh_last.  A step is off by the
    sine's and cosine's absolute error, at most 2^-21.2 each (CUDA's table of intrinsics, angles within half a turn), hence
    sqrt(2) times that and the number of steps if the errors all had one sign; where time is split, a state goes through
    the steps of one piece and then through sums of step sizes, each rounded once, which counts 2^-25 with the radians
    that the sum stands for.  No rounding of A or of a product delta A may come on top: in the first case the state turns
    by some 1e5 rad, so that 2^-25 of those would be 3e-3."""
    import torch
    from paper_2312_00752_b200 import binding as K
    g = torch.Generator("cuda").manual_seed(3)
    n = lambda *s: torch.randn(*s, generator=g, device="cuda")
    u = lambda *s: torch.rand(*s, generator=g, device="cuda")
    x = torch.zeros(batch, L, D, device="cuda")
    delta = (u(D) * np.log(10.0) + np.log(0.01)).exp() * (1 + 0.2 * u(batch, L, D))
    A = torch.stack((torch.zeros(D, 8, device="cuda"), im * u(D, 8)), -1).contiguous()
    B, C, h0, dh = n(batch, L, 8, 2), n(batch, L, 8, 2), n(batch, D, 8, 2), n(batch, D, 8, 2)
    h_last = torch.empty_like(h0)
    K.ssm_scan_fwd(x, delta, A, B, C, complex_state=True, h0=h0, h_last=h_last)
    dh0 = K.ssm_scan_bwd(x, delta, A, B, C, None, None, x, None, complex_state=True, h0=h0, dh_last=dh, want_dh0=True)["dh0"]
    angle = A[..., 1].double() * delta.double().sum(1)[:, :, None]
    turn = torch.polar(torch.ones_like(angle), angle)
    c = lambda v: torch.view_as_complex(v.double())
    err = lambda v, ref: float((c(v) - ref).norm() / ref.norm())
    step, sums = 2 ** 0.5 * 2 ** -21.2, float(angle.pow(2).mean().sqrt()) * 2 ** -25
    assert err(h_last, turn * c(h0)) <= (64 * step + sums if split else L * step)
    assert err(dh0, turn.conj() * c(dh)) <= (64 if split else L) * step + sums
