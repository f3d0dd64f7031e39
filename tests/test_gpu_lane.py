"""The lane-per-channel kernels (float32 io, any D, N > 16 or N < 16) against the oracle at the edges of their batches of
8 steps, channel groups of 32, pieces of the time split inside a cluster and segments of the launch."""
import numpy as np
import pytest

from paper_2312_00752_b200 import synth
from tests import _gpu_util as U

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch,L,D,N,io", [
    (1, 1, 1, 16, "f32"),          # one step of one channel
    (1, 8, 33, 16, "bf16"),        # one batch, one channel in the second group
    (1, 9, 31, 16, "bf16"),        # one step past a batch, one channel short of a group
    (2, 63, 36, 16, "f32"),        # 16-byte rows, partial group, one step short of 8 pieces of 8
    (1, 65, 34, 16, "f32"),        # rows not 16-byte aligned, one step past 8 pieces of 8
    (3, 257, 70, 1, "f32"),
    (1, 100, 40, 2, "f32"),
    (1, 131, 12, 4, "bf16"),
    (2, 200, 8, 8, "f32"),
    (1, 90, 24, 32, "bf16"),       # two and four groups of 16 states
    (1, 75, 17, 64, "f32"),
    (5, 40, 2048, 16, "f32"),      # more chains than SM sub-partitions: several chains per block, no split
    (1, 4133, 20, 16, "f32"),      # the launch itself split in time (summary and carry)
    (1, 4100, 33, 64, "bf16"),
    (2, 707, 1001, 16, "bf16"),    # odd rows, several pieces per chain (segments with a pre-pass: test_gpu_kernel_routes.py)
    (1, 650, 1300, 32, "f32"),
])
def test_edges(batch, L, D, N, io):
    cfg = synth.ScanConfig("lane", 21, batch, L, D, N, io, 1e-3, 1e-1)
    inp = synth.make_inputs(cfg, seed=L)
    dev = U.to_device(inp, io)
    ref = U.oracle_fwd_bwd(inp)
    for use_saved in (True, False):
        got = U.gpu_fwd_bwd(dev, use_saved=use_saved)
        U.assert_parity(got, ref, io, f"{(batch, L, D, N, io)} saved={use_saved}")
        if io == "bf16":
            U.assert_elementwise(got, ref, io, f"{(batch, L, D, N, io)} saved={use_saved}")


@pytest.mark.parametrize("batch,L,D,N", [
    (1, 37, 9440, 16),     # 295 chains: the last count that takes the lane kernels
    (1, 37, 9464, 16),     # 296: the first that does not
    (1, 1, 8, 16),
    (2, 333, 72, 16),
    (1, 1500, 256, 16),    # cut in time inside clusters
    (1, 200, 1536, 4),     # N < 16 without widened arrays
    (3, 70, 3200, 8),      # 300 chains: widened
])
def test_few_channels_of_the_tuned_shapes(batch, L, D, N):
    """Both sides of the choice between the lane and the tuned kernels, with everything that rides along: the fused step
    size, a state that arrives, an adjoint that arrives, saved and rebuilt checkpoints."""
    import torch
    from oracle import ssm_oracle as O
    from paper_2312_00752_b200 import binding as K
    inp = synth.make_inputs(synth.ScanConfig("lane", 22, batch, L, D, N, "bf16", 1e-3, 1e-1), seed=L)
    rng = np.random.default_rng(L)
    inp["delta"] = synth.round_to_io(0.1 * rng.standard_normal((batch, L, D)), "bf16")
    bias, h0, dh = (rng.standard_normal(s).astype(np.float32) for s in ((D,), (batch, D, N), (batch, D, N)))
    bias = 0.5 * bias - 4.0
    dev = U.to_device(inp, "bf16")
    tb, th0, tdh = (torch.from_numpy(v).cuda() for v in (bias, h0, dh))
    h_last = torch.empty_like(th0)
    args = (dev["x"], dev["delta"], tb, dev["A"], dev["B"], dev["C"], dev["D_skip"], dev["z"])
    kw = dict(delta_softplus=True, delta_bias=bias, h0=h0)
    ref_out, ref_h = O.scan_fwd(inp["x"], inp["delta"], inp["A"], inp["B"], inp["C"], inp["D_skip"], inp["z"],
                                return_h_last=True, **kw)
    ref = O.scan_bwd(inp["x"], inp["delta"], inp["A"], inp["B"], inp["C"], inp["D_skip"], inp["z"], inp["dout"],
                     dh_last=dh, **kw)
    out, saved = K.ssm_scan_fwd_fused_dt(*args, save_states=True, h0=th0, h_last=h_last)
    assert U.rel_err(U.to_host(out), ref_out) <= U.TOL["bf16"]["out"]
    assert U.rel_err(U.to_host(h_last), ref_h) <= 1e-4
    for sv in (saved, None):
        g = K.ssm_scan_bwd_fused_dt(*args, dev["dout"], sv, h0=th0, dh_last=tdh, want_dh0=True)
        for k in ("dx", "ddelta", "ddelta_bias", "dz", "dB", "dC", "dA", "dD", "dh0"):
            assert U.rel_err(U.to_host(g[k]), ref[k]) <= U.TOL["bf16"]["grad"], (k, sv is None)


@pytest.mark.parametrize("batch,L,D,N,io", [
    (1, 9, 33, 16, "bf16"),        # one step past a batch, one channel in the second group
    (1, 63, 36, 1, "f32"),         # 16-byte rows, one step short of 8 pieces of 8
    (2, 65, 31, 8, "f32"),         # one group of 16 columns, rows at odd addresses
    (1, 520, 17, 32, "bf16"),      # four groups of 16 columns
    (1, 4133, 20, 16, "f32"),      # forward cut inside clusters, backward into segments
    (2, 707, 1001, 8, "bf16"),     # odd rows, several pieces per chain
    (2, 1237, 1001, 8, "bf16"),    # backward split into segments with a pre-pass, ragged last segment
])
def test_complex_edges(batch, L, D, N, io):
    from oracle import ssm_oracle_complex as OC
    from paper_2312_00752_b200 import binding as K
    from tests.test_gpu_complex import _c, _case, _cerr, _dev
    inp = _case(batch, L, D, N, io)
    dev = _dev(inp, io)
    args = (dev["x"], dev["delta"], dev["A"], dev["B"], dev["C"], dev["D_skip"], dev["z"])
    host = (inp["x"], inp["delta"], inp["A"], inp["B"], inp["C"], inp["D_skip"], inp["z"])
    ref_out, ref = OC.scan_fwd(*host), OC.scan_bwd(*host, inp["dout"])
    out, saved = K.ssm_scan_fwd(*args, save_states=True, complex_state=True)
    assert U.rel_err(U.to_host(out), ref_out) <= U.TOL[io]["out"]
    for sv in (saved, None):
        g = K.ssm_scan_bwd(*args, dev["dout"], sv, complex_state=True)
        for k in ("dx", "ddelta", "dz", "dD"):
            assert U.rel_err(U.to_host(g[k]), ref[k]) <= U.TOL[io]["grad"], (k, sv is None)
        for k in ("dA", "dB", "dC"):
            assert _cerr(_c(g[k]), ref[k]) <= U.TOL[io]["grad"], (k, sv is None)


@pytest.mark.parametrize("which", ["x", "B"])
@pytest.mark.parametrize("batch,L,D,N,io", [
    (1, 33, 40, 16, "f32"),        # one step in the last batch of 8
    (1, 33, 41, 16, "bf16"),       # odd width
    (2, 61, 17, 64, "bf16"),       # four groups of states
    (1, 299, 24, 4, "f32"),        # cut in time
    (1, 33, 9480, 16, "bf16"),     # the tuned kernels
    (1, 33, 2568, 64, "bf16"),     # teams of warps
    (2, 75, 2568, 64, "bf16"),     # ... that share chains
])
def test_an_infinite_input_of_the_last_step_stays_infinite(batch, L, D, N, io, which):
    """Rows past the end of a ragged batch are identity steps: zero times what they hold must not make NaN of the state."""
    import torch
    from paper_2312_00752_b200 import binding as K
    dev = U.to_device(synth.make_inputs(synth.ScanConfig("inf", 31, batch, L, D, N, io, 1e-3, 1e-1), seed=L), io)
    dev["x"][:, -1].abs_().clamp_(min=0.5)
    dev["B"][:, -1].abs_().clamp_(min=0.5)
    args = lambda: (dev["x"], dev["delta"], dev["A"], dev["B"], dev["C"], dev["D_skip"], dev["z"])
    h_last = torch.empty(batch, D, N, device="cuda")
    before = K.ssm_scan_fwd(*args())
    dev[which] = dev[which].clone()
    dev[which][:, -1] = float("inf")
    out = K.ssm_scan_fwd(*args(), h_last=h_last)
    assert bool((h_last == float("inf")).all())
    assert torch.equal(out[:, :-1], before[:, :-1])
