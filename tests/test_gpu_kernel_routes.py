"""Which kernels a problem runs, and their results: the tuned kernels want bf16, N = 16 (or fewer, widened), aligned
pointers and at least 296 chains of 32 channels (or the zero-order-hold rule); small problems of the same kind run the
lane kernels, so what is to be tested of the tuned ones is wide here.  Every case asserts the route."""
import os
import re

import numpy as np
import pytest

from paper_2312_00752_b200 import synth
from tests import _gpu_util as U

pytestmark = pytest.mark.gpu

TUNED = ("ssm_fwd_warp_kernel", "ssm_bwd_warp_kernel")
LANE = ("ssm_fwd_lane_kernel", "ssm_bwd_lane_kernel")
GENERIC = ("ssm_fwd_kernel", "ssm_bwd_kernel")
TEAM = "ssm_fwd_team_kernel"   # forward of 32 or 64 states
# template arguments: summary pass of the tuned forward, its sweeps with output and with checkpoints only; rolled lane backward
SUMMARY, FULL, CKPT = (r"ssm_fwd_warp_kernelILi16ELi%dE" % mode for mode in (1, 0, 2))
ROLLED, UNROLLED = (r"ssm_bwd_lane_kernelI(f|13__nv_bfloat16)Li1ELi\dELb0ELb%dEE" % rolled for rolled in (1, 0))


def _shifted(t):
    """The same values at an address 8 bytes past a 16-byte boundary."""
    import torch
    buf = torch.empty(t.numel() + 8, dtype=t.dtype, device=t.device)
    off = 8 // t.element_size()
    v = buf[off:off + t.numel()].view(t.shape)
    v.copy_(t)
    assert v.data_ptr() % 16 == 8
    return v


def _no_workspace(buf):
    """An empty and a misaligned piece of a buffer (the bounds-checking build wants a status word of every call)."""
    return [] if os.environ.get("SSM_SCAN_LIBRARY", "").endswith("_debug.so") else [buf[:0], buf[128:]]


def _check(batch, L, D, N=16, io="bf16", *, fwd=TUNED[0], bwd=TUNED[1], more=(), gate=True, skip=True, zoh=False, fused=False,
           carry=False, saved=True, perturb_A=0.0, A=None, dt=(1e-3, 1e-1), off=(), instances=()):
    import torch
    from oracle import ssm_oracle as O
    from paper_2312_00752_b200 import binding as K
    inp = synth.make_inputs(synth.ScanConfig("routes", 29, batch, L, D, N, io, *dt), seed=L, perturb_A=perturb_A)
    rng = np.random.default_rng(L + N)
    if A is not None:
        inp["A"] = np.tile(np.asarray(A, dtype=np.float32), (D, 1))
    if not gate:
        inp["z"] = None
    if not skip:
        inp["D_skip"] = None
    kw, okw, bias = dict(zoh=zoh), dict(zoh=zoh), None
    if fused:
        inp["delta"] = synth.round_to_io(0.1 * rng.standard_normal((batch, L, D)), io)
        bias = (0.5 * rng.standard_normal(D) - 4.0).astype(np.float32)
        okw.update(delta_softplus=True, delta_bias=bias)
    state = (batch, D, N)
    h0, dh = (rng.standard_normal(state).astype(np.float32) for _ in range(2)) if carry else (None, None)
    t = lambda a: None if a is None else torch.from_numpy(a).cuda()
    dev = U.to_device(inp, io)
    x_fwd, x_bwd = (_shifted(dev["x"]) if k in off else dev["x"] for k in ("fwd", "bwd"))
    h_last = torch.empty(state, device="cuda")
    bkw = dict(h0=t(h0), dh_last=t(dh), want_dh0=True, **kw)
    fkw = dict(save_states=True, h0=t(h0), h_last=h_last, **kw)
    rest = (dev["A"], dev["B"], dev["C"], dev["D_skip"], dev["z"])
    tb = t(bias)

    def run():
        if fused:
            f = lambda x: (x, dev["delta"], tb, *rest)
            out, sv = K.ssm_scan_fwd_fused_dt(*f(x_fwd), **fkw)
            return dict(K.ssm_scan_bwd_fused_dt(*f(x_bwd), dev["dout"], sv if saved else None, **bkw), out=out)
        f = lambda x: (x, dev["delta"], *rest)
        out, sv = K.ssm_scan_fwd(*f(x_fwd), **fkw)
        return dict(K.ssm_scan_bwd(*f(x_bwd), dev["dout"], sv if saved else None, **bkw), out=out)
    got = run()
    K.check_status(K.make_problem(dev["x"], dev["B"], gate, skip, zoh=zoh), K.last_bwd_workspace("cuda"))
    ran = U.kernels(run)
    assert {k for k in ran if k in (*TUNED, *LANE, *GENERIC, TEAM)} == {fwd, bwd}, ran
    assert all(any(k.startswith(m) for k in ran) for m in more), ran
    ran = U.kernels(run, arguments=True)
    assert all(any(re.match(m, k) for k in ran) for m in instances), ran
    a = (inp["x"], inp["delta"], inp["A"], inp["B"], inp["C"])
    out, h = O.scan_fwd(*a, D_skip=inp["D_skip"], z=inp["z"], h0=h0, return_h_last=True, **okw)
    ref = dict(O.scan_bwd(*a, inp["D_skip"], inp["z"], inp["dout"], h0=h0, dh_last=dh, **okw), out=out)
    host = {k: U.to_host(v) for k, v in got.items() if v is not None}
    assert U.rel_err(U.to_host(h_last), h) <= (1e-5 if io == "f32" else 1e-4)
    U.assert_parity(host, {k: v for k, v in ref.items() if k in host}, io, "route")
    if io == "bf16":
        U.assert_elementwise(host, ref, io, "route")


@pytest.mark.parametrize("batch,L,D", [
    (1, 1, 9480),       # a single step; 296 whole groups of 32 channels and one of 8
    (2, 31, 4744),      # one step short of a tile
    (1, 33, 9544),      # one step past one, a last group of 8
    (4, 64, 2560),      # whole tiles and groups: the instantiations without range tests
    (2, 512, 4736),     # ... with the backward in two segments
    (1, 600, 9480),     # two ragged segments
    (2, 96, 9984),      # 624 chains for 592 warps in the first round: some are shared
])
@pytest.mark.parametrize("fused", [False, True])
def test_tuned_kernels_at_the_edges_of_tiles_groups_and_segments(batch, L, D, fused):
    more = ("ssm_bwd_local_warp_kernel", "ssm_carry") if L >= 512 else ()
    _check(batch, L, D, fused=fused, carry=fused, more=more)


@pytest.mark.parametrize("batch,L,D,options", [
    (2, 1024, 4736, {}),                                  # whole tiles and segments
    (2, 1030, 4744, dict(carry=True, perturb_A=0.05)),    # ragged tile, group and last segment
    (2, 1030, 4744, dict(saved=False)),                   # the states rebuilt by the split forward
    (2, 409, 4744, dict(fused=True, carry=True)),         # a last segment of 25 steps, less than a tile
    (2, 416, 4736, dict(fused=True, saved=False)),        # ... of one tile
])
def test_tuned_forward_split_in_time_with_more_than_half_the_sub_partitions(batch, L, D, options):
    instances = (SUMMARY, FULL) if options.get("saved", True) else (SUMMARY, FULL, CKPT)
    _check(batch, L, D, more=("ssm_carry",), instances=instances, **options)


@pytest.mark.parametrize("batch,L,D,carry", [(2, 1024, 4736, "ssm_carry_few_kernel"), (1, 16384, 1536, "ssm_carry_kernel")])
@pytest.mark.parametrize("which", ["x", "h0"])
def test_an_infinite_state_stays_infinite_across_time_segments(batch, L, D, carry, which):
    # the decay over a whole segment is zero in float32 for the fast states of many channels, that of a step is not
    import torch
    from paper_2312_00752_b200 import binding as K
    dev = U.to_device(synth.make_inputs(synth.ScanConfig("inf", 31, batch, L, D, 16, "bf16", 1e-3, 1e-1), seed=L), "bf16")
    h0, h_last = torch.zeros(batch, D, 16, device="cuda"), torch.empty(batch, D, 16, device="cuda")
    if which == "x":
        dev["x"][:, 100] = float("inf")
        dev["B"][:, 100].abs_().clamp_(min=0.5)
    else:
        h0.fill_(float("-inf"))
    run = lambda: K.ssm_scan_fwd(dev["x"], dev["delta"], dev["A"], dev["B"], dev["C"], dev["D_skip"], dev["z"], h0=h0, h_last=h_last)
    run()
    assert carry in U.kernels(run)
    assert bool((h_last == float("inf" if which == "x" else "-inf")).all())


def test_chains_of_the_tuned_kernels_nearly_one_per_warp():
    # 1136 chains for two rounds of 592 warps: the forward shares them among 1184, the backward leaves them whole
    _check(8, 40, 4544, instances=(FULL + r"\w+<<<296", r"ssm_bwd_warp_kernel\w+<<<284"))


@pytest.mark.parametrize("options", [dict(zoh=True), dict(static_B=True), dict(static_C=True), dict(static_B=True, static_C=True)])
@pytest.mark.parametrize("fused", [False, True])
def test_tuned_forward_split_in_time_by_the_other_rules(options, fused):
    # the zero-order hold, parameters B and C: four segments (a ragged last one, from a carried state) against one piece on the
    # generic kernel, which runs what is off the 16-byte grid
    import torch
    from paper_2312_00752_b200 import binding as K
    batch, L, D = 2, 1150, 4744
    dev = U.to_device(synth.make_inputs(synth.ScanConfig("routes", 29, batch, L, D, 16, "bf16", 1e-3, 1e-1), seed=L, perturb_A=0.05), "bf16")
    rng = torch.Generator(device="cuda").manual_seed(1)
    for name in "BC":
        if options.get("static_" + name):
            dev[name] = torch.randn(D, 16, generator=rng, device="cuda")
    h0 = torch.randn(batch, D, 16, generator=rng, device="cuda")
    bias = (torch.full((D,), -4.0, device="cuda"),) if fused else ()
    fwd = K.ssm_scan_fwd_fused_dt if fused else K.ssm_scan_fwd

    def run(x):
        h_last = torch.empty(batch, D, 16, device="cuda")
        out = fwd(x, dev["delta"], *bias, dev["A"], dev["B"], dev["C"], dev["D_skip"], dev["z"], h0=h0, h_last=h_last, **options)
        return out, h_last
    shifted = _shifted(dev["x"])
    (out, h), (ref_out, ref_h) = run(dev["x"]), run(shifted)
    assert "ssm_carry_few_kernel" in U.kernels(lambda: run(dev["x"])) and U.kernels(lambda: run(shifted)) == {GENERIC[0]}
    U.assert_elementwise({"out": U.to_host(out)}, {"out": U.to_host(ref_out)}, "bf16", "segments")
    assert U.rel_err(U.to_host(h), U.to_host(ref_h)) <= 1e-4


@pytest.mark.parametrize("options", [
    dict(gate=False), dict(skip=False), dict(gate=False, skip=False), dict(carry=True), dict(carry=True, saved=False),
    dict(perturb_A=0.05), dict(perturb_A=0.05, fused=True, saved=False), dict(fused=True, gate=False, carry=True),
], ids=lambda o: "-".join(f"{k}={v}" for k, v in o.items()))
@pytest.mark.parametrize("batch,L,D", [(1, 150, 9480), (4, 64, 2560)])   # ragged; whole
def test_options_on_the_tuned_kernels(batch, L, D, options):
    _check(batch, L, D, **options)


def test_tuned_forward_takes_the_unsplit_plan_where_the_split_one_has_no_room():
    # the fixed scratch of the static entry holds nothing of this split (8 MB), and the problem needs none without it
    import torch
    from oracle import ssm_oracle as O
    from paper_2312_00752_b200 import binding as K
    inp = synth.make_inputs(synth.ScanConfig("routes", 29, 2, 1024, 4736, 16, "bf16", 1e-3, 1e-1), seed=5)
    dev = U.to_device(inp, "bf16")
    args = (dev["x"], dev["delta"], dev["A"], dev["B"], dev["C"], dev["D_skip"], dev["z"])
    assert K.fwd_workspace_bytes(K.make_problem(dev["x"], dev["B"], True, True)) > 4 << 20
    out = torch.empty_like(dev["x"])
    got = K.ssm_scan_fwd_static(*args, out=out)
    got = got[0] if isinstance(got, tuple) else got
    ref = {"out": O.scan_fwd(inp["x"], inp["delta"], inp["A"], inp["B"], inp["C"], D_skip=inp["D_skip"], z=inp["z"])}
    U.assert_elementwise({"out": U.to_host(got)}, ref, "bf16", "static scratch")
    assert U.kernels(lambda: K.ssm_scan_fwd_static(*args, out=out)) == {TUNED[0]}


@pytest.mark.parametrize("batch,L,D,N", [(2, 1024, 4736, 16), (2, 1030, 4744, 16), (2, 1024, 4736, 8)])
def test_forward_results_depend_on_the_workspace_only_by_whether_the_split_has_room(batch, L, D, N):
    # what include/ssm_scan.h says of it: short, missing and misaligned workspaces and the fixed scratch give one result, bit
    # for bit, and one sweep; every workspace that has room gives another, bit for bit, and the split
    import torch
    from oracle import ssm_oracle as O
    from paper_2312_00752_b200 import binding as K
    inp = synth.make_inputs(synth.ScanConfig("routes", 29, batch, L, D, N, "bf16", 1e-3, 1e-1), seed=L)
    dev = U.to_device(inp, "bf16")
    args = (dev["x"], dev["delta"], dev["A"], dev["B"], dev["C"], dev["D_skip"], dev["z"])
    prob = K.make_problem(dev["x"], dev["B"], True, True)
    need = K.fwd_workspace_bytes(prob)
    assert K.plan(prob)["n_segments"] == 4 and need > K.SSM_STATIC_SCRATCH_BYTES
    big = torch.full((need + 256,), 255, dtype=torch.uint8, device="cuda")
    split = K.ssm_scan_fwd(*args)
    assert torch.equal(K.ssm_scan_fwd(*args, workspace=big[:need]), split)
    assert torch.equal(K.ssm_scan_fwd(*args, workspace=big), split)
    short = [big[:need - 1]]
    if N == 16:   # (N = 8 needs a workspace in any case)
        short += [big[:256], *_no_workspace(big)]
        assert torch.equal(K.ssm_scan_fwd_static(*args), K.ssm_scan_fwd(*args, workspace=short[0]))
    one = K.ssm_scan_fwd(*args, workspace=short[0])
    for ws in short[1:]:
        assert torch.equal(K.ssm_scan_fwd(*args, workspace=ws), one)
    assert "ssm_carry_few_kernel" in U.kernels(lambda: K.ssm_scan_fwd(*args, workspace=big))
    assert not any(k.startswith("ssm_carry") for k in U.kernels(lambda: K.ssm_scan_fwd(*args, workspace=short[0])))
    ref = {"out": O.scan_fwd(inp["x"], inp["delta"], inp["A"], inp["B"], inp["C"], D_skip=inp["D_skip"], z=inp["z"])}
    for out in (split, one):
        U.assert_elementwise({"out": U.to_host(out)}, ref, "bf16", "workspace")


@pytest.mark.parametrize("batch,L,D,N", [(2, 75, 2568, 64), (2, 200, 5128, 32)])   # 162 chains for 148 teams, 322 for 296
def test_teams_of_warps_leave_together_when_a_hand_off_stays_away(batch, L, D, N):
    # no flag is published: the teams that continue a chain give up after 1000 polls, which the host reads from the status
    # word; the next call on that workspace is complete again
    import ctypes
    import torch
    from paper_2312_00752_b200 import binding as K
    dev = U.to_device(synth.make_inputs(synth.ScanConfig("routes", 29, batch, L, D, N, "bf16", 1e-3, 1e-1), seed=L), "bf16")
    args = (dev["x"], dev["delta"], dev["A"], dev["B"], dev["C"], dev["D_skip"], dev["z"])
    prob = K.make_problem(dev["x"], dev["B"], True, True)
    ws = torch.empty(K.fwd_workspace_bytes(prob), dtype=torch.uint8, device="cuda")
    good = K.ssm_scan_fwd(*args, workspace=ws)
    K.check_status(prob, ws)
    out = torch.empty_like(good)
    prob.flags |= K.SSM_FLAG_TEST_WITHHOLD
    code = K.load_library().ssm_scan_fwd(
        ctypes.byref(prob), *[ctypes.c_void_p(t.data_ptr()) for t in (*args, out)], None, ctypes.c_void_p(ws.data_ptr()),
        ctypes.c_size_t(ws.numel()), ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert code == K.SSM_OK
    with pytest.raises(K.SsmScanError, match="TIMEOUT"):
        K.check_status(prob, ws)
    assert torch.equal(K.ssm_scan_fwd(*args, workspace=ws), good)
    K.check_status(prob, ws)


@pytest.mark.parametrize("batch,L,D,N", [(2, 1024, 4736, 16), (2, 1024, 4736, 8), (2, 75, 2568, 64)])
def test_the_status_word_of_a_workspace_without_room_is_that_of_the_call(batch, L, D, N):
    import torch
    from paper_2312_00752_b200 import binding as K
    dev = U.to_device(synth.make_inputs(synth.ScanConfig("routes", 29, batch, L, D, N, "bf16", 1e-3, 1e-1), seed=L), "bf16")
    args = (dev["x"], dev["delta"], dev["A"], dev["B"], dev["C"], dev["D_skip"], dev["z"])
    prob = K.make_problem(dev["x"], dev["B"], True, True)
    need = K.fwd_workspace_bytes(prob)
    big = torch.full((need + 256,), 255, dtype=torch.uint8, device="cuda")
    for ws in [big[:need - 1], *([] if N == 8 else [big[:256], *_no_workspace(big)[1:]])]:   # (N = 8 needs some in any case)
        big.fill_(255)
        K.ssm_scan_fwd(*args, workspace=ws)
        K.check_status(prob, ws)


@pytest.mark.parametrize("batch,L,D,N", [(2, 1024, 4736, 16), (2, 1030, 4744, 8), (2, 75, 2568, 64)])
def test_backward_without_room_for_what_its_rebuilding_sweep_can_do_without(batch, L, D, N):
    # the time segments taken by choice (N <= 16), the hand-offs between teams: as the forward without them, bit for bit
    import torch
    from paper_2312_00752_b200 import binding as K
    dev = U.to_device(synth.make_inputs(synth.ScanConfig("routes", 29, batch, L, D, N, "bf16", 1e-3, 1e-1), seed=L), "bf16")
    args = (dev["x"], dev["delta"], dev["A"], dev["B"], dev["C"], dev["D_skip"], dev["z"])
    prob = K.make_problem(dev["x"], dev["B"], True, True)
    need, need_fwd = K.bwd_workspace_bytes(prob), K.fwd_workspace_bytes(prob)
    wide = K.ssm_problem_t(batch, L, D, max(N, 16), prob.io_dtype, prob.flags)
    least = need - K.fwd_workspace_bytes(wide) + 256   # (256: the status word that the bounds-checking build wants)
    big = torch.full((need,), 255, dtype=torch.uint8, device="cuda")
    big_fwd = torch.full((need_fwd,), 255, dtype=torch.uint8, device="cuda")
    assert least < need and need_fwd > 0

    def bwd(saved, ws):
        got = K.ssm_scan_bwd(*args, dev["dout"], saved, workspace=ws)
        K.check_status(prob, ws)
        return got

    def equal(a, b):
        assert all(torch.equal(a[k], b[k]) for k in U.GRADS)
    split = K.ssm_scan_fwd(*args, save_states=True, workspace=big_fwd)[1]
    whole = K.ssm_scan_fwd(*args, save_states=True, workspace=big_fwd[:need_fwd - 1])[1]
    equal(bwd(split, big[:least]), bwd(split, big))
    equal(bwd(None, big), bwd(split, big))
    equal(bwd(None, big[:least]), bwd(whole, big))
    with pytest.raises(K.SsmScanError):
        bwd(None, big[:least - 512])


@pytest.mark.parametrize("batch,L,D,N,io,options", [   # (backward in pieces of one block of 8 steps: up to 32 pieces per chain)
    (1, 1, 40, 16, "f32", dict(carry=True)),
    (1, 8, 31, 16, "bf16", {}),
    (1, 9, 64, 4, "f32", dict(saved=False)),
    (1, 255, 33, 16, "f32", dict(carry=True, perturb_A=0.05)),
    (1, 256, 64, 16, "f32", {}),
    (2, 249, 32, 16, "bf16", dict(carry=True, fused=True)),
    (1, 64, 100, 8, "f32", dict(gate=False, skip=False)),
    (2, 31, 47, 16, "bf16", dict(perturb_A=0.05, saved=False)),
])
def test_lane_kernels_in_pieces_of_one_block(batch, L, D, N, io, options):
    _check(batch, L, D, N, io, fwd=LANE[0], bwd=LANE[1], instances=(ROLLED,), **options)


@pytest.mark.parametrize("L,D,rolled", [
    (250, 256, True), (250, 288, False),     # clusters of 8: 8 and 9
    (100, 896, True), (100, 928, False),     # of 4: 28 and 29
    (64, 1792, True), (64, 1824, False),     # of 2: 56 and 57
    (32, 4736, True), (32, 4768, False),     # a block per chain: 148 and 149
])
def test_rolled_lane_backward_only_where_its_blocks_run_at_once(L, D, rolled):
    _check(1, L, D, 16, "f32", fwd=LANE[0], bwd=LANE[1], instances=(ROLLED if rolled else UNROLLED,))


@pytest.mark.parametrize("batch,L,D,N,options", [
    (1, 1, 2568, 64, {}),                                        # a single step; 80 whole groups of channels and one of 8
    (1, 31, 2560, 64, dict(carry=True)),                         # one step short of a tile
    (1, 33, 2568, 64, dict(perturb_A=0.05, gate=False)),         # one past it
    (2, 64, 1280, 64, dict(fused=True, skip=False)),             # whole tiles
    (2, 75, 2568, 64, dict(carry=True, fused=True)),             # 162 chains for 148 teams: some are shared, ragged tile
    (2, 160, 2560, 64, dict(perturb_A=0.05, saved=False)),       # ... whole; states rebuilt by the team kernel
    (3, 40, 2560, 64, dict(saved=False, carry=True)),
    (2, 70, 2568, 32, dict(carry=True)),                         # 162 chains, two teams per block, a block with one
    (2, 200, 5128, 32, dict(fused=True, carry=True, perturb_A=0.05)),   # 322 chains for 296 teams
    (2, 128, 5120, 32, dict(saved=False, gate=False, skip=False)),
])
def test_teams_of_warps_for_large_states(batch, L, D, N, options):
    _check(batch, L, D, N, fwd=TEAM, bwd=LANE[1], **options)


@pytest.mark.parametrize("batch,L,D,N", [(2, 75, 2568, 64), (2, 200, 5128, 32)])   # 162 chains for 148 teams, 322 for 296
def test_teams_of_warps_without_room_for_their_hand_offs(batch, L, D, N):
    import torch
    from paper_2312_00752_b200 import binding as K
    dev = U.to_device(synth.make_inputs(synth.ScanConfig("routes", 29, batch, L, D, N, "bf16", 1e-3, 1e-1), seed=L), "bf16")
    args = (dev["x"], dev["delta"], dev["A"], dev["B"], dev["C"], dev["D_skip"], dev["z"])
    need = K.fwd_workspace_bytes(K.make_problem(dev["x"], dev["B"], True, True))
    assert need > 0
    big = torch.full((need + 256,), 255, dtype=torch.uint8, device="cuda")

    def run(ws):
        h_last = torch.empty(batch, D, N, device="cuda")
        return (*K.ssm_scan_fwd(*args, save_states=True, h_last=h_last, workspace=ws), h_last)
    shared = run(big[:need])
    for ws in (big[:need - 1], big[:256], *_no_workspace(big)):
        assert all(torch.equal(a, b) for a, b in zip(run(ws), shared))
    assert all(TEAM in U.kernels(lambda: run(ws)) for ws in (big, big[:256]))


def test_large_states_off_the_16_byte_grid_and_of_few_channels_keep_the_lane_kernel():
    _check(1, 100, 2560, 64, fwd=LANE[0], bwd=LANE[1], off=("fwd",), carry=True)
    _check(1, 300, 64, 32, fwd=LANE[0], bwd=LANE[1])


@pytest.mark.parametrize("N", [1, 2, 4, 8])
@pytest.mark.parametrize("saved", [True, False])
def test_small_states_widened_for_the_tuned_kernels(N, saved):
    _check(1, 70, 9480, N, carry=True, saved=saved, more=("ssm_repack_kernel",))


@pytest.mark.parametrize("A", [(-4.0, -3.0, -2.0, -1.0), (-16.0, -15.0, -14.0, -13.0), (-0.7, -0.7, -0.7, -0.7), (-0.3, -2.0, -0.9, -4.0)])
def test_rows_of_A_widened_for_the_tuned_kernels(A):
    # a progression that would turn positive, one that only just would, step 0, no progression
    _check(1, 40, 9480, 4, A=A, more=("ssm_repack_kernel",))


@pytest.mark.parametrize("D,N,route", [(9480, 16, TUNED), (40, 16, (TUNED[0], LANE[1])), (41, 16, LANE), (41, 32, LANE),
                                       (2568, 64, (TEAM, LANE[1]))])
@pytest.mark.parametrize("saved", [True, False])
def test_rising_rows_of_A_with_large_steps(D, N, route, saved):
    # exp(delta A) of the first state is below the smallest float32, that of the last one is not
    _check(1, 40, D, N, A=np.arange(-16.0, 0.0).tolist() * (N // 16), dt=(8.0, 20.0), carry=True, saved=saved,
           fwd=route[0], bwd=route[1])


@pytest.mark.parametrize("off,fwd,bwd", [
    (("fwd",), LANE[0], TUNED[1]), (("bwd",), TUNED[0], LANE[1]), (("fwd", "bwd"), *LANE),
])
def test_pointers_off_the_16_byte_grid_and_states_passed_between_the_families(off, fwd, bwd):
    _check(2, 150, 4744, fwd=fwd, bwd=bwd, off=off)


def test_no_time_segments_by_choice_off_the_16_byte_grid():
    # the lane kernel runs these, which cuts a chain in time by itself
    import torch
    from paper_2312_00752_b200 import binding as K
    dev = U.to_device(synth.make_inputs(synth.ScanConfig("routes", 29, 2, 1030, 4744, 16, "bf16", 1e-3, 1e-1), seed=4), "bf16")
    rest = (dev["delta"], dev["A"], dev["B"], dev["C"], dev["D_skip"], dev["z"])
    x = _shifted(dev["x"])
    assert K.plan(K.make_problem(x, dev["B"], True, True))["n_segments"] == 4
    out = K.ssm_scan_fwd(x, *rest)
    U.assert_elementwise({"out": U.to_host(out)}, {"out": U.to_host(K.ssm_scan_fwd(dev["x"], *rest))}, "bf16", "off the grid")
    assert U.kernels(lambda: K.ssm_scan_fwd(x, *rest)) == {LANE[0]}
    ran = U.kernels(lambda: K.ssm_scan_bwd(x, *rest, dev["dout"], None))
    assert LANE[0] in ran and not any(k.startswith("ssm_carry") for k in ran), ran


def test_states_rebuilt_off_the_16_byte_grid():
    _check(2, 150, 4744, fwd=LANE[0], bwd=LANE[1], off=("fwd", "bwd"), saved=False)


@pytest.mark.parametrize("batch,L,D,N,io,more", [
    (2, 1237, 1001, 16, "bf16", ("ssm_bwd_lane_local_kernel",)),   # odd width, the backward in segments with a pre-pass
    (1, 2000, 1500, 16, "f32", ("ssm_bwd_lane_local_kernel",)),
    (1, 900, 1300, 64, "bf16", ("ssm_bwd_lane_local_kernel",)),
    (1, 4133, 20, 16, "f32", ("ssm_carry",)),                      # the launch split in time
    (2, 100, 40, 16, "bf16", ()),                                  # a tuned shape with few channels
])
def test_lane_kernels(batch, L, D, N, io, more):
    _check(batch, L, D, N, io, fwd=LANE[0], bwd=LANE[1], more=more)


@pytest.mark.parametrize("D,io,fwd,bwd,off", [
    (40, "bf16", *TUNED, ()), (41, "bf16", *GENERIC, ()), (40, "f32", *GENERIC, ()), (40, "bf16", *GENERIC, ("fwd", "bwd")),
])
def test_zero_order_hold_keeps_to_the_tuned_and_generic_kernels(D, io, fwd, bwd, off):
    _check(2, 150, D, 16, io, zoh=True, fwd=fwd, bwd=bwd, off=off)
