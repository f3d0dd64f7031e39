"""Runs small problems through whatever library SSM_SCAN_LIBRARY names (the bounds-checking build), compares with the oracle,
asserts that no index check fired and that the kernels ran that each problem is there for.  Executed as a child process by
test_gpu_debug_bounds.py, because a process loads only one build of the library."""
import sys

import numpy as np

FWD, BWD, LOCAL, CARRY = "ssm_fwd_warp_kernel", "ssm_bwd_warp_kernel", "ssm_bwd_local_warp_kernel", "ssm_carry"
TEAM_FWD = "ssm_fwd_team_kernel"
LANE_FWD, LANE_BWD, LANE_LOCAL = "ssm_fwd_lane_kernel", "ssm_bwd_lane_kernel", "ssm_bwd_lane_local_kernel"

CASES = [  # batch, L, D, N, io, ZOH, the kernels that have to run
    # ragged tiles, partial channel groups, one step, time splits in both directions
    (2, 300, 192, 16, "bf16", False, (LANE_FWD, LANE_BWD)),
    (1, 1, 64, 16, "bf16", False, ()),
    (3, 33, 72, 16, "bf16", False, ()),
    (1, 31, 8, 16, "bf16", False, ()),
    (2, 257, 40, 16, "bf16", False, ()),
    (1, 4096, 64, 16, "bf16", False, ()),
    (2, 1000, 1600, 16, "bf16", False, ()),
    (5, 515, 104, 16, "bf16", False, ()),
    # tuned kernels with the default rule: at least 296 chains of 32 channels
    (1, 70, 9480, 16, "bf16", False, (FWD, BWD)),                      # 297 chains, the last one of 8 channels
    (1, 600, 9480, 16, "bf16", False, (FWD, BWD, LOCAL, CARRY)),       # backward in two segments, ragged
    (2, 100, 9992, 16, "bf16", False, (FWD, BWD)),                     # 626 chains for 592 warps: some are shared
    (1, 96, 9600, 16, "bf16", False, (FWD, BWD)),                      # whole tiles and groups
    (1, 70, 9480, 8, "bf16", False, (FWD, BWD, "ssm_repack_kernel")),  # widened
    (1, 8192, 704, 16, "bf16", False, (FWD, CARRY, LANE_BWD, LANE_LOCAL)),   # both families in one pass
    # tuned kernels with the zero-order-hold rule: any number of chains
    (2, 1000, 200, 16, "bf16", True, (FWD, BWD, LOCAL, CARRY)),
    (1, 33, 72, 16, "bf16", True, (FWD, BWD)),
    # lane kernels
    (2, 63, 36, 16, "f32", False, (LANE_FWD, LANE_BWD)),
    (1, 65, 34, 16, "f32", False, (LANE_FWD, LANE_BWD)),               # rows not 16-byte aligned
    (1, 9, 31, 16, "bf16", False, (LANE_FWD, LANE_BWD)),
    (1, 50, 17, 2, "f32", False, (LANE_FWD, LANE_BWD)),                # checkpoints in the plain layout
    (1, 4133, 20, 16, "f32", False, (LANE_FWD, LANE_BWD, CARRY)),      # the launch itself split in time
    (2, 1237, 1001, 16, "bf16", False, (LANE_FWD, LANE_BWD, LANE_LOCAL)),
    (1, 650, 1300, 32, "f32", False, (LANE_FWD, LANE_BWD, LANE_LOCAL)),
    (1, 90, 24, 64, "bf16", False, (LANE_FWD, LANE_BWD)),
    # teams of warps: ragged tile and group, chains shared between teams
    (1, 70, 2568, 64, "bf16", False, (TEAM_FWD, LANE_BWD)),
    (2, 40, 2568, 64, "bf16", False, (TEAM_FWD, LANE_BWD)),
    (2, 96, 5128, 32, "bf16", False, (TEAM_FWD, LANE_BWD)),
]
COMPLEX = [  # batch, L, D, N, io, the kernels that have to run
    (1, 63, 36, 1, "f32", (LANE_FWD, LANE_BWD)),
    (2, 65, 31, 8, "f32", (LANE_FWD, LANE_BWD)),
    (1, 520, 17, 32, "bf16", (LANE_FWD, LANE_BWD)),
    (2, 1237, 1001, 8, "bf16", (LANE_FWD, LANE_BWD, LANE_LOCAL)),
]


def check(K, prob, dev):
    K.check_status(prob, K.last_bwd_workspace(dev["x"].device))     # raises SsmScanError on SSM_ERR_BOUNDS / _TIMEOUT


def expect(U, run, wanted, what):
    ran = U.kernels(run)
    assert all(any(k.startswith(w) for k in ran) for w in wanted), (what, ran)


def real(i, batch, L, D, N, io, zoh, wanted):
    import torch
    from oracle import ssm_oracle as O
    from paper_2312_00752_b200 import binding as K, synth
    from tests import _gpu_util as U
    what = f"bounds-checking build, {batch, L, D, N, io, zoh}"
    inp = synth.make_inputs(synth.ScanConfig("bounds", 1, batch, L, D, N, io, 1e-3, 1e-1), seed=20 + i,
                            perturb_A=0.05 if i % 2 else 0.0)
    dev = U.to_device(inp, io)
    args = (dev["x"], dev["delta"], dev["A"], dev["B"], dev["C"], dev["D_skip"], dev["z"])
    prob = K.make_problem(dev["x"], dev["B"], True, True, save_states=True, zoh=zoh)
    kw = dict(zoh=zoh)
    ref = {"out": O.scan_fwd(inp["x"], inp["delta"], inp["A"], inp["B"], inp["C"], inp["D_skip"], inp["z"], **kw),
           **O.scan_bwd(inp["x"], inp["delta"], inp["A"], inp["B"], inp["C"], inp["D_skip"], inp["z"], inp["dout"], **kw)}
    out, saved = K.ssm_scan_fwd(*args, save_states=True, **kw)
    check(K, prob, dev)
    for sv in (saved, None):
        g = K.ssm_scan_bwd(*args, dev["dout"], sv, **kw)
        check(K, prob, dev)
        got = {"out": U.to_host(out), **{k: U.to_host(v) for k, v in g.items() if v is not None}}
        U.assert_parity(got, ref, io, f"{what}, saved {sv is not None}")
    # the fused step size and a carried state and adjoint take other template instances of the same kernels
    bias = torch.linspace(-3.0, -1.0, D, device=dev["x"].device)
    h0, h_last = torch.ones(batch, D, N, device="cuda"), torch.empty(batch, D, N, device="cuda")
    fused = (dev["x"], dev["delta"], bias, *args[2:])
    K.ssm_scan_fwd_fused_dt(*fused, h0=h0, h_last=h_last, **kw)
    check(K, prob, dev)
    K.ssm_scan_bwd_fused_dt(*fused, dev["dout"], None, h0=h0, dh_last=h0, want_dh0=True, **kw)
    check(K, prob, dev)

    def run():
        K.ssm_scan_fwd(*args, **kw)
        K.ssm_scan_bwd(*args, dev["dout"], saved, **kw)
    expect(U, run, wanted, what)


def cplx(batch, L, D, N, io, wanted):
    import torch
    from oracle import ssm_oracle_complex as OC
    from paper_2312_00752_b200 import binding as K
    from tests import _gpu_util as U
    from tests.test_gpu_complex import _c, _case, _cerr, _dev
    what = f"bounds-checking build, complex {batch, L, D, N, io}"
    inp = _case(batch, L, D, N, io)
    dev = _dev(inp, io)
    args = (dev["x"], dev["delta"], dev["A"], dev["B"], dev["C"], dev["D_skip"], dev["z"])
    host = (inp["x"], inp["delta"], inp["A"], inp["B"], inp["C"], inp["D_skip"], inp["z"])
    prob = K.make_problem(dev["x"], dev["B"], True, True, save_states=True, complex_state=True)
    ref_out, ref = OC.scan_fwd(*host), OC.scan_bwd(*host, inp["dout"])
    h_last = torch.empty(batch, D, N, 2, device="cuda")
    out, saved = K.ssm_scan_fwd(*args, save_states=True, complex_state=True, h_last=h_last)
    check(K, prob, dev)
    assert U.rel_err(U.to_host(out), ref_out) <= U.TOL[io]["out"], what
    for sv in (saved, None):
        g = K.ssm_scan_bwd(*args, dev["dout"], sv, complex_state=True, want_dh0=True)
        check(K, prob, dev)
        for k in ("dx", "ddelta", "dz", "dD"):
            assert U.rel_err(U.to_host(g[k]), ref[k]) <= U.TOL[io]["grad"], (what, k)
        for k in ("dA", "dB", "dC"):
            assert _cerr(_c(g[k]), ref[k]) <= U.TOL[io]["grad"], (what, k)

    def run():
        K.ssm_scan_fwd(*args, complex_state=True)
        K.ssm_scan_bwd(*args, dev["dout"], saved, complex_state=True)
    expect(U, run, wanted, what)


def main() -> int:
    for i, case in enumerate(CASES):
        real(i, *case)
    for case in COMPLEX:
        cplx(*case)
    print("bounds-checking build: no index left its range on", len(CASES) + len(COMPLEX), "shapes")
    return 0


if __name__ == "__main__":
    sys.exit(main())
