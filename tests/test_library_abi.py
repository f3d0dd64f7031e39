"""Host-only checks of the C-ABI library: it loads, exports every declared symbol, and validates arguments before
launching anything (no GPU needed: every call here returns before a CUDA call is made)."""
import ctypes
import os
import re

import pytest

from paper_2312_00752_b200 import binding as K

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _declared_symbols():
    import glob
    text = "".join(open(h).read() for h in sorted(glob.glob(os.path.join(ROOT, "include", "*.h"))))
    return sorted(set(re.findall(r"SSM_API[^;(]*?\b(ssm_\w+)\s*\(", text)))


def test_library_exports_every_declared_symbol():
    lib = K.load_library()
    names = _declared_symbols()
    assert set(names) == set(K.EXPORTED_SYMBOLS) and len(names) >= 8
    for n in names:
        assert getattr(lib, n) is not None


def _prob(batch=2, L=100, D=64, N=16, io=K.SSM_BF16, flags=3):
    return K.ssm_problem_t(batch, L, D, N, io, flags)


def test_queries_and_plan():
    ck = K.checkpoint_steps()
    assert ck in (8, 16, 32, 64)
    p = _prob(4, 2048, 5120)
    assert K.saved_state_bytes(p) == 4 * (2048 // ck) * 5120 * 16 * 4
    pl = K.plan(p)
    assert pl["n_segments"] == 1 and pl["segment_steps"] == 2048 and pl["states_per_thread"] in (4, 8, 16)
    # 640 groups of 32 channels for 592 resident warps: some groups are shared by two warps, which needs hand-off slots
    assert 0 < K.fwd_workspace_bytes(p) < 4 << 20
    assert K.fwd_workspace_bytes(_prob(64, 256, 64)) == 0 and K.fwd_workspace_bytes(_prob(2, 100, 64, io=K.SSM_F32)) == 0
    assert K.bwd_workspace_bytes(p) > 0
    long = _prob(1, 524288, 1536)
    pl = K.plan(long)
    assert pl["n_segments"] > 1 and pl["segment_steps"] % ck == 0
    assert pl["n_segments"] * pl["segment_steps"] >= 524288 > (pl["n_segments"] - 1) * pl["segment_steps"]
    assert K.fwd_workspace_bytes(long) >= 2 * pl["n_segments"] * 1536 * 16 * 4


@pytest.mark.parametrize("flags,batch,L,D,split", [
    # groups of 32 channels on 0.51 to 0.70 of the 592 sub-partitions; four segments only where they were measured shorter
    (0, 8, 2048, 1536, True), (0, 8, 1024, 1536, False), (0, 8, 2048, 1664, False), (32, 8, 1024, 1536, True),
    (64, 8, 2048, 1440, True), (64, 8, 2048, 1536, False), (64, 10, 1024, 960, True), (64, 8, 1024, 1344, False),
    (64, 8, 4096, 1536, True), (64, 8, 4096, 1664, False), (64, 10, 768, 960, False),
    (96, 8, 1024, 1344, True), (96, 8, 1024, 1440, False), (96, 8, 2048, 1536, False), (96, 8, 4096, 1792, False),
    (256, 8, 2048, 1536, True), (512, 8, 2048, 1536, True),
    (768, 8, 2048, 1440, True), (768, 10, 1024, 960, False), (768, 8, 4096, 1664, False), (800, 8, 1024, 1536, True), (800, 8, 4096, 1792, False),
])
def test_time_segments_of_the_tuned_forward_by_choice(flags, batch, L, D, split):
    for save in (0, K.SSM_FLAG_SAVE_STATES):
        assert K.plan(_prob(batch, L, D, flags=3 | flags | save))["n_segments"] == (4 if split else 1)


@pytest.mark.parametrize("batch,L,D,N", [(9, 4402, 592, 2), (17, 5238, 320, 2), (33, 4439, 200, 1), (2, 100, 64, 8)])
def test_the_host_arena_holds_the_last_piece_where_it_needs_more(batch, L, D, N):
    # pieces of 2, 3 and 5 batch entries and a last one of 1, 2 and 3, which is widened to 16 states where the others are not
    piece = -(-batch // 8)
    sizes = [_prob(b, L, D, N, flags=7) for b in {piece, batch - (-(-batch // piece) - 1) * piece}]
    buffers = 4 * (4 * piece * L * D * 2 + 2 * piece * L * N * 2)      # inputs and outputs, both twice
    arena = K.load_library().ssm_scan_host_arena_bytes(ctypes.byref(_prob(batch, L, D, N)))
    assert arena >= buffers + max(map(K.saved_state_bytes, sizes)) + max(map(K.bwd_workspace_bytes, sizes))


@pytest.mark.parametrize("bad,code", [
    (dict(N=3), 2), (dict(N=128), 2), (dict(io=5), 2), (dict(L=0), 1), (dict(batch=-1), 1), (dict(flags=1 << 12), 1),
])
def test_invalid_problems_are_rejected(bad, code):
    lib = K.load_library()
    p = _prob(**bad)
    assert lib.ssm_scan_plan(ctypes.byref(p), None, None, None, None) == code
    assert K.fwd_workspace_bytes(p) == 0 and K.bwd_workspace_bytes(p) == 0
    one = ctypes.c_void_p(256)
    assert lib.ssm_scan_fwd(ctypes.byref(p), one, one, one, one, one, one, one, one, None, None, 0, None) == code


def test_complex_state_queries_and_refused_combinations():
    lib = K.load_library()
    real = _prob(2, 100, 64, N=8, io=K.SSM_F32, flags=3)
    cplx = _prob(2, 100, 64, N=8, io=K.SSM_F32, flags=3 | K.SSM_FLAG_COMPLEX)
    assert K.saved_state_bytes(cplx) == 2 * K.saved_state_bytes(real)        # (re, im) pairs
    assert K.fwd_workspace_bytes(cplx) == 0 and K.bwd_workspace_bytes(cplx) > 0
    assert K.plan(_prob(1, 524288, 64, N=8, flags=3 | K.SSM_FLAG_COMPLEX))["n_segments"] == 1   # no time split
    for extra in (K.SSM_FLAG_ZOH_BBAR, K.SSM_FLAG_STATIC_B, K.SSM_FLAG_STATIC_C, K.SSM_FLAG_DELTA_SOFTPLUS):
        bad = _prob(2, 100, 64, N=8, flags=3 | K.SSM_FLAG_COMPLEX | extra)
        assert lib.ssm_scan_plan(ctypes.byref(bad), None, None, None, None) == 2
    assert lib.ssm_scan_plan(ctypes.byref(_prob(2, 100, 64, N=64, flags=3 | K.SSM_FLAG_COMPLEX)), None, None, None, None) == 2


def test_the_backward_plan_of_a_complex_state_is_the_one_that_runs():
    p = _prob(2, 1237, 1001, N=8, flags=3 | K.SSM_FLAG_COMPLEX)
    pl, wide = K.bwd_plan(p), K.bwd_plan(_prob(2, 1237, 1001, N=16))     # (8 complex states are 16 columns)
    assert pl == wide and pl["n_segments"] > 1 and pl["n_segments"] * pl["segment_steps"] >= 1237
    one = _prob(2, 64, 1001, N=8, flags=3 | K.SSM_FLAG_COMPLEX)
    assert K.bwd_plan(one)["n_segments"] == 1
    # what leaves a segment (16 rows and a sum of step sizes for 32 groups of 32 channels) lies in the workspace
    assert K.bwd_workspace_bytes(p) > 2 * pl["n_segments"] * 32 * 32 * 17 * 4


def test_null_misaligned_and_workspace_errors_before_launch():
    lib = K.load_library()
    p = _prob()
    a = ctypes.c_void_p(4096)
    args = [a] * 8
    assert lib.ssm_scan_fwd(ctypes.byref(p), None, *args[1:], None, None, 0, None) == 1          # x missing
    assert lib.ssm_scan_fwd(ctypes.byref(p), *args[:6], None, a, None, None, 0, None) == 1       # z flagged, missing
    assert lib.ssm_scan_fwd(ctypes.byref(p), ctypes.c_void_p(4097), *args[1:], None, None, 0, None) == 1  # misaligned
    ps = _prob(flags=7)
    assert lib.ssm_scan_fwd(ctypes.byref(ps), *args, None, None, 0, None) == 1                   # saved_states missing
    long = _prob(1, 524288, 1536)
    assert lib.ssm_scan_fwd(ctypes.byref(long), *args, None, None, 0, None) == 3                 # workspace missing
    assert lib.ssm_scan_fwd(ctypes.byref(long), *args, None, a, 16, None) == 3                   # workspace too small
    b16 = [a] * 16
    assert lib.ssm_scan_bwd(ctypes.byref(p), *b16, None, 0, None) == 3
    assert lib.ssm_scan_bwd(ctypes.byref(p), *b16[:7], None, *b16[8:], None, 0, None) == 1       # dout missing
    assert "WORKSPACE" in K.status_string(3) and K.status_string(0) == "SSM_OK"


def test_conv1d_argument_errors_before_launch():
    lib = K.load_library()
    a = ctypes.c_void_p(4096)
    ok = K.ssm_conv_problem_t(2, 100, 64, 4, K.SSM_BF16, 3)
    assert lib.ssm_conv1d_fwd(ctypes.byref(ok), None, a, a, None, a, None) == 1                  # x missing
    assert lib.ssm_conv1d_fwd(ctypes.byref(ok), a, a, None, None, a, None) == 1                  # bias flagged, missing
    for bad, code in [(dict(width=5), 2), (dict(width=0), 2), (dict(io=7), 2), (dict(L=0), 1), (dict(flags=8), 1)]:
        f = dict(batch=2, L=100, D=64, width=4, io=K.SSM_BF16, flags=3)
        f.update(bad)
        p = K.ssm_conv_problem_t(f["batch"], f["L"], f["D"], f["width"], f["io"], f["flags"])
        assert lib.ssm_conv1d_fwd(ctypes.byref(p), a, a, a, None, a, None) == code
        assert lib.ssm_conv1d_bwd_workspace_bytes(ctypes.byref(p)) == 0
    need = lib.ssm_conv1d_bwd_workspace_bytes(ctypes.byref(ok))
    assert need == 2 * 4 * 64 * 5 * 4                                                            # room for 4 chunks of 32 steps
    assert lib.ssm_conv1d_bwd(ctypes.byref(ok), a, a, a, None, a, a, a, a, None, None, 0, None) == 3
    assert lib.ssm_conv1d_bwd(ctypes.byref(ok), a, a, a, None, a, a, a, a, None, a, need - 1, None) == 3
