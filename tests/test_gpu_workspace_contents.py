"""The contents of a workspace are undefined between calls: whatever lies where the status word and the hand-off flags go,
a call clears what it uses before it uses it."""
import pytest

from paper_2312_00752_b200 import synth
from tests import _gpu_util as U

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch,L,D,N", [
    # backward on the lane kernels, its checkpoints rebuilt by the tuned forward with chains shared between warps, which
    # give up waiting for each other once they find the status word set
    (1, 8192, 704, 16),
    (2, 8192, 320, 16),
    (1, 8192, 704, 8),      # the same through the widened arrays
    (1, 2048, 256, 16),     # lane kernels in both directions
    (1, 700, 9536, 16),     # tuned kernels in both directions
])
def test_backward_without_saved_states_in_a_dirty_workspace(batch, L, D, N):
    import torch
    from paper_2312_00752_b200 import binding as K
    inp = synth.make_inputs(synth.ScanConfig("dirty", 27, batch, L, D, N, "bf16", 1e-3, 1e-1), seed=L + D)
    dev = U.to_device(inp, "bf16")
    args = (dev["x"], dev["delta"], dev["A"], dev["B"], dev["C"], dev["D_skip"], dev["z"])
    prob = K.make_problem(dev["x"], dev["B"], True, True)
    ref = U.oracle_fwd_bwd(inp)
    ws = torch.ones(K.bwd_workspace_bytes(prob) // 4 + 1, dtype=torch.int32, device="cuda")
    fws = torch.ones(max(K.fwd_workspace_bytes(prob) // 4, 1), dtype=torch.int32, device="cuda")
    out = K.ssm_scan_fwd(*args, workspace=fws)
    g = K.ssm_scan_bwd(*args, dev["dout"], None, workspace=ws)
    K.check_status(prob, ws)
    got = {"out": U.to_host(out), **{k: U.to_host(v) for k, v in g.items()}}
    U.assert_parity(got, ref, "bf16", f"{(batch, L, D, N)}, workspace full of ones")
