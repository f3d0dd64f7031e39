"""The adjoint pre-pass of the tuned backward walks every segment in two pieces: pieces at the edges of a tile, a last
piece that is short or empty, an adjoint that arrives from outside."""
import numpy as np
import pytest

from paper_2312_00752_b200 import synth
from tests import _gpu_util as U

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch,L,D,zoh", [
    (10, 545, 2048, False),   # two segments of 288 and 257 steps, pieces of 160
    (1, 1281, 64, True),      # five segments (the ZOH rule keeps to the tuned kernels): the last piece is empty
    (1, 1030, 40, True),      # four segments: 6 steps in the last piece, half a channel group
    (2, 512, 32, True),       # two segments of 256, pieces of 128
    (1, 2304, 32, True),      # nine segments: the carry of many segments
])
def test_against_the_oracle(batch, L, D, zoh):
    import torch
    from oracle import ssm_oracle as O
    from paper_2312_00752_b200 import binding as K
    inp = synth.make_inputs(synth.ScanConfig("pieces", 23, batch, L, D, 16, "bf16", 1e-3, 1e-2), seed=L)
    rng = np.random.default_rng(L)
    h0, dh = (rng.standard_normal((batch, D, 16)).astype(np.float32) for _ in range(2))
    dev = U.to_device(inp, "bf16")
    th0, tdh = torch.from_numpy(h0).cuda(), torch.from_numpy(dh).cuda()
    args = (dev["x"], dev["delta"], dev["A"], dev["B"], dev["C"], dev["D_skip"], dev["z"])
    ref = O.scan_bwd(inp["x"], inp["delta"], inp["A"], inp["B"], inp["C"], inp["D_skip"], inp["z"], inp["dout"], zoh=zoh,
                     h0=h0, dh_last=dh)
    _, saved = K.ssm_scan_fwd(*args, save_states=True, h0=th0, zoh=zoh)
    g = K.ssm_scan_bwd(*args, dev["dout"], saved, h0=th0, dh_last=tdh, want_dh0=True, zoh=zoh)
    for k in ("dx", "ddelta", "dz", "dB", "dC", "dA", "dD", "dh0"):
        assert U.rel_err(U.to_host(g[k]), ref[k]) <= U.TOL["bf16"]["grad"], k
