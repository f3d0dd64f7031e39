"""The lane-per-channel kernels (float32 io, any D, N > 16 or N < 16) against the oracle at the edges of their batches of
8 steps, channel groups of 32, pieces of the time split inside a cluster and segments of the launch."""
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
    (2, 707, 1001, 16, "bf16"),    # backward split into segments with a pre-pass: odd rows, ragged last segment
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
