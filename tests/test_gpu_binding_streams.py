"""The binding's scratch memory beside graphs and streams."""
import pytest

from paper_2312_00752_b200 import synth
from tests import _gpu_util as U

pytestmark = pytest.mark.gpu


def _call(L, D=64):
    from paper_2312_00752_b200 import binding as K
    dev = U.to_device(synth.make_inputs(synth.ScanConfig("streams", 30, 1, L, D, 16, "bf16", 1e-3, 1e-1), seed=L), "bf16")
    args = (dev["x"], dev["delta"], dev["A"], dev["B"], dev["C"], dev["D_skip"], dev["z"])
    return lambda **kw: K.ssm_scan_bwd(*args, dev["dout"], None, **kw)


def test_a_captured_call_does_not_use_the_buffer_that_is_kept_for_its_stream():
    # (that buffer is given back when a larger call comes along, the graph would go on writing to it)
    import torch
    from paper_2312_00752_b200 import binding as K
    run, larger = _call(300), _call(3000)
    torch.cuda.synchronize()
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        ref = run()
    kept = K.last_bwd_workspace("cuda", s)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s):
        got = run()
    torch.cuda.synchronize()
    kept.fill_(0x5a)
    graph.replay()
    torch.cuda.synchronize()
    assert bool((kept == 0x5a).all())
    assert all(torch.equal(got[k], ref[k]) for k in ref)
    with torch.cuda.stream(s):
        larger()
    assert K.last_bwd_workspace("cuda", s).numel() > kept.numel()
    for v in got.values():
        v.zero_()
    graph.replay()
    torch.cuda.synchronize()
    assert all(torch.equal(got[k], ref[k]) for k in ref)


def test_the_buffer_of_a_stream_is_a_block_of_that_stream():
    # (`stream` is not the current one: a block of the current stream may still be in use by its pending work, and would be
    # given back to it)
    import torch
    from paper_2312_00752_b200 import binding as K
    s = torch.cuda.Stream()
    run, ref = _call(400), _call(400)()
    torch.cuda.synchronize()
    got = run(stream=s)
    s.synchronize()
    assert all(torch.equal(got[k], ref[k]) for k in ref)
    at = K.last_bwd_workspace("cuda", s).data_ptr()
    owner = [seg["stream"] for seg in torch.cuda.memory_snapshot() if seg["address"] <= at < seg["address"] + seg["total_size"]]
    assert owner == [s.cuda_stream]


def test_a_result_that_is_dropped_is_not_handed_on_while_the_call_still_writes_to_it():
    import torch
    from paper_2312_00752_b200 import binding as K
    x = torch.randn(2, 500, 64, device="cuda")
    w = torch.randn(64, 4, device="cuda")
    s = torch.cuda.Stream()
    K.ssm_conv1d_fwd(x, w, stream=s)                 # (everything set up)
    run = _call(500)
    run(stream=s)
    torch.cuda.synchronize()
    with torch.cuda.stream(s):
        torch.cuda._sleep(200_000_000)               # the calls below wait behind this, a tenth of a second
    y = K.ssm_conv1d_fwd(x, w, stream=s)
    g = run(stream=s)
    gone = {t.data_ptr() for t in (y, *g.values()) if t is not None}
    shapes = [(t.shape, t.dtype) for t in (y, *g.values()) if t is not None]
    assert not s.query()
    del y, g
    new = [torch.empty(shape, dtype=dtype, device="cuda") for shape, dtype in shapes]
    assert not s.query() and not {t.data_ptr() for t in new} & gone
    torch.cuda.synchronize()
