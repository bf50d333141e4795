"""Calls on both sides of the size up to which a call outside a graph clears its workspace by a memset and a captured one by a
kernel: eager and captured, the workspace dirty before every run, the graph replayed on other inputs - against the CPU
oracle, bit for bit."""
import pytest
import torch

from gpu_util import assert_parity, make_case, same_bits, to_dev, to_np
from oracle import granq_oracle as orc
from test_parity_gpu import b  # noqa: F401

pytestmark = pytest.mark.gpu

# dims, channel axis, group mode: channels-last, ragged slabs, one group - below and above 400 000 elements
CASES = [
    ((10, 14, 14, 64), 3, 0), ((40, 14, 14, 64), 3, 0),
    ((8, 75, 5, 7), 1, 0), ((24, 75, 27, 27), 1, 0),
    ((16, 16, 32, 32), 1, 2), ((64, 16, 32, 32), 1, 2),
]


@pytest.mark.parametrize("shape,axis,mode", CASES, ids=lambda v: "x".join(map(str, v)) if isinstance(v, tuple) else str(v))
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_eager_and_captured_calls_clear_what_they_are_given(b, shape, axis, mode, dtype):
    cases = [make_case(shape, seed=21 + i, dtype=dtype) for i in range(2)]
    refs = [orc.fused(x, 4, gy=gy, channel_axis=axis, group_mode=mode) for x, gy in cases]
    inputs = [(to_dev(x), to_dev(gy)) for x, gy in cases]
    x, gy = (torch.empty_like(t) for t in inputs[0])
    ws = b.make_workspace(x, axis, mode)
    outs = [b.FakeQuantOut(y=torch.empty_like(x), gx=torch.empty_like(x), workspace=ws), b.FakeQuantOut(y=torch.empty_like(x), workspace=ws)]
    lo, hi = (torch.empty(refs[0].lo.shape, device="cuda") for _ in range(2))

    def step():
        ws.fill_(255)
        both = b.granq_fakequant_fused(x, 4, gy=gy, channel_axis=axis, group=mode, out=outs[0])
        ws.fill_(255)
        fwd = b.granq_fakequant_fused(x, 4, channel_axis=axis, group=mode, out=outs[1])
        ws.fill_(255)
        b.granq_range(x, channel_axis=axis, group=mode, lo=lo, hi=hi, workspace=ws)
        return both, fwd

    def check(results, ref):
        assert_parity(results[0], ref, shape, axis, mode, backward=True)
        assert_parity(results[1], ref, shape, axis, mode, backward=False)
        assert same_bits(to_np(lo), ref.lo) and same_bits(to_np(hi), ref.hi)

    def load(i):
        x.copy_(inputs[i][0])
        gy.copy_(inputs[i][1])

    load(0)
    check(step(), refs[0])
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        captured = step()
    for i in (1, 0):
        load(i)
        graph.replay()
        check(captured, refs[i])


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_captured_streaming_calls_of_a_size_that_states_its_layout(b, dtype):
    """Elementwise calls on 17 MB: captured and replayed on other inputs they give what the eager calls give, and the eager
    ones what the oracle does."""
    shape = (128, 33 if dtype == "f32" else 66, 32, 32)
    cases = [make_case(shape, seed=31 + i, dtype=dtype) for i in range(2)]
    inputs = [(to_dev(x), to_dev(gy)) for x, gy in cases]
    x, gy = (torch.empty_like(t) for t in inputs[0])
    lo, hi = torch.full((shape[1],), -1.5, device="cuda"), torch.full((shape[1],), 1.5, device="cuda")

    def step():
        fwd = b.granq_fakequant_fwd(x, 4, lo, hi)
        gx = b.granq_fakequant_bwd(gy, x, 4, lo, hi).gx
        half = b.granq_fakequant_fwd_packmask(x, 4, lo, hi)
        gm = b.granq_fakequant_bwd_packmask(gy, half.packed_mask)
        codes = b.granq_quantize_packed(x, 5, lo, hi)
        back = b.granq_dequantize_packed(codes.packed_codes, shape, x.dtype, 5, codes.s, codes.z)
        return fwd.y, gx, half.y, half.packed_mask, gm, codes.packed_codes, back

    eager = []
    for i in range(2):
        x.copy_(inputs[i][0])
        gy.copy_(inputs[i][1])
        eager.append([t.clone() for t in step()])
        ref = orc.fakequant(cases[i][0], 4, to_np(lo), to_np(hi), gy=cases[i][1])
        for t, want in zip(eager[i], (ref.y, ref.gx, ref.y, None, ref.gx)):
            assert want is None or same_bits(to_np(t), want)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        captured = step()
    for i in (1, 0):
        x.copy_(inputs[i][0])
        gy.copy_(inputs[i][1])
        graph.replay()
        for got, want in zip(captured, eager[i]):
            assert torch.equal(got, want)
