"""The binding's calls in native code against the same calls marshalled in Python: the same fields, shapes, types and bits, the same
objects handed back, on the current stream and under capture; and what they leave to Python, errors included."""
import dataclasses

import pytest
import torch

from gpu_util import Guarded

pytestmark = pytest.mark.gpu


@pytest.fixture
def b(monkeypatch):
    from paper_2503_18339_b200 import binding
    binding.lib()
    assert binding._native is not None, "granq_host.cpp has not been built"
    monkeypatch.setattr(binding, "_new", binding._plain_new)      # guard bands are put around what Python allocates
    return binding


def flat(r):
    """name -> tensor of a record, a tuple or a tensor"""
    if isinstance(r, torch.Tensor):
        return {"": r}
    if isinstance(r, tuple):
        return {str(i): t for i, t in enumerate(r)}
    return {f.name: getattr(r, f.name) for f in dataclasses.fields(r) if getattr(r, f.name) is not None}


def both(b, monkeypatch, call, native=True, scratch=("workspace",)):
    """`call` twice, here and there; scratch is compared by its size only"""
    asked = []
    spy = lambda name: lambda *a: asked.append(getattr(b_native, name)(*a)) or asked[-1]
    b_native = b._native
    with monkeypatch.context() as m:
        m.setattr(b, "_native", type("Spy", (), {n: staticmethod(spy(n)) for n in dir(b_native) if n.endswith("_call")}))
        got = call()
    assert asked and (asked[-1] is not None) == native
    with monkeypatch.context() as m:
        m.setattr(b, "_native", None)
        want = call()
    assert type(got) is type(want)
    got, want = flat(got), flat(want)
    assert list(got) == list(want)
    for name, t in want.items():
        g = got[name]
        assert (g.shape, g.dtype, g.device, g.stride(), g.requires_grad) == (t.shape, t.dtype, t.device, t.stride(), False)
        if name not in scratch:
            plain = lambda v: v.as_subclass(torch.Tensor).view(torch.uint8)
            assert torch.equal(plain(g), plain(t)), name


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("shape,axis", [((3, 8, 5, 8), 1), ((6, 13, 7, 7), 1), ((4, 6, 6, 16), 3), ((1, 1, 1, 5), 1)])
def test_same_results(b, monkeypatch, dtype, shape, axis):
    torch.manual_seed(sum(shape))
    x, gy = torch.randn(shape, device="cuda").to(dtype), torch.randn(shape, device="cuda").to(dtype)
    for group in (b.GROUP_CHANNEL, b.GROUP_SAMPLE_CHANNEL, b.GROUP_TENSOR):
        how = dict(channel_axis=axis, group=group)
        run = lambda f, *a, **k: both(b, monkeypatch, lambda: f(*a, **how, **k), scratch=("workspace", "sums"))
        run(b.granq_range, x)
        for params in (False, True):
            run(b.granq_fakequant_fused, x, 4, want_params=params)
            run(b.granq_fakequant_fused, x, 4, gy=gy, want_params=params)
            run(b.granq_fakequant_fused_fwd_packmask, x, 3, want_params=params)
            run(b.granq_fakequant_fused_stats, x, 5, want_params=params)
            lo, hi = b.granq_range(x, **how)
            run(b.granq_fakequant_fwd_packmask, x, 4, lo, hi, want_params=params)
        run(b.granq_quantize_packed_fused, x, 5)
        q = b.granq_quantize_packed_fused(x, 5, **how)
        run(b.granq_dequantize_packed, q.packed_codes, x.shape, dtype, 5, q.s, q.z)
        run(b.granq_dequantize_packed, q.packed_codes, shape, dtype, 5, q.s, q.z, y=torch.empty_like(x))
    mask = b.granq_fakequant_fused_fwd_packmask(x, 4, channel_axis=axis).packed_mask
    both(b, monkeypatch, lambda: b.granq_fakequant_bwd_packmask(gy, mask))
    q = b.granq_quantize_packed_fused(x, 4, channel_axis=axis)
    w = torch.randn(24, shape[axis], device="cuda")
    both(b, monkeypatch, lambda: b.granq_accumulate_codes(q.packed_codes, x.shape, 4, q.s, q.z, w, channel_axis=axis), scratch=("1",))


def test_what_was_passed_comes_back(b):
    x = torch.randn(4, 8, 6, 6, device="cuda")
    gy = torch.randn_like(x)
    out = b.FakeQuantOut(y=torch.empty_like(x), lo=torch.empty(8, device="cuda"), workspace=b.make_workspace(x))
    y, lo, ws = out.y, out.lo, out.workspace
    got = b.granq_fakequant_fused(x, 4, gy=gy, out=out)
    assert got is out and got.y is y and got.lo is lo and got.workspace is ws and got.hi is not None and got.gx is not None
    lo, hi = torch.empty(8, device="cuda"), torch.empty(8, device="cuda")
    assert all(a is c for a, c in zip(b.granq_range(x, lo=lo, hi=hi), (lo, hi)))
    got = b.granq_fakequant_fwd_packmask(x, 4, lo, hi, y=y)
    assert got.lo is lo and got.hi is hi and got.y is y
    gx = torch.empty_like(x)
    assert b.granq_fakequant_bwd_packmask(gy, got.packed_mask, gx=gx) is gx
    codes = b.granq_quantize_packed_fused(x, 4)
    w = torch.randn(5, 8, device="cuda")
    acc, aws = b.granq_accumulate_codes(codes.packed_codes, x.shape, 4, codes.s, codes.z, w)
    again = b.granq_accumulate_codes(codes.packed_codes, x.shape, 4, codes.s, codes.z, w, y=acc, workspace=aws)
    assert again[0] is acc and again[1] is aws


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("shape,axis", [((3, 8, 5, 8), 1), ((9, 13, 7, 7), 1), ((40, 3, 4, 4), 1), ((4, 6, 6, 16), 3), ((1, 1, 1, 5), 1), ((5, 41, 27, 27), 1)])
def test_nothing_is_written_beside_the_outputs(b, monkeypatch, dtype, shape, axis):
    """Every output of every native call between guard bands, of the size that the binding would have made it."""
    asked = []
    native = b._native
    spy = lambda name: lambda *a: asked.append(getattr(native, name)(*a)) or asked[-1]
    monkeypatch.setattr(b, "_native", type("Spy", (), {n: staticmethod(spy(n)) for n in dir(native) if n.endswith("_call")}))
    torch.manual_seed(sum(shape))
    x, gy = torch.randn(shape, device="cuda").to(dtype), torch.randn(shape, device="cuda").to(dtype)
    guard = Guarded()
    for group in (b.GROUP_CHANNEL, b.GROUP_SAMPLE_CHANNEL, b.GROUP_TENSOR):
        G, how = b.num_groups(shape, axis, group), dict(channel_axis=axis, group=group)
        few = lambda: guard.empty((G,), torch.float32)
        work = lambda: guard.empty((b.workspace_bytes(b.F32 if dtype == torch.float32 else b.BF16, shape, axis, group),), torch.uint8)
        mask = lambda: guard.empty((b.packmask_bytes(shape) // 4,), torch.int32)
        like = lambda: guard.empty(shape, dtype)
        record = lambda **more: b.FakeQuantOut(lo=few(), hi=few(), s=few(), z=few(), workspace=work(), **more)
        b.granq_fakequant_fused(x, 4, gy=gy, out=record(y=like(), gx=like()), want_params=True, **how)
        b.granq_fakequant_fused(x, 4, out=record(y=like()), **how)
        m = b.granq_fakequant_fused_fwd_packmask(x, 3, out=record(y=like(), packed_mask=mask()), **how).packed_mask
        b.granq_fakequant_fused_stats(x, 5, out=record(y=like(), sums=guard.empty((4,), torch.float64)), **how)
        lo, hi = b.granq_range(x, lo=few(), hi=few(), workspace=work(), **how)
        b.granq_fakequant_fwd_packmask(x, 4, lo, hi, y=like(), packed_mask=mask(), **how)
        b.granq_fakequant_bwd_packmask(gy, m, gx=like())
        q = b.granq_quantize_packed_fused(x, 5, out=record(packed_codes=guard.empty((b.packed_codes_bytes(shape, 5) // 4,), torch.int32)), **how)
        b.granq_dequantize_packed(q.packed_codes, shape, dtype, 5, q.s, q.z, y=like(), **how)
        if group == b.GROUP_CHANNEL:
            out = tuple(24 if i == axis else d for i, d in enumerate(shape))
            b.granq_accumulate_codes(q.packed_codes, shape, 5, q.s, q.z, torch.randn(24, shape[axis], device="cuda"), channel_axis=axis,
                                     y=guard.empty(out, torch.float32),
                                     workspace=guard.empty((b.accumulate_workspace_bytes(shape, axis, 24),), torch.uint8))
    assert len(asked) == 3 * 9 + 1 and all(r is not None for r in asked)
    guard.check_and_release()


def test_what_is_left_to_python(b, monkeypatch):
    x = torch.randn(4, 8, 6, 6, device="cuda")
    both(b, monkeypatch, lambda: b.granq_fakequant_fused(x.as_subclass(type("Sub", (torch.Tensor,), {})), 4), native=False)
    for call, error in ((lambda: b.granq_fakequant_fused(x.transpose(2, 3), 4), ValueError),
                        (lambda: b.granq_fakequant_fused(x.cpu(), 4), ValueError),
                        (lambda: b.granq_fakequant_fused(x.double(), 4), TypeError),
                        (lambda: b.granq_fakequant_fused(x[0], 4), ValueError),
                        (lambda: b.granq_fakequant_fused(x, 4, gy=x[:2]), ValueError),
                        (lambda: b.granq_fakequant_fused(x, 4, gy=x.bfloat16()), ValueError),
                        (lambda: b.granq_fakequant_fused(x, 9), b.GranqError),
                        (lambda: b.granq_fakequant_fused(x, 4, out=b.FakeQuantOut(workspace=torch.empty(8, dtype=torch.uint8, device="cuda"))), b.GranqError),
                        (lambda: b.granq_range(x, channel_axis=7), ValueError),
                        (lambda: b.granq_fakequant_bwd_packmask(x, torch.zeros(1, dtype=torch.int32, device="cuda")), ValueError),
                        (lambda: b.granq_accumulate_codes(x, (4, 8, 6, 6), 4, x, x, torch.zeros(3, 9, device="cuda")), ValueError)):
        with pytest.raises(error) as here:
            call()
        with monkeypatch.context() as m:
            m.setattr(b, "_native", None)
            with pytest.raises(error) as there:
                call()
        assert str(here.value) == str(there.value)


def test_current_stream_and_capture(b):
    x = torch.randn(16, 32, 14, 14, device="cuda")
    want = b.granq_fakequant_fused(x, 4)
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        torch.cuda._sleep(1000000)
        y = torch.randn_like(x)
        got = b.granq_fakequant_fused(y.copy_(x), 4)        # behind the copy only on its own stream
    torch.cuda.current_stream().wait_stream(side)
    assert torch.equal(got.y, want.y)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        q = b.granq_quantize_packed_fused(x, 4)
        back = b.granq_dequantize_packed(q.packed_codes, x.shape, x.dtype, 4, q.s, q.z)
    back.zero_()
    graph.replay()
    assert torch.equal(back, want.y)
