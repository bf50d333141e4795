"""The kernel that holds a tensor on chip piece by piece (planes and slabs that are not whole 16-byte units, one group over the
whole tensor) against the CPU oracle, bit for bit: pieces that begin and end inside planes, planes shorter than a thread's run
and longer than a piece, units that straddle two planes, fewer units than threads, one group that stays on chip and one of
which a part is read again - forward, with a gradient, with the distortion sums, packed
mask and packed codes; the workspace zero again afterwards."""
import numpy as np
import pytest
import torch

from gpu_util import assert_parity, make_case, to_dev, to_np
from oracle import granq_oracle as orc
from paper_2503_18339_b200 import workloads as wl
from test_parity_gpu import b, knobs  # noqa: F401
from test_rounding_gpu import assert_same_string

pytestmark = pytest.mark.gpu

# dims, group mode; the number of elements is a multiple of 8
CASES = [
    ((8, 3, 3, 3), 0),          # fewer units than one CTA has threads
    ((8, 75, 5, 7), 0),         # planes shorter than a thread's run of units, an odd number of channels
    ((8, 301, 7, 7), 0),        # several planes to a thread
    ((16, 5, 27, 27), 0),       # planes of several runs
    ((32, 5, 27, 27), 0),       # whole words of mask and codes
    ((8, 3, 111, 111), 0),      # a plane over many pieces
    ((24, 75, 27, 27), 0),      # several units to a thread
    ((3, 7, 9, 24), 2),         # one group that a cluster holds instead
    ((5, 11, 40, 50), 2),       # one group, pieces that do not come out even
    ((32, 128, 28, 29), 2),     # one group over several units a thread
    ((3, 2, 256, 256), 1),      # planes of whole units, too long for a cluster to hold
]


def takes(b, dtype, shape, mode, with_backward=False, packed=False):
    """Does the call take the held form?"""
    geo = b.hold_geometry(b.BF16 if dtype == "bf16" else b.F32, shape, group=mode, with_backward=with_backward, packed=packed)
    return geo is not None and geo["taken"] == 1


@pytest.mark.parametrize("shape,mode", CASES, ids=lambda v: "x".join(map(str, v)) if isinstance(v, tuple) else f"g{v}")
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_held_tensor(b, shape, mode, dtype):
    x, gy = make_case(shape, seed=sum(shape), dtype=dtype, relu=shape[0] % 2 == 0)
    bits = 2 + sum(shape) % 7
    ref = orc.fused(x, bits, gy=gy, group_mode=mode)
    xd, gyd = to_dev(x), to_dev(gy)
    assert takes(b, dtype, shape, mode) == (x.size > 8192 or mode != 2)
    assert takes(b, dtype, shape, mode, packed=True) == (x.size % 32 == 0)
    ws = b.make_workspace(xd, group=mode, zeroed=True)
    new = lambda: b.FakeQuantOut(workspace=ws)
    clean = lambda: b.workspace_status(ws) == b.OK and int(ws.view(torch.int32).abs().sum().item()) == 0
    for _ in range(2):
        got = b.granq_fakequant_fused(xd, bits, gy=gyd, group=mode, out=new(), want_params=True, flags=b.FLAG_WORKSPACE_ZEROED)
        assert clean()
        assert_parity(got, ref, shape, 1, mode, backward=True)
    got = b.granq_fakequant_fused(xd, bits, group=mode, out=new(), flags=b.FLAG_WORKSPACE_ZEROED)
    assert clean()
    assert_parity(got, ref, shape, 1, mode, backward=False)
    got = b.granq_fakequant_fused_stats(xd, bits, group=mode, out=new(), flags=b.FLAG_WORKSPACE_ZEROED)
    assert clean()
    assert_parity(got, ref, shape, 1, mode, backward=False)
    # fp32 inside a pack, fp64 beyond: about 8 roundings of 2^-24 of a sum of same-signed terms
    assert np.allclose(to_np(got.sums), orc.distortion_sums(x, ref.y), rtol=1e-6, atol=0)
    got = b.granq_fakequant_fused_fwd_packmask(xd, bits, group=mode, out=new(), flags=b.FLAG_WORKSPACE_ZEROED)
    assert clean()
    assert_parity(got, ref, shape, 1, mode, backward=False)
    assert_same_string(got.packed_mask, orc.pack_mask(ref.mask))
    for code_bits in (1, 3, 4, 5, 8):
        got = b.granq_quantize_packed_fused(xd, code_bits, group=mode, out=new(), flags=b.FLAG_WORKSPACE_ZEROED)
        assert clean()
        assert_same_string(got.packed_codes, orc.pack_codes(orc.fused(x, code_bits, group_mode=mode).codes, code_bits))
    dirty = b.FakeQuantOut(workspace=b.make_workspace(xd, group=mode).fill_(255))
    assert_parity(b.granq_fakequant_fused(xd, bits, gy=gyd, group=mode, out=dirty), ref, shape, 1, mode, backward=True)


@pytest.mark.parametrize("shape,mode", [
    ((1, 1, 3, 3), 0),          # one unit of bf16 and one element
    ((3, 5, 7, 7), 0),          # 7 elements behind the last whole byte of a mask
    ((3, 2, 5, 9), 1),
    ((33, 7, 2, 5), 0),         # planes of little more than a unit of bf16
    ((3, 7, 5, 13), 2),
    ((21, 379, 7, 7), 0),       # several planes to a thread
    ((13, 13, 93, 93), 0),      # a plane over several pieces
    ((5, 41, 97, 10), 1),       # whole units of bf16 and half a unit of fp32 more than whole bytes
    ((7, 3, 2, 3), 0),          # planes shorter than what a thread handles: two passes
    ((1, 1, 4999, 5001), 2),    # one group of which bf16 reads a part again
], ids=lambda v: "x".join(map(str, v)) if isinstance(v, tuple) else f"g{v}")
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_elements_behind_the_last_whole_unit(b, shape, mode, dtype):
    """The last elements, the top of their group's range in one call and not in the other; masks and codes up to the end of the
    last word, in buffers that held something else; the workspace zero again; both kinds of call agree with two passes."""
    x, gy = make_case(shape, seed=sum(shape), dtype=dtype)
    for peak in (False, True):
        if peak:
            x.reshape(-1)[-1] = 0x42C8 if dtype == "bf16" else 100.0
        xd, gyd = to_dev(x), to_dev(gy)
        ws = b.make_workspace(xd, group=mode, zeroed=True)
        new = lambda: b.FakeQuantOut(workspace=ws)
        clean = lambda: b.workspace_status(ws) == b.OK and int(ws.view(torch.int32).abs().sum().item()) == 0
        for bits in (4, 7) if x.size < 1 << 20 else (4,):
            ref = orc.fused(x, bits, gy=gy, group_mode=mode)
            got = b.granq_fakequant_fused(xd, bits, gy=gyd, group=mode, out=new(), want_params=True, flags=b.FLAG_WORKSPACE_ZEROED)
            assert clean()
            assert_parity(got, ref, shape, 1, mode, backward=True)
            assert_parity(b.granq_fakequant_fused(xd, bits, group=mode), ref, shape, 1, mode, backward=False)
            got = b.granq_fakequant_fused_stats(xd, bits, group=mode, out=new(), flags=b.FLAG_WORKSPACE_ZEROED)
            assert clean()
            assert_parity(got, ref, shape, 1, mode, backward=False)
            # fp32 inside a pack, fp64 beyond: about 8 roundings of 2^-24 of a sum of same-signed terms
            assert np.allclose(to_np(got.sums), orc.distortion_sums(x, ref.y), rtol=1e-6, atol=0)
            out = new()
            out.packed_mask = torch.full(((x.size + 31) // 32,), -1, dtype=torch.int32, device="cuda")
            got = b.granq_fakequant_fused_fwd_packmask(xd, bits, group=mode, out=out, flags=b.FLAG_WORKSPACE_ZEROED)
            assert clean()
            assert_parity(got, ref, shape, 1, mode, backward=False)
            assert_same_string(got.packed_mask, orc.pack_mask(ref.mask))
            for code_bits in (1, 3, 4, 7, 8) if bits == 4 else ():
                out = new()
                out.packed_codes = torch.full(((x.size * code_bits + 31) // 32,), -1, dtype=torch.int32, device="cuda")
                got = b.granq_quantize_packed_fused(xd, code_bits, group=mode, out=out, flags=b.FLAG_WORKSPACE_ZEROED)
                assert clean()
                assert_same_string(got.packed_codes, orc.pack_codes(orc.fused(x, code_bits, group_mode=mode).codes, code_bits))


@pytest.mark.parametrize("dtype,shape,mode,launches", [
    ("f32", (101, 75, 27, 27), 0, 1),
    ("bf16", (101, 75, 27, 27), 0, 1),
    ("f32", (83, 2677, 3, 3), 1, 1),             # 222 191 groups of one plane
    ("f32", (119, 3767, 3, 3), 1, 3),            # 448 273
    ("bf16", (51, 1601, 7, 7), 1, 1),            # 81 651 groups, 4 M elements
    ("bf16", (67, 2133, 7, 7), 1, 3),            # 142 911 groups, 7 M elements
    ("f32", (1651, 18, 2, 2), 0, 1),             # plane after plane of few channels: codes by two passes
    ("f32", (401, 31, 2, 2), 0, 1),              # ... and held
], ids=lambda v: "x".join(map(str, v)) if isinstance(v, tuple) else str(v))
def test_many_groups_with_a_remainder(b, dtype, shape, mode, launches):
    """Held or, with very many groups or codes of very many short planes, not: the same bits either way."""
    x, _ = make_case(shape, seed=2, dtype=dtype)
    xd = to_dev(x)
    ref = orc.fused(x, 5, group_mode=mode)
    plan, n = b.fused_plan(b.BF16 if dtype == "bf16" else b.F32, shape, group=mode, with_backward=False)
    assert n == launches or plan != b.PLAN_TWO_PASS
    ws = b.make_workspace(xd, group=mode, zeroed=True)
    for kw in (dict(out=b.FakeQuantOut(workspace=ws), flags=b.FLAG_WORKSPACE_ZEROED), {}):
        assert_parity(b.granq_fakequant_fused(xd, 5, group=mode, **kw), ref, shape, 1, mode, backward=False)
        got = b.granq_quantize_packed_fused(xd, 5, group=mode, **kw)
        assert_same_string(got.packed_codes, orc.pack_codes(ref.codes, 5))
        assert b.workspace_status(ws) == b.OK and int(ws.view(torch.int32).abs().sum().item()) == 0


@pytest.mark.parametrize("dtype,shape,mode,calls", [
    ("bf16", (8, 16, 8, 8), 1, ""),                      # planes of whole units, too short
    ("bf16", (8, 8, 11, 12), 1, "fs"),                   # 8448 elements in planes that are not
    ("bf16", (8, 7, 11, 12), 1, ""),                     # 7392
    ("bf16", (64, 256, 3, 3), 1, "fsm"),                 # planes of little more than a unit
    ("bf16", (1, 304, 21, 21), 0, "fsm"),                # a batch of one
    ("bf16", (4, 5, 16, 16), 1, "s"),
    ("bf16", (8, 3, 64, 64), 1, "s"),
    ("bf16", (4, 17, 128, 128), 1, "fsm"),
    ("f32", (8, 8, 11, 13), 1, ""),
    ("f32", (60, 128, 20, 20), 1, "s"),
    ("f32", (7, 1072, 20, 20), 1, "s"),
    ("bf16", (75, 2800, 3, 3), 1, ""),                   # 210 000 groups
    ("bf16", (9, 72, 88, 88), 1, "fsm"),                 # beyond a wave of clusters
    ("bf16", (33, 1080, 15, 15), 1, ""),                 # ... with 35 640 groups
], ids=lambda v: "x".join(map(str, v)) if isinstance(v, tuple) else str(v))
def test_groups_of_one_plane(b, dtype, shape, mode, calls):
    """Where the launch that holds pieces stands in for the cluster-local one: f forward and with a gradient, s sums, m packed mask
    and codes; both give the oracle's bits, also where the cooperative launch is refused."""
    x, gy = make_case(shape, seed=sum(shape), dtype=dtype)
    ref = orc.fused(x, 5, gy=gy, group_mode=mode)
    xd, gyd = to_dev(x), to_dev(gy)
    assert b.fused_plan(b.BF16 if dtype == "bf16" else b.F32, shape, group=mode)[0] == b.PLAN_CLUSTER
    assert takes(b, dtype, shape, mode) == takes(b, dtype, shape, mode, with_backward=True) == ("f" in calls)
    assert takes(b, dtype, shape, mode, packed=True) == ("m" in calls and x.size % 32 == 0)
    ws = b.make_workspace(xd, group=mode, zeroed=True)
    clean = lambda: b.workspace_status(ws) == b.OK and int(ws.view(torch.int32).abs().sum().item()) == 0
    for flags in (0, b.FLAG_WORKSPACE_ZEROED, b.FLAG_FORCE_CLUSTER):
        new = lambda: b.FakeQuantOut(workspace=ws) if flags == b.FLAG_WORKSPACE_ZEROED else b.FakeQuantOut()
        got = b.granq_fakequant_fused(xd, 5, gy=gyd, group=mode, out=new(), want_params=True, flags=flags)
        assert clean()
        assert_parity(got, ref, shape, 1, mode, backward=True)
        assert_parity(b.granq_fakequant_fused(xd, 5, group=mode, out=new(), flags=flags), ref, shape, 1, mode, backward=False)
        got = b.granq_fakequant_fused_stats(xd, 5, group=mode, out=new(), flags=flags)
        assert clean()
        assert_parity(got, ref, shape, 1, mode, backward=False)
        # fp32 inside a pack, fp64 beyond: about 8 roundings of 2^-24 of a sum of same-signed terms
        assert np.allclose(to_np(got.sums), orc.distortion_sums(x, ref.y), rtol=1e-6, atol=0)
        got = b.granq_fakequant_fused_fwd_packmask(xd, 5, group=mode, out=new(), flags=flags)
        assert_parity(got, ref, shape, 1, mode, backward=False)
        assert_same_string(got.packed_mask, orc.pack_mask(ref.mask))
        if not flags & b.FLAG_FORCE_CLUSTER:
            got = b.granq_quantize_packed_fused(xd, 5, group=mode, out=new(), flags=flags)
            assert clean()
            assert_same_string(got.packed_codes, orc.pack_codes(ref.codes, 5))
    try:
        b.tune(b.KNOB_TEST_COOP_CTAS, 1)
        assert_parity(b.granq_fakequant_fused(xd, 5, gy=gyd, group=mode), ref, shape, 1, mode, backward=True)
        assert_parity(b.granq_fakequant_fused_stats(xd, 5, group=mode), ref, shape, 1, mode, backward=False)
        assert_same_string(b.granq_fakequant_fused_fwd_packmask(xd, 5, group=mode).packed_mask, orc.pack_mask(ref.mask))
        assert_same_string(b.granq_quantize_packed_fused(xd, 5, group=mode).packed_codes, orc.pack_codes(ref.codes, 5))
    finally:
        b.tune(b.KNOB_TEST_COOP_CTAS, 0)


@pytest.mark.parametrize("dtype,shape", [("f32", (96, 128, 28, 28)), ("bf16", (192, 128, 28, 28))])
def test_one_group_beyond_what_stays_on_chip(b, dtype, shape):
    x, gy = make_case(shape, seed=3, dtype=dtype)
    ref = orc.fused(x, 4, gy=gy, group_mode=2)
    xd, gyd = to_dev(x), to_dev(gy)
    assert takes(b, dtype, shape, 2) and takes(b, dtype, shape, 2, with_backward=True) == (dtype == "bf16")
    assert_parity(b.granq_fakequant_fused(xd, 4, gy=gyd, group=2), ref, shape, 1, 2, backward=True)
    assert_parity(b.granq_fakequant_fused(xd, 4, group=2), ref, shape, 1, 2, backward=False)
    got = b.granq_fakequant_fused_stats(xd, 4, group=2)
    assert_parity(got, ref, shape, 1, 2, backward=False)
    assert np.allclose(to_np(got.sums), orc.distortion_sums(x, ref.y), rtol=1e-6, atol=0)


@pytest.mark.parametrize("dtype,shape", [
    ("f32", (96, 128, 28, 28)),
    ("f32", (128, 128, 28, 28)),
    ("f32", (32, 315, 1667, 1)),      # next to twice what stays, the last piece a sixth shorter than the others
    ("bf16", (192, 128, 28, 28)),
], ids=lambda v: "x".join(map(str, v)) if isinstance(v, tuple) else v)
def test_packed_outputs_of_one_group_beyond_what_stays_on_chip(b, dtype, shape):
    """Mask and codes of the part that is read again.  At 4 bits lo = -hi = -7.5 makes s = 1 and z = 8: the elements at the
    top, one in ten, land on 16 and get no gradient, so that a bit in the wrong place shows in the mask too."""
    x = np.clip(6.0 * np.random.default_rng(17).standard_normal(shape, dtype=np.float32), -7.5, 7.5)
    x = wl.to_bf16_bits(x) if dtype == "bf16" else x
    xd = to_dev(x)
    geo = b.hold_geometry(b.BF16 if dtype == "bf16" else b.F32, shape, group=2, with_backward=False, packed=True)
    assert geo["taken"] == 1 and geo["kept"] < geo["units"]
    zeroed = b.make_workspace(xd, group=2, zeroed=True)
    for code_bits in (1, 3, 4, 5, 8):
        ref = orc.fused(x, code_bits, group_mode=2)
        for ws, flags in ((b.make_workspace(xd, group=2).fill_(255), 0), (zeroed, b.FLAG_WORKSPACE_ZEROED)):
            got = b.granq_quantize_packed_fused(xd, code_bits, group=2, out=b.FakeQuantOut(workspace=ws), flags=flags)
            assert b.workspace_status(ws) == b.OK
            assert_same_string(got.packed_codes, orc.pack_codes(ref.codes, code_bits))
            if code_bits == 4:
                got = b.granq_fakequant_fused_fwd_packmask(xd, 4, group=2, out=b.FakeQuantOut(workspace=ws), flags=flags)
                assert b.workspace_status(ws) == b.OK
                assert_parity(got, ref, shape, 1, 2, backward=False)
                assert 0.05 < 1 - ref.mask.mean() < 0.2
                assert_same_string(got.packed_mask, orc.pack_mask(ref.mask))
    assert int(zeroed.view(torch.int32).abs().sum().item()) == 0


@pytest.mark.parametrize("stats", [False, True])
def test_a_hand_over_that_never_completes_is_reported(b, knobs, stats):
    x, _ = make_case((8, 75, 5, 7), seed=1)
    assert takes(b, "f32", x.shape, 0)
    xd = to_dev(x)
    call = b.granq_fakequant_fused_stats if stats else b.granq_fakequant_fused
    knobs(extra_arrivals=1, spin_limit=500)
    assert b.workspace_status(call(xd, 4).workspace) == b.ERR_TIMEOUT
    knobs(extra_arrivals=0, spin_limit=0)
    got = call(xd, 4)
    assert b.workspace_status(got.workspace) == b.OK
    assert_parity(got, orc.fused(x, 4), x.shape, 1, 0, backward=False)


@pytest.mark.parametrize("shape,mode", [((24, 75, 27, 27), 0), ((5, 11, 40, 50), 2), ((3, 2, 256, 256), 1)])
def test_a_refused_cooperative_launch_falls_back(b, knobs, shape, mode):
    x, gy = make_case(shape, seed=6)
    assert takes(b, "f32", shape, mode) and takes(b, "f32", shape, mode, with_backward=True)
    ref = orc.fused(x, 4, gy=gy, group_mode=mode)
    xd, gyd = to_dev(x), to_dev(gy)
    ws = b.make_workspace(xd, group=mode, zeroed=True)
    b.tune(b.KNOB_TEST_COOP_CTAS, 1)
    got = b.granq_fakequant_fused(xd, 4, gy=gyd, group=mode, out=b.FakeQuantOut(workspace=ws), flags=b.FLAG_WORKSPACE_ZEROED)
    assert_parity(got, ref, shape, 1, mode, backward=True)
    got = b.granq_fakequant_fused_stats(xd, 4, group=mode, out=b.FakeQuantOut(workspace=ws), flags=b.FLAG_WORKSPACE_ZEROED)
    assert_parity(got, ref, shape, 1, mode, backward=False)
    assert b.workspace_status(ws) == b.OK and int(ws.view(torch.int32).abs().sum().item()) == 0
