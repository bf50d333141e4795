"""The two forms of the column walk on aligned planes, mostly the resident one (a channel held in the shared memory of a team of CTAs) against the CPU
oracle, bit for bit: teams of one CTA and of many, one round of channels and several, shares that are not whole
runs of 8 units, planes shorter and longer than a block's stride, gy staged whole and in part - with every output
that the form writes, between guard bands, the workspace zero again afterwards; and the waves on the same shapes."""
import numpy as np
import pytest
import torch

from gpu_util import assert_parity, make_case, same_bits, to_dev, to_np
from oracle import granq_oracle as orc
from test_parity_gpu import b, knobs  # noqa: F401
from test_rounding_gpu import assert_same_string

pytestmark = pytest.mark.gpu

SHAPES = [
    (8, 400, 8, 8),      # one CTA per channel, two rounds
    (13, 700, 2, 4),     # planes of one bf16 unit
    (9, 24, 12, 12),     # several CTAs per channel, one round
    (8, 3, 4, 4),        # fewer units than a team could share
    (33, 310, 4, 8),     # rounds that do not come out even
    (11, 5, 20, 22),     # planes that are no multiple of the block
    (8, 4, 112, 112),    # planes longer than a block's stride
    (128, 16, 56, 56),   # shares beyond half the shared memory: gy staged in part
    (64, 300, 20, 20),   # two CTAs per channel and the next channel's copies on the heels of this one's
]
SEVERAL_ROUNDS = [(8, 400, 8, 8), (13, 700, 2, 4), (33, 310, 4, 8), (64, 300, 20, 20)]


@pytest.mark.parametrize("dtype,shape", [("f32", (8, 1500, 36, 36)), ("bf16", (16, 1500, 36, 36))],
                         ids=lambda v: "x".join(map(str, v)) if isinstance(v, tuple) else v)
def test_forward_whose_finer_cut_is_refused(b, dtype, shape):
    """Where the GPU does not hold twice the CTAs at once the call takes the cut that was asked for, not another plan."""
    x, _ = make_case(shape, seed=sum(shape), dtype=dtype)
    form = b.team_geometry(b.BF16 if dtype == "bf16" else b.F32, shape, with_backward=False)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert form["taken"] == 1 and form["rounds"] >= 5
    xd, ref = to_dev(x), orc.fused(x, 5)
    ran = []
    try:
        for cap in (0, 2 * sms):         # the finer cut has 4 CTAs of 256 threads per SM, the other 2 of 512
            b.tune(b.KNOB_TEST_COOP_CTAS, cap)
            with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CUDA]) as p:
                got = b.granq_fakequant_fused(xd, 5, flags=b.FLAG_FORCE_COLWALK)
                torch.cuda.synchronize()
            assert_parity(got, ref, shape, 1, orc.GROUP_CHANNEL, backward=False)
            ran.append([e.key for e in p.key_averages() if "granq" in e.key])
    finally:
        b.tune(b.KNOB_TEST_COOP_CTAS, 0)
    if not any(ran):
        pytest.skip("the profiler shows no kernels on this machine")
    for names, threads in zip(ran, (256, 512)):
        assert any("colteam_kernel" in n and f", {threads}>" in n for n in names), names


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_resident_walk(b, knobs, shape, dtype):
    x, gy = make_case(shape, seed=sum(shape), dtype=dtype, relu=shape[0] % 2 == 0)
    bits = 2 + sum(shape) % 7
    ref = orc.fused(x, bits, gy=gy)
    xd, gyd = to_dev(x), to_dev(gy)
    flags = b.FLAG_FORCE_COLWALK | b.FLAG_WORKSPACE_ZEROED
    knobs(col_team=1)          # also where the waves are the faster form
    for backward in (False, True):
        form = b.team_geometry(b.BF16 if dtype == "bf16" else b.F32, shape, with_backward=backward)
        assert form["taken"] == 1 and (form["rounds"] > 1) == (shape in SEVERAL_ROUNDS)
    ws = b.make_workspace(xd, zeroed=True)
    clean = lambda: b.workspace_status(ws) == b.OK and int(ws.view(torch.int32).abs().sum().item()) == 0
    for _ in range(2):
        got = b.granq_fakequant_fused(xd, bits, gy=gyd, out=b.FakeQuantOut(workspace=ws), want_params=True, flags=flags)
        assert clean()
        assert_parity(got, ref, shape, 1, orc.GROUP_CHANNEL, backward=True)
    got = b.granq_fakequant_fused(xd, bits, out=b.FakeQuantOut(workspace=ws), flags=flags)
    assert clean()
    assert_parity(got, ref, shape, 1, orc.GROUP_CHANNEL, backward=False)
    if (shape[1] * shape[2] * shape[3]) % 32 == 0:
        got = b.granq_fakequant_fused_fwd_packmask(xd, bits, out=b.FakeQuantOut(workspace=ws), flags=flags)
        assert clean()
        assert_parity(got, ref, shape, 1, orc.GROUP_CHANNEL, backward=False)
        assert_same_string(got.packed_mask, orc.pack_mask(ref.mask))
        got = b.granq_quantize_packed_fused(xd, bits, out=b.FakeQuantOut(workspace=ws), flags=flags)
        assert clean()
        assert_same_string(got.packed_codes, orc.pack_codes(ref.codes, bits))
    got = b.granq_fakequant_fused_stats(xd, bits, out=b.FakeQuantOut(workspace=ws), flags=flags)
    assert clean()
    assert_parity(got, ref, shape, 1, orc.GROUP_CHANNEL, backward=False)
    sums = orc.distortion_sums(x, ref.y)
    # fp32 inside a pack, fp64 beyond: about 8 roundings of 2^-24 of a sum of same-signed terms
    assert np.allclose(to_np(got.sums), sums, rtol=1e-6, atol=0)


@pytest.mark.parametrize("dtype,shape", [
    ("f32", (143, 15, 64, 64)),      # three rounds, shares that do not come out even
    ("f32", (232, 3, 112, 112)),     # a channel over all SMs, one team
    ("f32", (90, 40, 60, 44)),       # ten teams, four rounds
    ("bf16", (65, 28, 96, 96)),      # shares next to the smallest that are planned
    ("bf16", (69, 33, 96, 96)),
], ids=lambda v: "x".join(map(str, v)) if isinstance(v, tuple) else v)
def test_two_channels_side_by_side_by_default(b, dtype, shape):
    x, gy = make_case(shape, seed=sum(shape), dtype=dtype, relu=shape[0] % 2 == 0)
    form = b.team_geometry(b.BF16 if dtype == "bf16" else b.F32, shape)
    units = shape[0] * shape[2] * shape[3] // (8 if dtype == "bf16" else 4)
    assert form["taken"] == 1 and form["rounds"] > 1 and form["ctas"] * form["units"] >= 2 * units      # of both channels
    ref = orc.fused(x, 5, gy=gy)
    xd, gyd = to_dev(x), to_dev(gy)
    dirty, zeroed = b.make_workspace(xd).fill_(255), b.make_workspace(xd, zeroed=True)
    for ws, flags in ((dirty, 0), (zeroed, b.FLAG_WORKSPACE_ZEROED), (zeroed, b.FLAG_WORKSPACE_ZEROED)):
        got = b.granq_fakequant_fused(xd, 5, gy=gyd, out=b.FakeQuantOut(workspace=ws), want_params=True, flags=flags)
        assert b.workspace_status(ws) == b.OK
        assert_parity(got, ref, shape, 1, orc.GROUP_CHANNEL, backward=True)
    assert int(zeroed.view(torch.int32).abs().sum().item()) == 0


@pytest.mark.parametrize("shape", [(40, 290, 16, 20), (9, 310, 4, 8), (37, 300, 8, 12)], ids=lambda s: "x".join(map(str, s)))
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_strings_of_every_width(b, knobs, shape, dtype):
    """Codes and mask bits that neighbouring lanes write together: planes of whole words of codes and others, lanes with four
    units at a time, two, one, and warps whose first lanes alone have one more."""
    x, _ = make_case(shape, seed=sum(shape), dtype=dtype)
    xd = to_dev(x)
    knobs(col_team=1)
    assert b.team_geometry(b.BF16 if dtype == "bf16" else b.F32, shape, with_backward=False)["taken"] == 1
    ws = b.make_workspace(xd, zeroed=True)
    flags = b.FLAG_FORCE_COLWALK | b.FLAG_WORKSPACE_ZEROED
    for bits in range(1, 9):
        ref = orc.fused(x, bits)
        got = b.granq_quantize_packed_fused(xd, bits, out=b.FakeQuantOut(workspace=ws), flags=flags)
        assert_same_string(got.packed_codes, orc.pack_codes(ref.codes, bits))
        got = b.granq_fakequant_fused_fwd_packmask(xd, bits, out=b.FakeQuantOut(workspace=ws), flags=flags)
        assert_same_string(got.packed_mask, orc.pack_mask(ref.mask))


@pytest.mark.parametrize("dtype,shape", [("f32", (8, 1500, 36, 36)), ("bf16", (16, 1500, 36, 36)), ("f32", (25, 480, 36, 40))],
                         ids=lambda v: "x".join(map(str, v)) if isinstance(v, tuple) else v)
def test_forward_with_a_finer_cut(b, dtype, shape):
    """Half the threads and twice the CTAs, where that saves rounds: one CTA per channel and several, every output of the form."""
    x, _ = make_case(shape, seed=sum(shape), dtype=dtype, relu=shape[0] % 2 == 0)
    form = b.team_geometry(b.BF16 if dtype == "bf16" else b.F32, shape, with_backward=False)
    assert form["taken"] == 1 and form["rounds"] >= 5
    ref = orc.fused(x, 5)
    xd = to_dev(x)
    ws = b.make_workspace(xd, zeroed=True)
    flags = b.FLAG_FORCE_COLWALK | b.FLAG_WORKSPACE_ZEROED
    new = lambda: b.FakeQuantOut(workspace=ws)
    clean = lambda: b.workspace_status(ws) == b.OK and int(ws.view(torch.int32).abs().sum().item()) == 0
    assert_parity(b.granq_fakequant_fused(xd, 5, out=new(), flags=flags), ref, shape, 1, orc.GROUP_CHANNEL, backward=False)
    got = b.granq_fakequant_fused_fwd_packmask(xd, 5, out=new(), flags=flags)
    assert clean()
    assert_parity(got, ref, shape, 1, orc.GROUP_CHANNEL, backward=False)
    assert_same_string(got.packed_mask, orc.pack_mask(ref.mask))
    got = b.granq_quantize_packed_fused(xd, 5, out=new(), flags=flags)
    assert_same_string(got.packed_codes, orc.pack_codes(ref.codes, 5))
    got = b.granq_fakequant_fused_stats(xd, 5, out=new(), flags=flags)
    assert clean()
    assert_parity(got, ref, shape, 1, orc.GROUP_CHANNEL, backward=False)
    # fp32 inside a pack, fp64 beyond: about 8 roundings of 2^-24 of a sum of same-signed terms
    assert np.allclose(to_np(got.sums), orc.distortion_sums(x, ref.y), rtol=1e-6, atol=0)


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_waves_on_aligned_planes(b, knobs, shape, dtype):
    """The form that the resident one stands in for, with its own cut of the waves: every output it writes."""
    x, gy = make_case(shape, seed=sum(shape) + 1, dtype=dtype, relu=shape[0] % 2 == 1)
    ref = orc.fused(x, 5, gy=gy)
    xd, gyd = to_dev(x), to_dev(gy)
    knobs(col_team=2)
    assert b.team_geometry(b.BF16 if dtype == "bf16" else b.F32, shape)["taken"] == 0
    flags = b.FLAG_FORCE_COLWALK | b.FLAG_WORKSPACE_ZEROED
    ws = b.make_workspace(xd, zeroed=True)
    new = lambda: b.FakeQuantOut(workspace=ws)
    clean = lambda: b.workspace_status(ws) == b.OK and int(ws.view(torch.int32).abs().sum().item()) == 0
    assert_parity(b.granq_fakequant_fused(xd, 5, gy=gyd, out=new(), want_params=True, flags=flags), ref, shape, 1,
                  orc.GROUP_CHANNEL, backward=True)
    assert clean()
    assert_parity(b.granq_fakequant_fused(xd, 5, out=new(), flags=flags), ref, shape, 1, orc.GROUP_CHANNEL, backward=False)
    assert clean()
    got = b.granq_fakequant_fused_stats(xd, 5, out=new(), flags=flags)
    assert_parity(got, ref, shape, 1, orc.GROUP_CHANNEL, backward=False)
    # fp32 inside a pack, fp64 beyond: about 8 roundings of 2^-24 of a sum of same-signed terms
    assert clean() and np.allclose(to_np(got.sums), orc.distortion_sums(x, ref.y), rtol=1e-6, atol=0)
    if (shape[1] * shape[2] * shape[3]) % 32 == 0:
        got = b.granq_fakequant_fused_fwd_packmask(xd, 5, out=new(), flags=flags)
        assert clean()
        assert_parity(got, ref, shape, 1, orc.GROUP_CHANNEL, backward=False)
        assert_same_string(got.packed_mask, orc.pack_mask(ref.mask))
        for bits in range(1, 9):
            got = b.granq_quantize_packed_fused(xd, bits, out=new(), flags=flags)
            assert clean()
            assert_same_string(got.packed_codes, orc.pack_codes(orc.fused(x, bits).codes, bits))


def test_a_hand_over_that_never_completes_is_reported(b, knobs):
    x, gy = make_case((8, 24, 12, 12), seed=1)
    assert b.team_geometry(b.F32, x.shape)["taken"] == 1
    knobs(extra_arrivals=1, spin_limit=500)
    got = b.granq_fakequant_fused(to_dev(x), 4, gy=to_dev(gy), flags=b.FLAG_FORCE_COLWALK)
    assert b.workspace_status(got.workspace) == b.ERR_TIMEOUT
    knobs(extra_arrivals=0, spin_limit=0)
    got = b.granq_fakequant_fused(to_dev(x), 4, gy=to_dev(gy), flags=b.FLAG_FORCE_COLWALK)
    assert b.workspace_status(got.workspace) == b.OK
    assert same_bits(to_np(got.y), orc.fused(x, 4, gy=gy).y)


@pytest.mark.parametrize("dtype,shape", [("f32", (256, 168, 28, 28)), ("bf16", (256, 256, 28, 28))])
def test_large_tensors_take_the_resident_form_by_default(b, dtype, shape):
    """The first sizes that the default route hands to the resident form although a cluster would hold a channel,
    with a workspace that is not zero on entry; forward and with a gradient, packed mask, packed codes, sums."""
    x, gy = make_case(shape, seed=5, dtype=dtype)
    ref = orc.fused(x, 4, gy=gy)
    xd, gyd = to_dev(x), to_dev(gy)
    ws = b.make_workspace(xd)
    new = lambda: b.FakeQuantOut(workspace=ws.fill_(255))
    assert_parity(b.granq_fakequant_fused(xd, 4, out=new()), ref, shape, 1, orc.GROUP_CHANNEL, backward=False)
    assert_parity(b.granq_fakequant_fused(xd, 4, gy=gyd, out=new()), ref, shape, 1, orc.GROUP_CHANNEL, backward=True)
    got = b.granq_fakequant_fused_fwd_packmask(xd, 4, out=new())
    assert_parity(got, ref, shape, 1, orc.GROUP_CHANNEL, backward=False)
    assert_same_string(got.packed_mask, orc.pack_mask(ref.mask))
    got = b.granq_quantize_packed_fused(xd, 4, out=new())
    assert_same_string(got.packed_codes, orc.pack_codes(ref.codes, 4))
    got = b.granq_fakequant_fused_stats(xd, 4, out=new())
    assert_parity(got, ref, shape, 1, orc.GROUP_CHANNEL, backward=False)
    assert b.workspace_status(ws) == b.OK


def test_a_reported_timeout_outlives_later_calls_on_the_same_zeroed_workspace(b, knobs):
    """A call on a workspace handed over as zero whose hand-over never completes leaves keys and counters behind;
    a cluster-local call on the same workspace clears none of them, so it must not clear the report either."""
    shape = (8, 24, 12, 12)
    assert b.team_geometry(b.F32, shape)["taken"] == 1
    x, gy = make_case(shape, seed=2)
    xd, gyd = to_dev(x), to_dev(gy)
    ws = b.make_workspace(xd, zeroed=True)
    knobs(extra_arrivals=1, spin_limit=500)
    b.granq_fakequant_fused(xd, 4, gy=gyd, out=b.FakeQuantOut(workspace=ws), flags=b.FLAG_FORCE_COLWALK | b.FLAG_WORKSPACE_ZEROED)
    assert b.workspace_status(ws) == b.ERR_TIMEOUT
    knobs(extra_arrivals=0, spin_limit=0)
    zeroed = b.FLAG_FORCE_CLUSTER | b.FLAG_WORKSPACE_ZEROED
    new = lambda: b.FakeQuantOut(workspace=ws)
    for call in (lambda: b.granq_fakequant_fused(xd, 4, gy=gyd, out=new(), flags=zeroed),
                 lambda: b.granq_fakequant_fused(xd, 4, out=new(), flags=zeroed),
                 lambda: b.granq_fakequant_fused_fwd_packmask(xd, 4, out=new(), flags=b.FLAG_WORKSPACE_ZEROED),
                 lambda: b.granq_quantize_packed_fused(xd, 4, out=new(), flags=b.FLAG_WORKSPACE_ZEROED),
                 lambda: b.granq_fakequant_fused_stats(xd, 4, out=new(), flags=b.FLAG_WORKSPACE_ZEROED)):
        got = call()
        assert b.workspace_status(ws) == b.ERR_TIMEOUT
        assert same_bits(to_np(got.lo), orc.fused(x, 4).lo)
    got = b.granq_fakequant_fused(xd, 4, gy=gyd, out=new(), flags=b.FLAG_FORCE_CLUSTER)      # clears the word itself
    assert b.workspace_status(ws) == b.OK
    assert same_bits(to_np(got.y), orc.fused(x, 4, gy=gy).y)


@pytest.mark.parametrize("dtype,shape,forced", [("f32", (256, 168, 28, 28), False), ("bf16", (256, 256, 28, 28), False),
                                                ("f32", (9, 24, 12, 12), True), ("bf16", (9, 24, 12, 12), True)])
def test_a_refused_cooperative_launch_falls_back(b, knobs, dtype, shape, forced):
    """A GPU that is shared out holds fewer CTAs at once than its attributes say: where a cluster holds a channel the
    call takes the cluster, else the waves (whose grid follows the occupancy)."""
    x, gy = make_case(shape, seed=6, dtype=dtype)
    ref = orc.fused(x, 4, gy=gy)
    xd, gyd = to_dev(x), to_dev(gy)
    ws = b.make_workspace(xd)
    new = lambda: b.FakeQuantOut(workspace=ws.fill_(255))
    flags = b.FLAG_FORCE_COLWALK if forced else 0
    b.tune(b.KNOB_TEST_COOP_CTAS, 1)
    assert_parity(b.granq_fakequant_fused(xd, 4, out=new(), flags=flags), ref, shape, 1, orc.GROUP_CHANNEL, backward=False)
    assert b.workspace_status(ws) == b.OK
    assert_parity(b.granq_fakequant_fused(xd, 4, gy=gyd, out=new(), flags=flags), ref, shape, 1, orc.GROUP_CHANNEL, backward=True)
    assert b.workspace_status(ws) == b.OK
    got = b.granq_fakequant_fused_fwd_packmask(xd, 4, out=new(), flags=flags)
    assert_parity(got, ref, shape, 1, orc.GROUP_CHANNEL, backward=False)
    assert_same_string(got.packed_mask, orc.pack_mask(ref.mask))
    got = b.granq_quantize_packed_fused(xd, 4, out=new(), flags=flags)
    assert_same_string(got.packed_codes, orc.pack_codes(ref.codes, 4))
    got = b.granq_fakequant_fused_stats(xd, 4, out=new(), flags=flags)
    assert_parity(got, ref, shape, 1, orc.GROUP_CHANNEL, backward=False)
    assert b.workspace_status(ws) == b.OK
