"""The single-multiply-add rounding of the kernels where it is closest to going wrong, against the CPU oracle, bit
for bit: elements on a tie and one unit in the last place beside it, groups whose top element the clamp catches
(lo = -hi), zero-points on both sides of the limit up to which the shortcut is taken, scales outside the range of
the short division, constant groups - through every kernel that quantizes."""
import numpy as np
import pytest
import torch

from gpu_util import assert_parity, same_bits, to_dev, to_np
from oracle import granq_oracle as orc
from paper_2503_18339_b200 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def b():
    from paper_2503_18339_b200 import binding
    binding.lib()
    for k in range(binding.N_KNOBS):
        binding.tune(k, 0)
    return binding


def hard_groups(n: int, bits: int, seed: int) -> np.ndarray:
    """[16, n] values, one awkward group per row; n even and at least 16."""
    rng = np.random.default_rng(seed)
    top = 2 ** bits - 1
    x = rng.standard_normal((16, n)).astype(np.float32)

    def ties(step, lo):         # every half step and its neighbours, between the ends lo and lo + top * step
        k = rng.integers(0, top, n) + np.float32(0.5)
        v = (np.float32(lo) + np.float32(step) * k).astype(np.float32)
        side = rng.integers(0, 3, n)
        v = np.where(side == 1, np.nextafter(v, np.float32(np.inf)), np.where(side == 2, np.nextafter(v, np.float32(-np.inf)), v))
        v[0], v[1] = lo, np.float32(lo) + np.float32(top) * np.float32(step)
        return v.astype(np.float32)

    x[0], x[1], x[2] = ties(1.0, 0.0), ties(0.1, -0.3), ties(0.37, -5.0)
    x[3] = np.clip(x[3], -1.5, 1.5)
    x[3, 0], x[3, 1] = -1.5, 1.5                                     # lo = -hi: the top element is a tie above the range
    x[4] = ties(1.0, -top / 2)                                       # the same, all elements on ties
    for row, z in ((5, 2.0 ** 20), (6, 2.0 ** 20 + 4), (7, 2.0 ** 22), (8, 1000.0)):
        x[row] = np.float32(z) + rng.integers(0, top + 1, n).astype(np.float32)      # s = 1: zero-point -z
        x[row, 0], x[row, 1] = z, z + top
    x[9] *= np.float32(1e-25)                                        # scale below 2^-60
    x[10] *= np.float32(1e25)                                        # above 2^60
    x[11], x[12] = 0.0, -3.25                                        # constant groups
    x[13] = np.maximum(x[13], 0)
    x[14] = rng.integers(-3, 4, n)
    return x + np.float32(0)


def assert_same_string(words, ref):
    """device words against the oracle's bytes (the last word's padding bits are zero)"""
    got, ref = words.cpu().numpy().view(np.uint8), np.ascontiguousarray(ref).view(np.uint8).reshape(-1)
    assert np.array_equal(got[:ref.size], ref) and not got[ref.size:].any()


LAYOUTS = [("nchw", (32, 16, 8, 8), 1), ("nchw", (8, 16, 7, 7), 1), ("nchw", (3, 16, 5, 5), 1), ("nhwc", (6, 5, 8, 16), 3)]


@pytest.mark.parametrize("layout,shape,axis", LAYOUTS, ids=lambda v: "x".join(map(str, v)) if isinstance(v, tuple) else str(v))
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("bits", [1, 2, 4, 7, 8])
def test_hard_groups_through_every_kernel(b, layout, shape, axis, dtype, bits):
    n = int(np.prod(shape)) // 16
    rows = hard_groups(n, bits, seed=bits + n)
    others = tuple(d for i, d in enumerate(shape) if i != axis)
    x = np.ascontiguousarray(np.moveaxis(rows.reshape((16,) + others), 0, axis))
    gy = np.random.default_rng(n).standard_normal(shape).astype(np.float32)
    if dtype == "bf16":
        x, gy = wl.to_bf16_bits(x), wl.to_bf16_bits(gy)
    ref = orc.fused(x, bits, gy=gy, channel_axis=axis)
    xd, gyd = to_dev(x), to_dev(gy)
    for flags in (0, b.FLAG_FORCE_CLUSTER, b.FLAG_FORCE_COLWALK, b.FLAG_FORCE_L2WAVE, b.FLAG_FORCE_TWO_PASS):
        try:
            for extras in (False, True):
                got = b.granq_fakequant_fused(xd, bits, gy=gyd, channel_axis=axis, want_codes=extras, want_mask=extras,
                                              want_params=True, flags=flags)
                assert b.workspace_status(got.workspace) == b.OK
                assert_parity(got, ref, shape, axis, orc.GROUP_CHANNEL, backward=True)
            if flags in (0, b.FLAG_FORCE_CLUSTER, b.FLAG_FORCE_COLWALK, b.FLAG_FORCE_TWO_PASS):
                got = b.granq_fakequant_fused_fwd_packmask(xd, bits, channel_axis=axis, flags=flags)
                assert_parity(got, ref, shape, axis, orc.GROUP_CHANNEL, backward=False)
                assert_same_string(got.packed_mask, orc.pack_mask(ref.mask))
                got = b.granq_quantize_packed_fused(xd, bits, channel_axis=axis, flags=flags)
                assert_same_string(got.packed_codes, orc.pack_codes(ref.codes, bits))
        except b.GranqError as err:         # a forced plan need not take every geometry
            assert flags and err.status == b.ERR_UNSUPPORTED


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("bits", [1, 4, 8])
def test_hard_groups_with_a_range_narrower_than_the_tensor(b, dtype, bits):
    """Elements far outside the given range, up to the largest finite values, where both sides of the clamp act."""
    shape, n = (4, 16, 6, 6), 144
    x = np.ascontiguousarray(np.moveaxis(hard_groups(n, bits, seed=3).reshape(16, 4, 6, 6), 0, 1))
    x[1, :, 2, 3], x[2, :, 1, 1] = 3.0e38, -3.0e38
    gy = np.random.default_rng(1).standard_normal(shape).astype(np.float32)
    lo, hi = orc.range_(np.clip(np.delete(x, (1, 2), axis=0), -0.8, 0.9))
    if dtype == "bf16":
        x, gy = wl.to_bf16_bits(x), wl.to_bf16_bits(gy)
    ref = orc.fakequant(x, bits, lo, hi, gy=gy)
    lod, hid = to_dev(lo), to_dev(hi)
    fwd = b.granq_fakequant_fwd(to_dev(x), bits, lod, hid, want_codes=True, want_params=True)
    assert_parity(fwd, ref, shape, 1, orc.GROUP_CHANNEL, backward=False, exact=True)
    bwd = b.granq_fakequant_bwd(to_dev(gy), to_dev(x), bits, lod, hid, want_mask=True)
    assert_parity(bwd, ref, shape, 1, orc.GROUP_CHANNEL, backward=True)


@pytest.mark.parametrize("layout,shape,axis", LAYOUTS, ids=lambda v: "x".join(map(str, v)) if isinstance(v, tuple) else str(v))
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("where", ["scattered", "clamped"])
def test_a_nan_is_code_zero_without_a_gradient_and_spoils_no_neighbour(b, layout, shape, axis, dtype, where):
    """NaN is outside the contract, but what it gives is the same from every kernel: it does not enter the range, its
    code is 0, no gradient passes, and every other element is as without it.  Groups where nothing is clamped, and
    (values on the ties of lo = -hi) groups where the top element is."""
    bits = 4
    n = int(np.prod(shape)) // 16
    rng = np.random.default_rng(n)
    rows = rng.standard_normal((16, n)).astype(np.float32)
    if where == "clamped":
        rows = np.clip(rows, -1.5, 1.5)
        rows[:, 0], rows[:, 1] = -1.5, 1.5
    others = tuple(d for i, d in enumerate(shape) if i != axis)
    x = np.ascontiguousarray(np.moveaxis(rows.reshape((16,) + others), 0, axis))
    gy = rng.standard_normal(shape).astype(np.float32)
    nan = rng.random((16, n)) < 0.05
    nan[:, :2] = False
    nan[3:6, 5] = True
    nan = np.ascontiguousarray(np.moveaxis(nan.reshape((16,) + others), 0, axis))
    x[nan] = 0.0                                # inside every group's range: the oracle takes no NaN
    bad = x.copy()
    bad[nan] = np.nan
    if dtype == "bf16":
        x, gy = wl.to_bf16_bits(x), wl.to_bf16_bits(gy)
    ref = orc.fused(x, bits, gy=gy, channel_axis=axis)
    badd = torch.from_numpy(bad).cuda().to(torch.bfloat16 if dtype == "bf16" else torch.float32)
    view = [1] * 4
    view[axis] = 16
    zero_code = torch.from_numpy((ref.s * (np.float32(0) - ref.z)).reshape(view)).expand(shape)
    zero_code = to_np(zero_code.to(badd.dtype).contiguous())
    ref.y[nan], ref.codes[nan], ref.mask[nan], ref.gx[nan] = zero_code[nan], 0, 0, 0
    gyd = to_dev(gy)
    for flags in (0, b.FLAG_FORCE_CLUSTER, b.FLAG_FORCE_COLWALK, b.FLAG_FORCE_L2WAVE, b.FLAG_FORCE_TWO_PASS):
        if axis == 3 and flags:          # two passes read such a tensor one element at a time: a NaN is then the maximum
            continue
        try:
            for extras in (False, True):
                got = b.granq_fakequant_fused(badd, bits, gy=gyd, channel_axis=axis, want_codes=extras, want_mask=extras,
                                              want_params=True, flags=flags)
                assert_parity(got, ref, shape, axis, orc.GROUP_CHANNEL, backward=True)
            if axis == 1 and flags != b.FLAG_FORCE_L2WAVE:
                got = b.granq_fakequant_fused_fwd_packmask(badd, bits, channel_axis=axis, flags=flags)
                assert_parity(got, ref, shape, axis, orc.GROUP_CHANNEL, backward=False)
                assert_same_string(got.packed_mask, orc.pack_mask(ref.mask))
                got = b.granq_quantize_packed_fused(badd, bits, channel_axis=axis, flags=flags)
                assert_same_string(got.packed_codes, orc.pack_codes(ref.codes, bits))
        except b.GranqError as err:         # a forced plan need not take every geometry
            assert flags and err.status == b.ERR_UNSUPPORTED
    if axis == 3:
        return
    out = b.WeightBatch([badd.movedim(1, 0).contiguous()], bits, [gyd.movedim(1, 0).contiguous()]).run()[0]
    first = lambda a: np.ascontiguousarray(np.moveaxis(a, 1, 0))
    assert same_bits(to_np(out.y), first(ref.y)) and same_bits(to_np(out.gx), first(ref.gx))
