"""The passes over memory where the number of elements is no multiple of a 16-byte unit or of a string of 8 codes: range, forward,
both directions, mask, codes, sums and the ways back, against the CPU oracle, bit for bit."""
import numpy as np
import pytest
import torch

from gpu_util import assert_parity, make_case, to_dev, to_np
from oracle import granq_oracle as orc
from test_parity_gpu import b  # noqa: F401
from test_rounding_gpu import assert_same_string

pytestmark = pytest.mark.gpu

SHAPES = [
    ((1, 1, 3, 3), 0),           # a unit of bf16 and one element
    ((3, 5, 7, 7), 0),
    ((1, 1, 1, 8193), 2),        # one element in the last tile
    ((1, 3, 25, 331), 1),        # whole units of bf16 less one element
    ((1, 1, 4097, 2), 0),        # two elements of a string of eight
    ((33, 7, 2, 5), 0),          # planes of little more than a unit
    ((9, 2001, 3, 3), 0),        # more groups, and planes of a tile, than the tables hold
    ((21, 379, 7, 7), 0),
    ((11, 111, 5, 11), 0),       # 67 155 elements: few more than decode by strings takes of bf16
    ((11, 219, 5, 11), 0),       # 132 495: ... of fp32
    ((1291, 15, 3, 3), 0),       # short planes, whose range takes packs from here on
    ((301, 33, 3, 3), 0),        # ... and scalars up to here
    ((2, 1501, 7, 7), 0),        # packs again, more groups than a block keeps
    ((13, 13, 93, 93), 0),       # (of bf16, the way back from the mask by packs)
    ((13, 14, 93, 97), 0),       # (of fp32 too)
    ((7, 3, 2, 3), 0),           # planes of less than a unit of bf16: the scalar forms
]


@pytest.mark.parametrize("shape,mode", SHAPES, ids=lambda v: "x".join(map(str, v)) if isinstance(v, tuple) else f"g{v}")
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("peak", [False, True])
def test_passes_over_a_remainder(b, shape, mode, dtype, peak):
    x, gy = make_case(shape, seed=sum(shape), dtype=dtype)
    if peak:                     # the last element is its group's largest
        x.reshape(-1)[-1] = 0x42C8 if dtype == "bf16" else 100.0
    xd, gyd = to_dev(x), to_dev(gy)
    bits = 2 + sum(shape) % 7
    ref = orc.fused(x, bits, gy=gy, group_mode=mode)
    two = dict(group=mode, flags=b.FLAG_FORCE_TWO_PASS)
    assert_parity(b.granq_fakequant_fused(xd, bits, gy=gyd, **two), ref, shape, 1, mode, backward=True)
    assert_parity(b.granq_fakequant_fused(xd, bits, **two), ref, shape, 1, mode, backward=False)
    got = b.granq_fakequant_fused_stats(xd, bits, **two)
    assert_parity(got, ref, shape, 1, mode, backward=False)
    # fp32 inside a pack, fp64 beyond: about 8 roundings of 2^-24 of a sum of same-signed terms
    assert np.allclose(to_np(got.sums), orc.distortion_sums(x, ref.y), rtol=1e-6, atol=0)
    lo, hi = orc.range_(x, group_mode=mode)
    got = b.granq_range(xd, group=mode)
    assert np.array_equal(to_np(got[0]), lo) and np.array_equal(to_np(got[1]), hi)
    narrow = ((lo + 0.2 * (hi - lo)).astype(np.float32), (lo + 0.7 * (hi - lo)).astype(np.float32))
    for low, high in ((lo, hi), narrow):
        ref = orc.fakequant(x, bits, low, high, gy=gy, group_mode=mode)
        lowd, highd = to_dev(low), to_dev(high)
        assert_parity(b.granq_fakequant_fwd(xd, bits, lowd, highd, group=mode), ref, shape, 1, mode, backward=False)
        gx = b.granq_fakequant_bwd(gyd, xd, bits, lowd, highd, group=mode).gx
        words = torch.full(((x.size + 31) // 32,), -1, dtype=torch.int32, device="cuda")
        got = b.granq_fakequant_fwd_packmask(xd, bits, lowd, highd, group=mode, packed_mask=words)
        assert_parity(got, ref, shape, 1, mode, backward=False)
        assert_same_string(got.packed_mask, orc.pack_mask(ref.mask))
        assert torch.equal(gx.view(torch.uint8), b.granq_fakequant_bwd_packmask(gyd, got.packed_mask).view(torch.uint8))
        assert np.array_equal(to_np(gx).view(np.uint8), np.ascontiguousarray(ref.gx).view(np.uint8))
        for code_bits in range(1, 9):
            words = torch.full(((x.size * code_bits + 31) // 32,), -1, dtype=torch.int32, device="cuda")
            got = b.granq_quantize_packed(xd, code_bits, lowd, highd, group=mode, packed_codes=words)
            codes = orc.pack_codes(orc.fakequant(x, code_bits, low, high, group_mode=mode).codes, code_bits)
            assert_same_string(got.packed_codes, codes)
            y = b.granq_dequantize_packed(got.packed_codes, shape, xd.dtype, code_bits, got.s, got.z, group=mode)
            want = orc.fakequant(x, code_bits, low, high, group_mode=mode).y
            assert np.array_equal(to_np(y).view(np.uint8), np.ascontiguousarray(want).view(np.uint8))
