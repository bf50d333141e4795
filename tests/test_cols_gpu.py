"""Forward with a given range by columns (granq_flat.cu): y and the packed mask against the CPU oracle, bit for bit."""
import numpy as np
import pytest

from gpu_util import assert_parity, make_case, to_dev
from oracle import granq_oracle as orc
from paper_2503_18339_b200 import workloads as wl
from test_parity_gpu import b  # noqa: F401
from test_rounding_gpu import assert_same_string, hard_groups

pytestmark = pytest.mark.gpu

SHAPES = [
    (8, 16, 7, 7),        # one column tile, not full; units that straddle planes
    (9, 264, 7, 7),       # slabs of more than a tile; chunks of 4 slabs and a rest of one
    (37, 40, 9, 9),       # an odd last chunk
    (10, 24, 12, 12),     # whole units, a rest of two slabs
    (67, 64, 28, 28),     # blocks of more than 4 slabs
    (11, 8, 1, 8),        # planes of one bf16 unit
    (8, 6, 3, 5),         # slabs that are no whole units: left to tiles
    (160, 1184, 5, 5),    # 16 slabs to a block, more than a wave of blocks
    (1003, 3, 8, 8),      # several short slabs side by side in a row, the last row not full
    (5001, 4, 4, 4),      # the same, rows of one and of several blocks
    (2050, 8, 3, 3),      # ... with units that straddle planes
    (333, 1, 28, 28),     # one channel
    (70000, 1, 2, 4),     # slabs of a unit or two
    (9, 1, 4, 4),         # fewer slabs than would fill a block
]


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_forward_by_columns(b, shape, dtype):
    x, gy = make_case(shape, seed=sum(shape), dtype=dtype, relu=shape[0] % 2 == 0)
    xd = to_dev(x)
    bits = 2 + sum(shape) % 7
    lo, hi = orc.range_(x)
    narrow = ((lo + 0.2 * (hi - lo)).astype(np.float32), (lo + 0.7 * (hi - lo)).astype(np.float32))
    wide = ((lo - 1).astype(np.float32), (hi + 1).astype(np.float32))
    far = ((lo + 2.0 ** 30).astype(np.float32), (hi + 2.0 ** 30).astype(np.float32))      # a zero-point beyond any shortcut, a scale of 1e-8
    for low, high in ((lo, hi), narrow, wide, far):
        ref = orc.fakequant(x, bits, low, high, gy=gy)
        got = b.granq_fakequant_fwd(xd, bits, to_dev(low), to_dev(high))
        assert_parity(got, ref, shape, 1, orc.GROUP_CHANNEL, backward=False)
        got = b.granq_fakequant_fwd_packmask(xd, bits, to_dev(low), to_dev(high))
        assert_parity(got, ref, shape, 1, orc.GROUP_CHANNEL, backward=False)
        assert_same_string(got.packed_mask, orc.pack_mask(ref.mask))


@pytest.mark.parametrize("plane", [(6, 6), (7, 7)], ids=["whole", "ragged"])
@pytest.mark.parametrize("bits", [2, 4, 8])
def test_ties_by_columns(b, plane, bits):
    n = 16 * plane[0] * plane[1]
    x = np.ascontiguousarray(np.moveaxis(hard_groups(n, bits, seed=bits).reshape((16, 16) + plane), 0, 1))
    for low, high in (orc.range_(x), tuple((0.6 * v).astype(np.float32) for v in orc.range_(x))):
        ref = orc.fakequant(x, bits, low, high)
        got = b.granq_fakequant_fwd_packmask(to_dev(x), bits, to_dev(low), to_dev(high))
        assert_parity(got, ref, x.shape, 1, orc.GROUP_CHANNEL, backward=False)
        assert_same_string(got.packed_mask, orc.pack_mask(ref.mask))


@pytest.mark.parametrize("plane", [(6, 6), (7, 7), (8, 4)], ids=["whole", "ragged", "long"])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("bits", [1, 4, 8])
def test_elements_up_to_the_largest_finite_value(b, plane, dtype, bits):
    """Far outside the given range on both sides, up to where the quotient overflows, beside elements inside it."""
    x = np.ascontiguousarray(np.moveaxis(hard_groups(8 * plane[0] * plane[1], bits, seed=3).reshape((16, 8) + plane), 0, 1))
    lo, hi = orc.range_(np.clip(x, -0.8, 0.9))
    for i, v in enumerate((3.0e38, -3.0e38, 3.3e38, -3.3e38, 1.0e20, -1.0e30)):
        x[i, :, i % plane[0], (2 * i + 1) % plane[1]] = v
    if dtype == "bf16":
        x = wl.to_bf16_bits(x)
    assert b.forward_geometry(b.BF16 if dtype == "bf16" else b.F32, x.shape, packed_mask=True) is not None
    ref = orc.fakequant(x, bits, lo, hi, gy=x)
    for got in (b.granq_fakequant_fwd(to_dev(x), bits, to_dev(lo), to_dev(hi)), b.granq_fakequant_fwd_packmask(to_dev(x), bits, to_dev(lo), to_dev(hi))):
        assert_parity(got, ref, x.shape, 1, orc.GROUP_CHANNEL, backward=False)
    assert_same_string(got.packed_mask, orc.pack_mask(ref.mask))
