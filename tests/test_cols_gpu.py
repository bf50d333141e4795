"""Forward with a given range by columns (granq_flat.cu): y and the packed mask against the CPU oracle, bit for bit."""
import numpy as np
import pytest

from gpu_util import assert_parity, make_case, to_dev
from oracle import granq_oracle as orc
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
