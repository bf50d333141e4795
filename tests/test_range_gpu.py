"""The stand-alone range (Eq. 4) where its column path begins and ends, against the CPU oracle, bit for bit: planes that
are no whole 16-byte units, planes of one unit, units that straddle two channels at a tile's edge, fewer slabs than a
chunk and many, slabs of one column tile and of several, as many groups as one block finishes and more."""
import numpy as np
import pytest

from gpu_util import make_case, same_bits, to_dev, to_np
from oracle import granq_oracle as orc

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def b():
    from paper_2503_18339_b200 import binding
    binding.lib()
    for k in range(binding.N_KNOBS):
        binding.tune(k, 0)
    return binding


SHAPES = [(8, 8, 7, 7), (9, 24, 5, 5), (130, 5, 4, 4), (33, 300, 2, 4), (64, 8, 11, 11), (100, 1032, 1, 9), (8, 4096, 2, 2),
          (8, 4104, 2, 2), (7, 8, 7, 7), (31, 3, 16, 16), (12, 16, 23, 24), (257, 64, 3, 3)]


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_range_and_two_pass_parameters(b, shape, dtype):
    x, gy = make_case(shape, seed=sum(shape), dtype=dtype)
    if dtype == "f32":
        x[0, 0, 0, 0], x[-1, -1, -1, -1] = -3.0e38, 3.0e38           # first and last element carry an extreme
        x[:, 1] = np.float32(-0.0)                                   # an all -0 channel: reported as +0
    for mode in (orc.GROUP_CHANNEL, orc.GROUP_SAMPLE_CHANNEL, orc.GROUP_TENSOR):
        lo, hi = orc.range_(x, group_mode=mode)
        for _ in range(2):
            glo, ghi = b.granq_range(to_dev(x), group=mode)
            assert same_bits(to_np(glo), lo) and same_bits(to_np(ghi), hi)
    ref = orc.fused(x, 4, gy=gy)
    got = b.granq_fakequant_fused(to_dev(x), 4, gy=to_dev(gy), want_params=True, flags=b.FLAG_FORCE_TWO_PASS)
    assert same_bits(to_np(got.s), ref.s) and same_bits(to_np(got.z), ref.z)
    assert same_bits(to_np(got.y), ref.y) and same_bits(to_np(got.gx), ref.gx)
