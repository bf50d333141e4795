"""Lists of tensors of the same dims that the resident walk takes in one launch: every tensor bit for bit as the CPU oracle has
it, with bit-widths of their own, beside tensors that are calls of their own; workspaces zero again; what may not be taken
together (shared memory, other dims, no gradient, workspaces that are not zero) comes out as before."""
import pytest
import torch

from gpu_util import assert_parity, make_case, to_dev
from oracle import granq_oracle as orc
from test_parity_gpu import b, knobs  # noqa: F401

pytestmark = pytest.mark.gpu

SMALL = (4, 16, 32, 32)


def prepare(b, shapes, dtype="f32", zeroed=True, no_gradient=()):
    cases = [make_case(s, seed=40 + i, dtype=dtype, relu=i % 2 == 0) for i, s in enumerate(shapes)]
    bits = [2 + (3 * i) % 7 for i in range(len(shapes))]
    gys = [None if i in no_gradient else gy for i, (_, gy) in enumerate(cases)]
    items = [(to_dev(x), bt, None if gy is None else to_dev(gy)) for (x, _), bt, gy in zip(cases, bits, gys)]
    batch = b.FusedBatch(items, want_params=True, zeroed=zeroed)
    refs = [orc.fused(x, bt, gy=gy) for (x, _), bt, gy in zip(cases, bits, gys)]
    return batch, refs, gys


def check(b, batch, refs, gys, shapes, zero=True):
    for o, ref, gy, s in zip(batch.outs, refs, gys, shapes):
        assert b.workspace_status(o.workspace) == b.OK
        assert_parity(o, ref, s, 1, orc.GROUP_CHANNEL, backward=gy is not None)
        assert not zero or int(o.workspace.view(torch.int32).abs().sum().item()) == 0


@pytest.mark.parametrize("dtype,shapes", [
    ("f32", [(256, 16, 32, 32)] * 3),                                       # shares of several units a thread
    ("f32", [SMALL] + [(24, 50, 60, 40)] * 5 + [SMALL, SMALL]),             # 12 MB, 50 channels: rounds that do not come out even
    ("f32", [(256, 32, 16, 16)] * 7),                                       # 8 MB
    ("f32", [(200, 9, 42, 42)] * 18),                                       # more than one launch takes
    ("bf16", [(256, 32, 32, 32)] * 2),                                      # calls of their own
])
@pytest.mark.parametrize("zeroed", [True, False])
def test_list_of_equal_dims(b, dtype, shapes, zeroed):
    batch, refs, gys = prepare(b, shapes, dtype, zeroed)
    for _ in range(2):
        batch.run()
        check(b, batch, refs, gys, shapes, zero=zeroed)


def test_what_is_not_taken_together(b):
    shapes = [(256, 16, 32, 32)] * 2 + [(256, 16, 32, 31)] + [(256, 16, 32, 32)] * 3
    batch, refs, gys = prepare(b, shapes, no_gradient=(4,))
    batch.run()
    check(b, batch, refs, gys, shapes)
    # the second call reads what the first one wrote
    x, gy = make_case(shapes[0], seed=7)
    first = orc.fused(x, 4, gy=gy)
    second = orc.fused(first.y, 3, gy=gy)
    y, gyd = torch.empty(shapes[0], device="cuda"), to_dev(gy)
    outs = [b.FakeQuantOut(y=y), b.FakeQuantOut()]
    chain = b.FusedBatch([(to_dev(x), 4, gyd), (y, 3, gyd)], outs=outs, zeroed=True)
    chain.run()
    assert_parity(chain.outs[0], first, shapes[0], 1, 0, backward=True)
    assert_parity(chain.outs[1], second, shapes[0], 1, 0, backward=True)


def test_a_bad_descriptor_stops_the_list_at_its_index(b):
    shapes = [(256, 16, 32, 32)] * 4
    batch, refs, gys = prepare(b, shapes)
    batch._descs[2].bits = 9
    batch.outs[3].y.fill_(7.0)
    with pytest.raises(b.GranqError, match="tensor 2"):
        batch.run()
    check(b, batch, refs[:2], gys[:2], shapes[:2])
    assert bool((batch.outs[3].y == 7.0).all())


def test_refused_launch_and_a_wait_that_runs_out(b, knobs):
    shapes = [(256, 16, 32, 32)] * 2
    batch, refs, gys = prepare(b, shapes)
    b.tune(b.KNOB_TEST_COOP_CTAS, 1)
    batch.run()
    check(b, batch, refs, gys, shapes)
    b.tune(b.KNOB_TEST_COOP_CTAS, 0)
    knobs(extra_arrivals=1, spin_limit=500)
    batch.run()
    assert all(b.workspace_status(o.workspace) == b.ERR_TIMEOUT for o in batch.outs)
