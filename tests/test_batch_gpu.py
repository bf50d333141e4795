"""granq_fakequant_fused_batch: a list of tensors in one host call.  Every tensor must come out bit for bit as the
oracle computes it (and as the single call does); a bad descriptor stops the batch at its index."""
import threading

import numpy as np
import pytest
import torch

from gpu_util import assert_parity, make_case, same_bits, to_dev, to_np
from oracle import granq_oracle as orc

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def b():
    from paper_2503_18339_b200 import binding
    binding.lib()
    return binding


SHAPES = [(4, 16, 32, 32), (4, 32, 16, 16), (8, 64, 8, 8), (3, 20, 7, 7), (16, 8, 14, 14), (2, 3, 5, 5)]


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("backward", [True, False], ids=["fwd+bwd", "fwd"])
def test_batch_matches_the_oracle_and_the_single_calls(b, dtype, backward):
    cases = [make_case(s, seed=100 + i, dtype=dtype, relu=(i % 2 == 0)) for i, s in enumerate(SHAPES)]
    bits = [2 + (i * 3) % 7 for i in range(len(SHAPES))]
    xs = [to_dev(x) for x, _ in cases]
    gys = [to_dev(gy) if backward else None for _, gy in cases]
    batch = b.FusedBatch(list(zip(xs, bits, gys)), want_params=True)
    outs = batch.run()
    torch.cuda.synchronize()
    for i, ((x, gy), o) in enumerate(zip(cases, outs)):
        ref = orc.fused(x, bits[i], gy=gy if backward else None)
        assert b.workspace_status(o.workspace) == b.OK
        assert_parity(o, ref, SHAPES[i], 1, orc.GROUP_CHANNEL, backward=backward)
        single = b.granq_fakequant_fused(xs[i], bits[i], gy=gys[i], want_params=True)
        assert same_bits(to_np(single.y), to_np(o.y)) and same_bits(to_np(single.lo), to_np(o.lo))
        if backward:
            assert same_bits(to_np(single.gx), to_np(o.gx))
    # a second run over the same descriptors (workspaces are left as they were found)
    outs = batch.run()
    torch.cuda.synchronize()
    for i, ((x, gy), o) in enumerate(zip(cases, outs)):
        assert same_bits(to_np(o.y), orc.fused(x, bits[i]).y)


def test_batch_per_sample_groups(b):
    x, gy = make_case((6, 10, 9, 9), seed=7)
    batch = b.FusedBatch([(to_dev(x), 4, to_dev(gy))], group=b.GROUP_SAMPLE_CHANNEL, want_params=True)
    o = batch.run()[0]
    assert_parity(o, orc.fused(x, 4, gy=gy, group_mode=orc.GROUP_SAMPLE_CHANNEL), x.shape, 1, orc.GROUP_SAMPLE_CHANNEL,
                  backward=True)


def test_batch_stops_at_the_bad_descriptor(b):
    xs = [to_dev(make_case(s, seed=i)[0]) for i, s in enumerate(SHAPES[:3])]
    batch = b.FusedBatch([(x, 4, None) for x in xs])
    batch._descs[1].bits = 9                       # out of range: tensor 0 runs, tensor 1 is refused, tensor 2 is not reached
    before = to_np(batch.outs[2].y.fill_(-7.0)).copy()
    with pytest.raises(b.GranqError) as err:
        batch.run()
    assert err.value.status == b.ERR_INVALID_ARG and "tensor 1" in str(err.value)
    torch.cuda.synchronize()
    assert same_bits(to_np(batch.outs[2].y), before)
    assert same_bits(to_np(batch.outs[0].y), orc.fused(to_np(xs[0]), 4).y)


def test_batch_tensors_that_run_beside_one_another_and_tensors_that_depend(b):
    """More tensors than run together, in which some read what an earlier one of the list wrote (next to it and further
    back), one writes what an earlier one read, and two share a workspace: as if made one after the other."""
    shape = (16, 16, 14, 14)
    n = 24
    cases = [make_case(shape, seed=50 + i) for i in range(n)]
    src = [x for x, _ in cases]
    xs = [to_dev(x) for x in src]
    gys = [to_dev(gy) for _, gy in cases]
    outs = [b.FakeQuantOut(y=torch.empty_like(x), gx=torch.empty_like(x), workspace=b.make_workspace(x, zeroed=True)) for x in xs]
    reads = {3: 2, 9: 5, 17: 16, 18: 17}                   # tensor i quantizes what tensor reads[i] wrote
    for i, k in reads.items():
        xs[i] = outs[k].y
    outs[13].y = xs[11]                                    # tensor 13 overwrites what tensor 11 has read
    outs[21].workspace = outs[20].workspace
    batch = b.FusedBatch(list(zip(xs, [4] * n, gys)), outs=outs, zeroed=True)
    for _ in range(3):
        xs[11].copy_(to_dev(src[11]))
        batch.run()
        torch.cuda.synchronize()
        ys = []
        for i in range(n):
            ref = orc.fused(ys[reads[i]] if i in reads else src[i], 4, gy=cases[i][1])
            ys.append(ref.y)
            assert b.workspace_status(outs[i].workspace) == b.OK
            assert same_bits(to_np(outs[i].y), ref.y) and same_bits(to_np(outs[i].gx), ref.gx), f"tensor {i}"
            assert same_bits(to_np(outs[i].lo), ref.lo) and same_bits(to_np(outs[i].hi), ref.hi)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_batch_reads_what_was_written_just_before_it(b, dtype):
    """The inputs of all tensors of a list are rewritten by the kernel ahead of it, in place, round after round: the
    tensors that start beside the first one must see the new values (bf16 reads gy in the quantize walk)."""
    shape, n = (16, 64, 14, 14), 9
    src = [make_case(shape, seed=90 + i, dtype=dtype) for i in range(3)]
    t = torch.bfloat16 if dtype == "bf16" else torch.float32
    X, GY = (torch.empty((n,) + shape, dtype=t, device="cuda") for _ in range(2))
    outs = [b.FakeQuantOut(y=torch.empty(shape, dtype=t, device="cuda"), gx=torch.empty(shape, dtype=t, device="cuda")) for _ in range(n)]
    batch = b.FusedBatch([(X[i], 4, GY[i]) for i in range(n)], outs=outs, zeroed=True)
    srcd = [(to_dev(x), to_dev(gy)) for x, gy in src]
    refs = [orc.fused(x, 4, gy=gy) for x, gy in src]
    kept = [(torch.empty((n,) + shape, dtype=t, device="cuda"), torch.empty((n,) + shape, dtype=t, device="cuda")) for _ in range(6)]
    torch.cuda.synchronize()
    for r, (ys, gxs) in enumerate(kept):
        x, gy = srcd[r % 3]
        GY.copy_(gy.expand_as(GY))
        X.copy_(x.expand_as(X))
        batch.run()
        for i in range(n):
            ys[i].copy_(outs[i].y)
            gxs[i].copy_(outs[i].gx)
    torch.cuda.synchronize()
    for r, (ys, gxs) in enumerate(kept):
        for i in range(n):
            assert same_bits(to_np(ys[i]), refs[r % 3].y) and same_bits(to_np(gxs[i]), refs[r % 3].gx), f"round {r}, tensor {i}"


@pytest.mark.parametrize("axis,big,small,forced", [(1, (128, 16, 56, 56), (8, 16, 8, 8), "FORCE_COLWALK"), (3, (9, 14, 14, 2048), (4, 4, 4, 16), None),
                                                   (1, (32, 48, 28, 28), (4, 16, 8, 8), "FORCE_CLUSTER")],
                         ids=["resident column walk", "channels-last", "cluster-local"])
def test_calls_of_different_sizes_from_several_threads(b, axis, big, small, forced):
    """Threads with a stream each whose calls take the same kernel with much and with little shared memory."""
    flags = getattr(b, "FLAG_" + forced) if forced else 0
    errors, outs = [], {}

    def work(name, x, stream):
        try:
            out = b.FakeQuantOut(y=torch.empty_like(x), workspace=b.make_workspace(x, axis),
                                 **{k: torch.empty(x.shape[axis], device="cuda") for k in ("lo", "hi")})
            for _ in range(400):
                b.granq_fakequant_fused(x, 4, channel_axis=axis, out=out, flags=flags, stream=stream)
            outs[name] = out
        except Exception as err:
            errors.append(err)

    cases = {f"{k} {i}": make_case(s, seed=i)[0] for k, s in (("big", big), ("small", small)) for i in range(2)}
    xs = {name: to_dev(x) for name, x in cases.items()}
    torch.cuda.synchronize()
    threads = [threading.Thread(target=work, args=(name, x, torch.cuda.Stream())) for name, x in xs.items()]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not errors, errors
    for name, x in cases.items():
        assert b.workspace_status(outs[name].workspace) == b.OK
        assert same_bits(to_np(outs[name].y), orc.fused(x, 4, channel_axis=axis).y)
