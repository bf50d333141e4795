"""Host-only checks of the C ABI: the library builds, loads, exports every symbol that
include/granq.h declares, rejects bad arguments before anything is launched, and plans the
staged kernel's waves within the shared-memory budget."""
import ctypes
import os
import random
import re

import pytest

from paper_2503_18339_b200 import build as granq_build
from paper_2503_18339_b200 import workloads as wl

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def lib():
    granq_build.build()
    from paper_2503_18339_b200 import binding
    return binding.lib()


def declared_functions():
    text = open(os.path.join(ROOT, "include", "granq.h")).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return sorted(set(re.findall(r"\b(granq_[a-z_0-9]+)\s*\(", text)))


def test_every_declared_symbol_is_exported(lib):
    from paper_2503_18339_b200 import binding
    names = declared_functions()
    assert len(names) >= 13
    for n in names:
        assert hasattr(lib, n), n
    assert sorted(binding.EXPORTS) == names


def test_status_strings(lib):
    from paper_2503_18339_b200 import binding
    seen = {binding.status_string(i) for i in range(6)}
    assert len(seen) == 6 and binding.status_string(99) == "unknown status"


def test_geometry_queries(lib):
    from paper_2503_18339_b200 import binding as b
    shape = (8, 16, 7, 7)
    assert b.num_groups(shape, 1, b.GROUP_CHANNEL) == 16
    assert b.num_groups(shape, 1, b.GROUP_SAMPLE_CHANNEL) == 128
    assert b.num_groups(shape, 1, b.GROUP_TENSOR) == 1
    assert b.num_groups(shape, 0, b.GROUP_CHANNEL) == 8
    assert b.workspace_bytes(b.F32, shape) % 256 == 0 and b.workspace_bytes(b.F32, shape) >= 256 + 16 * 12
    assert b.workspace_bytes(7, shape) == 0
    with pytest.raises(ValueError):
        b.num_groups((8, 0, 7, 7))
    with pytest.raises(ValueError):
        b.num_groups((8, 16, 7, 7), channel_axis=4)
    with pytest.raises(ValueError):
        b.num_groups((1 << 20, 1 << 20, 2, 1))       # more than 2^40 elements


def test_argument_errors_are_detected_before_any_launch(lib):
    """Null pointers, bad bit-widths, bad enums and a missing workspace never reach the GPU
    (this runs on a machine without one)."""
    from paper_2503_18339_b200 import binding as b
    dims = (ctypes.c_int64 * 4)(2, 3, 4, 4)
    fake = ctypes.c_void_p(256 * 1024)                # never dereferenced on the host
    far = ctypes.c_void_p(256 * 1024 * 1024)
    r = lib.granq_range(None, b.F32, dims, 1, 0, fake, fake, fake, 4096, 0, None)
    assert r == b.ERR_INVALID_ARG
    r = lib.granq_range(fake, b.F32, dims, 1, 0, fake, fake, None, 0, 0, None)
    assert r == b.ERR_WORKSPACE
    r = lib.granq_range(fake, b.F32, dims, 1, 0, fake, fake, ctypes.c_void_p(256 * 1024 + 8), 4096, 0, None)
    assert r == b.ERR_WORKSPACE                       # misaligned workspace
    r = lib.granq_range(fake, b.F32, dims, 1, 0, fake, fake, fake, 64, 0, None)
    assert r == b.ERR_WORKSPACE                       # too small
    for bits in (0, 9, -1):
        r = lib.granq_fakequant_fwd(fake, b.F32, dims, 1, 0, bits, fake, fake, far, None, None, None, 0, None)
        assert r == b.ERR_INVALID_ARG
    r = lib.granq_fakequant_fwd(fake, 5, dims, 1, 0, 4, fake, fake, far, None, None, None, 0, None)
    assert r == b.ERR_INVALID_ARG                     # bad dtype
    r = lib.granq_fakequant_fwd(fake, b.F32, dims, 1, 3, 4, fake, fake, far, None, None, None, 0, None)
    assert r == b.ERR_INVALID_ARG                     # bad group mode
    r = lib.granq_fakequant_fwd(fake, b.F32, dims, 1, 0, 4, fake, fake, fake, None, None, None, 0, None)
    assert r == b.ERR_INVALID_ARG                     # y overlaps x
    r = lib.granq_fakequant_bwd(fake, far, b.F32, dims, 1, 0, 4, fake, fake, None, None, 0, None)
    assert r == b.ERR_INVALID_ARG                     # gx missing
    # fused: gy without gx, mask without gy
    r = lib.granq_fakequant_fused(fake, far, b.F32, dims, 1, 0, 4, ctypes.c_void_p(3 << 28), None, fake, fake,
                                  None, None, None, None, fake, 4096, 0, None)
    assert r == b.ERR_INVALID_ARG
    r = lib.granq_fakequant_fused(fake, None, b.F32, dims, 1, 0, 4, far, None, fake, fake,
                                  None, fake, None, None, fake, 4096, 0, None)
    assert r == b.ERR_INVALID_ARG
    assert lib.granq_tune(99, 0) == b.ERR_INVALID_ARG
    assert lib.granq_workspace_status(None, None) == b.ERR_INVALID_ARG
    # the later entry points: missing outputs, misaligned buffers, bad bit-widths
    odd = ctypes.c_void_p(3 << 28 | 2)
    r = lib.granq_fakequant_fwd_packmask(fake, b.F32, dims, 1, 0, 4, fake, fake, far, None, None, None, 0, None)
    assert r == b.ERR_INVALID_ARG                     # packed mask missing
    r = lib.granq_fakequant_fwd_packmask(fake, b.F32, dims, 1, 0, 4, fake, fake, far, odd, None, None, 0, None)
    assert r == b.ERR_INVALID_ARG                     # packed mask not on a 4-byte boundary
    r = lib.granq_fakequant_bwd_packmask(fake, ctypes.c_void_p(3 << 28), b.F32, dims, fake, 0, None)
    assert r == b.ERR_INVALID_ARG                     # gx on top of gy
    r = lib.granq_fakequant_fused_fwd_packmask(fake, b.F32, dims, 1, 0, 4, far, ctypes.c_void_p(3 << 28), fake, fake,
                                               None, None, None, 0, 0, None)
    assert r == b.ERR_WORKSPACE
    r = lib.granq_distortion(fake, far, b.F32, dims, odd, 0, None)
    assert r == b.ERR_INVALID_ARG                     # sums not on an 8-byte boundary
    r = lib.granq_fakequant_fused_stats(fake, b.F32, dims, 1, 0, 4, far, fake, fake, None, None, None, fake, 4096, 0,
                                        None)
    assert r == b.ERR_INVALID_ARG                     # sums missing
    r = lib.granq_quantize_packed(fake, b.F32, dims, 1, 0, 9, fake, fake, far, None, fake, fake, 0, None)
    assert r == b.ERR_INVALID_ARG                     # 9 bits
    r = lib.granq_quantize_packed(fake, b.F32, dims, 1, 0, 4, fake, fake, far, None, None, fake, 0, None)
    assert r == b.ERR_INVALID_ARG                     # scale output missing
    r = lib.granq_dequantize_packed(far, b.F32, dims, 1, 0, 4, fake, None, fake, 0, None)
    assert r == b.ERR_INVALID_ARG                     # zero-point missing
    assert b.packmask_bytes((2, 3, 4, 4)) == 12 and b.packed_codes_bytes((2, 3, 4, 4), 3) == 36
    desc = (b.WeightDesc * 1)(b.WeightDesc(256 * 1024, None, 3 << 28, None, 256 * 1024, 256 * 1024, None, None, 4, 8,
                                           0, 0))
    assert lib.granq_fakequant_weights(desc, 1, b.F32, fake, 4096, 0, None) == b.ERR_INVALID_ARG      # 0 bits
    desc[0].bits = 4
    assert lib.granq_fakequant_weights(desc, 1, b.F32, None, 0, 0, None) == b.ERR_WORKSPACE
    assert lib.granq_fakequant_weights(desc, 0, b.F32, fake, 4096, 0, None) == b.ERR_INVALID_ARG
    assert lib.granq_host_arena_status(b.F32, dims, 1, 0, 1, None, None) == b.ERR_INVALID_ARG


def test_binding_refuses_cpu_tensors(lib):
    import torch
    from paper_2503_18339_b200 import binding as b
    x = torch.zeros(2, 3, 4, 4)
    with pytest.raises(ValueError):
        b.granq_fakequant_fused(x, 4, out=b.FakeQuantOut(
            y=torch.empty_like(x), lo=torch.empty(3), hi=torch.empty(3), workspace=torch.empty(4096, dtype=torch.uint8)))


def _check_geometry(shape, dt, grp, geo):
    n, c, h, w = shape
    V = 4 if dt == 0 else 8
    outer, groups = (n, c) if grp == 0 else (1, n * c)
    inner = h * w
    cw, cu, nw = geo["cw"], geo["cu"], geo["nwaves"]
    assert geo["smem_bytes"] <= 232448 and 1 <= geo["depth"] <= 3
    assert (nw - 1) * cw < groups <= nw * cw
    if nw > 1:
        assert (cw * inner) % V == 0                       # every wave's slab starts on a 16-byte boundary
    for ch in ({cw, groups - (nw - 1) * cw} if nw > 1 else {groups}):
        units = ch * inner // V
        cps = -(-units // cu)
        nk = -(-outer * cps // geo["grid"])
        assert nk * cu <= geo["buf_units"], (shape, geo, nk)


def test_staged_plan_fits_the_shared_memory_budget_for_every_workload(lib):
    from paper_2503_18339_b200 import binding as b
    for cfg in range(1, 6):
        for spec in wl.config_tensors(cfg):
            for dt in ([b.F32, b.BF16] if cfg == 5 else [b.F32]):
                for grp in (b.GROUP_CHANNEL, b.GROUP_SAMPLE_CHANNEL):
                    geo = b.staged_geometry(dt, spec.shape, 1, grp)
                    assert geo is not None, (spec.name, dt, grp)
                    _check_geometry(spec.shape, dt, grp, geo)


def test_staged_plan_under_forced_small_buffers(lib):
    from paper_2503_18339_b200 import binding as b
    rnd = random.Random(1)
    planned = 0
    try:
        for _ in range(1500):
            shape = (rnd.randint(1, 9), rnd.randint(1, 40), rnd.choice([1, 2, 4, 7, 8, 14, 28]),
                     rnd.choice([4, 7, 8, 14, 16]))
            dt = rnd.choice([0, 1])
            V = 4 if dt == 0 else 8
            b.tune(b.KNOB_STAGED_DEPTH, rnd.choice([0, 1, 2, 3]))
            b.tune(b.KNOB_STAGED_MAX_BUF_UNITS, rnd.choice([0, 64, 100, 500]))
            grid = rnd.choice([3, 5, 148])
            geo = b.staged_geometry(dt, shape, sm_count=grid)
            if (shape[1] * shape[2] * shape[3]) % V or shape[2] * shape[3] < V:
                assert geo is None
                continue
            if geo is not None:
                planned += 1
                _check_geometry(shape, dt, 0, geo)
    finally:
        for k in range(b.N_KNOBS):
            b.tune(k, 0)
    assert planned > 500


def test_distortion_stats_against_the_oracle_and_closed_forms(lib):
    """Table 2's two statistics from the four sums: the C entry point against the oracle's and against
    closed forms (Q = X, Q = 0, a 3-4-5 pair), and its degenerate cases."""
    from oracle import granq_oracle as orc
    from paper_2503_18339_b200 import binding as b
    assert b.distortion_from_sums([4.0, 4.0, 4.0, 0.0]) == (1.0, 0.0)               # Q = X
    assert b.distortion_from_sums([4.0, 0.0, 0.0, 4.0]) == (0.0, 1.0)               # Q = 0
    assert b.distortion_from_sums([0.0, 0.0, 0.0, 0.0]) == (0.0, 0.0)               # X = 0
    cos, rel = b.distortion_from_sums([9.0, 16.0, 0.0, 25.0])                       # X = (3, 0), Q = (0, 4)
    assert cos == 0.0 and abs(rel - 5.0 / 3.0) < 1e-15
    rnd = random.Random(3)
    for _ in range(50):
        sxx, sqq = rnd.uniform(0.1, 1e6), rnd.uniform(0.1, 1e6)
        sxq = rnd.uniform(-1, 1) * (sxx * sqq) ** 0.5
        sums = [sxx, sqq, sxq, sxx + sqq - 2 * sxq]
        got, want = b.distortion_from_sums(sums), orc.distortion(sums)
        assert abs(got[0] - want[0]) <= 1e-15 * max(1.0, abs(want[0])) and abs(got[1] - want[1]) <= 1e-15 * max(1.0, want[1])
    assert lib.granq_distortion_stats(None, None, None) == b.ERR_INVALID_ARG


def test_cluster_plan_cuts_within_its_limits(lib):
    """Host-only: whatever the cluster-local planner answers respects its own invariants - a run is a whole
    number of 16-byte units in every slab, a CTA's tiles fit the shared memory of an SM twice over (or the
    forced limit), the cluster size is a portable power of two no larger than the number of slabs."""
    from paper_2503_18339_b200 import binding as b
    rnd = random.Random(11)
    planned = 0
    try:
        for _ in range(3000):
            shape = (rnd.choice([1, 2, 3, 8, 13, 64, 128, 256]), rnd.randint(1, 600),
                     rnd.choice([1, 2, 4, 7, 8, 14, 28, 56]), rnd.choice([1, 4, 7, 8, 14, 16, 28, 56]))
            dt, mode, bwd = rnd.choice([0, 1]), rnd.choice([0, 1]), rnd.choice([False, True])
            V, esize = (4, 4) if dt == 0 else (8, 2)
            b.tune(b.KNOB_CLUSTER_CTAS, rnd.choice([0, 0, 0, 1, 2, 4, 8]))
            b.tune(b.KNOB_CLUSTER_TILE_KB, rnd.choice([0, 0, 8, 32, 200]))
            b.tune(b.KNOB_CLUSTER_LOAD, rnd.choice([0, 0, 1, 2, 3, 4, 5]))
            b.tune(b.KNOB_CLUSTER_KMUL, rnd.choice([0, 0, 0, 2, 5]))
            geo = b.cluster_geometry(dt, shape, group=mode, with_backward=bwd)
            inner = shape[2] * shape[3]
            outer, C = (shape[0], shape[1]) if mode == 0 else (1, shape[0] * shape[1])
            if (C * inner) % V or inner < V:
                assert geo is None
                continue
            if geo is None:
                continue
            planned += 1
            k, R = geo["channels_per_run"], geo["cluster"]
            assert (k * inner) % V == 0 and k >= 1
            assert R in (1, 2, 4, 8) and R <= outer
            assert geo["grid"] == -(-C // k) * R
            assert geo["tile_bytes"] == -(-outer // R) * min(k, C if k > C else k) * inner * esize or k > C
            tiles = 2 if geo["staging"] in (2, 4) else 1
            assert tiles == 1 or bwd
            assert geo["smem_bytes"] >= tiles * geo["tile_bytes"] and geo["smem_bytes"] <= 227 * 1024
            assert geo["threads"] % 32 == 0 and 32 <= geo["threads"] <= 512
    finally:
        for k in range(b.N_KNOBS):
            b.tune(k, 0)
    assert planned > 300


def test_rows_plan_cuts_within_what_the_gpu_holds(lib):
    """Host-only: every cut of the channels-last planner covers the row, keeps a block of rows within the threads of a
    CTA and asks for no more CTAs than are resident at once; a GPU (or a part of one) with fewer SMs than there would
    be slices gets no cut instead of an empty one."""
    from paper_2503_18339_b200 import binding as b
    rnd = random.Random(12)
    refused = 0
    for _ in range(4000):
        dt, sms = rnd.choice([0, 1]), rnd.choice([1, 2, 3, 4, 8, 16, 66, 132, 148])
        V, top = (4, 448) if dt == 0 else (8, 384)
        C = V * rnd.randint(1, 4096 // V)
        shape = (rnd.choice([1, 7, 128, 40_000]), rnd.choice([1, 3]), 2, C)
        geo = b.rows_geometry(dt, shape, with_backward=rnd.choice([False, True]), sm_count=sms)
        ncol, ctas = C // V, 2 * sms
        if geo is None:
            refused += 1
            assert (ncol + 63) // 64 > ctas
            continue
        assert 1 <= geo["columns"] <= 64 and geo["columns"] * geo["slices"] >= ncol > geo["columns"] * (geo["slices"] - 1)
        assert geo["lanes"] >= 1 and geo["columns"] * geo["lanes"] <= top
        assert geo["team"] >= 1 and geo["team"] * geo["slices"] <= ctas
        if geo["slices"] > 1:                    # no slice ends inside a line, or, of a tensor that stays on chip, a sector
            beyond = shape[0] * shape[1] * 2 * ncol * 16 > ctas * 111 * 1024
            assert geo["columns"] % (8 if beyond else 2 if ncol % 2 == 0 else 1) == 0
    assert refused


def test_team_plan_cuts_within_its_limits_and_takes_over_where_it_should(lib):
    """Host-only: a team's shares cover a channel and fit half an SM's shared memory, teams take every channel; the form
    is taken with one round or long shares, the knob forces or forbids it, a knob of the waves keeps them."""
    from paper_2503_18339_b200 import binding as b
    rnd = random.Random(13)
    seen = set()
    try:
        for _ in range(3000):
            dt, bwd, sms = rnd.choice([0, 1]), rnd.choice([False, True]), rnd.choice([8, 132, 148])
            shape = (rnd.choice([8, 13, 64, 128, 256]), rnd.randint(1, 1200), rnd.choice([1, 4, 8, 14, 28, 56, 112]), rnd.choice([4, 7, 8, 28, 56]))
            for k in (b.KNOB_COLWALK_TEAM, b.KNOB_L2_WAVE_KB):
                b.tune(k, 0)
            geo = b.team_geometry(dt, shape, with_backward=bwd, sm_count=sms)
            V, C = (4, 8)[dt], shape[1]
            if geo is None:
                continue
            units = shape[0] * shape[2] * shape[3] // V
            assert geo["ctas"] * geo["units"] >= units and geo["units"] <= 111 * 1024 // 16
            assert geo["ctas"] * geo["teams"] <= 2 * sms and geo["teams"] <= C
            assert geo["rounds"] == -(-C // geo["teams"])
            rule = geo["units"] >= 2500 or geo["rounds"] == 1
            assert geo["taken"] == rule
            seen.add(rule)
            b.tune(b.KNOB_L2_WAVE_KB, 64)
            assert b.team_geometry(dt, shape, with_backward=bwd, sm_count=sms)["taken"] == 0
            b.tune(b.KNOB_COLWALK_TEAM, 1)
            assert b.team_geometry(dt, shape, with_backward=bwd, sm_count=sms)["taken"] == 1
            b.tune(b.KNOB_COLWALK_TEAM, 2)
            assert b.team_geometry(dt, shape, with_backward=bwd, sm_count=sms)["taken"] == 0
        assert seen == {False, True}
    finally:
        for k in range(b.N_KNOBS):
            b.tune(k, 0)


def test_no_channel_that_a_team_would_take_alone_is_left_to_the_waves(lib):
    """Host-only: where one channel at a time has one round or long shares, the plan with a gradient is taken too, be it that
    one or two channels side by side; the shapes named are ones whose two-channel shares are short."""
    from paper_2503_18339_b200 import binding as b
    rnd = random.Random(14)

    def one_channel(units, C, ctas):
        runs = -(-units // 8)
        cuts = [(-(-C // min(ctas // R, C)), 8 * -(-runs // R)) for R in range(1, min(ctas, runs) + 1)]
        return min((rounds * (share + 700), rounds, share) for rounds, share in cuts if share <= 111 * 1024 // 16)[1:]

    named = [(0, (222, 96, 80, 80)), (0, (112, 111, 56, 56)), (0, (212, 366, 40, 40)), (0, (143, 15, 64, 64)), (0, (143, 7, 96, 96)),
             (1, (69, 56, 96, 96)), (1, (45, 328, 128, 127)), (0, (11, 90, 96, 96))]
    drawn = [(rnd.choice([0, 1]), (rnd.randint(8, 256), rnd.randint(3, 500), rnd.choice([28, 40, 56, 96, 112]), rnd.choice([28, 48, 56, 80])))
             for _ in range(400)]
    two = 0
    for dt, shape in named + drawn:
        geo = b.team_geometry(dt, shape)
        if geo is None:
            continue
        rounds, share = one_channel(shape[0] * shape[2] * shape[3] // (4, 8)[dt], shape[1], 296)
        assert geo["taken"] == 1 or (rounds > 1 and share < 2500), (dt, shape)
        two += geo["rounds"] > rounds
    assert two > 100


def test_lists_go_together_where_that_is_the_faster_way(lib):
    """Host-only: lists that measured slower in one launch than as separate calls are separate, those that measured faster
    go together, and neighbouring batch sizes take the same way."""
    from paper_2503_18339_b200 import binding as b
    for shape, n in (((70, 256, 14, 14), 2), ((488, 128, 7, 8), 12), ((854, 64, 8, 8), 4), ((70, 64, 28, 28), 6), ((183, 16, 32, 32), 6),
                     ((160, 16, 32, 32), 7), ((256, 32, 16, 16), 4), ((200, 32, 16, 16), 6), ((10, 128, 32, 32), 4), ((256, 64, 8, 8), 6),
                     ((256, 16, 32, 32), 1)):
        assert b.batch_geometry(b.F32, shape, n) == 0, (shape, n)
    for shape, n in (((256, 32, 16, 16), 6), ((255, 32, 16, 16), 6), ((232, 32, 16, 16), 6), ((256, 16, 32, 32), 7), ((255, 16, 32, 32), 2),
                     ((17, 144, 56, 56), 2), ((8, 72, 80, 80), 3), ((977, 64, 8, 8), 6), ((249, 72, 16, 16), 12), ((128, 64, 56, 56), 6)):
        assert b.batch_geometry(b.F32, shape, n) == n, (shape, n)
    assert b.batch_geometry(b.F32, (256, 16, 32, 32), 40) == 16
    assert b.batch_geometry(b.BF16, (256, 32, 32, 32), 8) == 0


def test_teams_take_tensors_of_more_than_2_32_units(lib):
    """Host-only: 64 GB and more (one channel at a time: two side by side count units in 32 bits)."""
    from paper_2503_18339_b200 import binding as b
    for dt, shape in ((0, (2048, 6000, 32, 48)), (1, (2048, 6000, 64, 48))):
        for bwd in (False, True):
            geo = b.team_geometry(dt, shape, with_backward=bwd)
            assert geo["taken"] == 1 and geo["ctas"] * geo["units"] >= 2048 * 32 * 48 // 4


def test_held_form_cuts_within_its_limits_and_leaves_the_waves_to_their_knobs(lib):
    """Host-only: pieces cover the tensor and fit half an SM's shared memory; more is read again of one group only, of fp32
    with a gradient nothing; a knob of the L2-resident waves keeps one group on them."""
    from paper_2503_18339_b200 import binding as b
    rnd = random.Random(15)
    again = 0
    try:
        for _ in range(3000):
            dt, sms = rnd.choice([0, 1]), rnd.choice([8, 132, 148])
            bwd = rnd.choice([False, True])
            packed = not bwd and rnd.choice([False, True])
            mode = rnd.choice([0, 1, 2])
            shape = (rnd.choice([1, 8, 13, 64, 128]), rnd.randint(1, 300), rnd.choice([5, 7, 14, 27, 56]), rnd.choice([4, 7, 15, 28, 56]))
            geo = b.hold_geometry(dt, shape, group=mode, with_backward=bwd, packed=packed, sm_count=sms)
            if geo is None:
                continue
            V, E = (4, 8)[dt], shape[0] * shape[1] * shape[2] * shape[3]
            assert E % (32 if packed else V) == 0 and geo["ctas"] <= 2 * sms
            assert geo["ctas"] * geo["units"] >= E // V > (geo["ctas"] - 1) * geo["units"] and geo["units"] % 8 == 0
            assert geo["kept"] % 2 == 0 and geo["kept"] * 16 <= 111 * 1024 and geo["kept"] <= geo["units"] <= 2 * geo["kept"] + 4
            if geo["kept"] < geo["units"]:
                again += 1
                assert (mode == 2 or shape[1] == 1 and shape[0] == 1) and (dt == 1 or not bwd)
        assert again > 20
        one_group = dict(group=2, with_backward=False)
        assert b.hold_geometry(0, (64, 64, 28, 28), **one_group)["taken"] == 1
        for k in (b.KNOB_L2_WAVE_KB, b.KNOB_L2_UPL, b.KNOB_L2_CTAS_PER_SM):
            b.tune(k, 2)
            assert b.hold_geometry(0, (64, 64, 28, 28), **one_group)["taken"] == 0
            b.tune(k, 0)
    finally:
        for k in range(b.N_KNOBS):
            b.tune(k, 0)


def test_forward_by_columns_covers_the_tensor_and_fills_its_blocks(lib):
    """Every 16-byte unit is walked once, by a thread that knows its channel, and the lanes of a row's blocks are units to 15 of 16
    wherever some number of slabs side by side, up to 8192 units, makes them so."""
    from paper_2503_18339_b200 import binding as b
    rnd = random.Random(5)
    shapes = [(65536, 4, 4, 4), (100000, 3, 8, 8), (60000, 1, 28, 28), (20000, 16, 2, 2), (5000, 8, 4, 8), (8, 1, 1, 4), (9, 3, 5, 5)]
    shapes += [(rnd.choice([8, 9, 50, 333, 4001]), rnd.randint(1, 40), rnd.randint(1, 12), rnd.randint(1, 12)) for _ in range(200)]
    seen = 0
    for shape in shapes:
        for dtype, v in ((b.F32, 4), (b.BF16, 8)):
            n, c, inner = shape[0], shape[1], shape[2] * shape[3]
            for packed in (False, True):
                g = b.forward_geometry(dtype, shape, packed_mask=packed)
                ok = inner >= v and c * inner % v == 0 and (not packed or (c * inner % 8 == 0 and n * c * inner % 32 == 0))
                assert (g is not None) == ok
                if not ok:
                    continue
                seen += 1
                units, row = c * inner // v, g["side"] * (c * inner // v)
                lanes = lambda side: -(-side * units // 256) * 256
                assert g["columns"] * 256 == lanes(g["side"]) and 1 <= g["side"] <= n and (g["side"] == 1 or row <= 8192)
                assert (g["rows"] - 1) * row < n * units <= g["rows"] * row and 4 <= g["walk"] <= 16
                best = min(lanes(s) / (s * units) for s in range(1, max(1, min(n, 8192 // units)) + 1))
                assert lanes(g["side"]) / row <= max(16 / 15, best)
                # the thread of column u quantizes element u * v of a row, in channel (u * v // inner) % c
                u = rnd.randrange(row)
                at = rnd.randrange(g["rows"]) * row + u
                if at < n * units:
                    assert at * v // inner % c == u * v // inner % c
    assert seen > 100
