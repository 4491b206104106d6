"""Host logic of the tensor path's tile planner (rtoss_tensor_plan_of: plain arithmetic through the C ABI, no GPU):
the invariants the kernel and the TMA descriptors rely on, over the layer shapes of both model families and a sweep of
odd ones."""
import ctypes
import itertools
import random
import time

import pytest

from paper_2303_02191_b200 import binding as rt
from paper_2303_02191_b200 import synth

BF16, F16, F32 = rt.DTYPE_NAMES["bf16"], rt.DTYPE_NAMES["f16"], rt.DTYPE_NAMES["f32"]
CAP = 227 * 1024


def check(N, H, W, S, ks, Cin, Cout, dt, residual=False):
    p = rt.rtoss_tensor_plan_of(N, H, W, S, ks, Cin, Cout, dt, residual=residual)
    es = 4 if dt == F32 else 2
    if not p.eligible:
        return p
    Ho, Wo = synth.out_hw(H, W, S)
    if ks == 1 and S == 1:      # cut as one row of all pixels
        N, Ho, Wo = 1, 1, N * H * W
    halo = (2 if S == 1 else 1) if ks == 3 else 0
    assert p.shared_bytes <= CAP
    assert 16 <= p.positions <= 256 and p.positions % 16 == 0
    assert p.pitch == p.cols_per_tile + halo and p.rows_per_tile * p.pitch <= p.positions
    assert p.staged_rows == p.rows_per_tile + halo
    # a TMA box traverses at most 256 elements per dimension (stride-2 boxes traverse every second one)
    assert p.pitch * S <= 256 and p.staged_rows * S <= 256
    assert p.row_bytes == (64 if (dt != F32 and Cin <= 32) else 128)
    # stage sizes are multiples of the swizzle atom (8 rows), so every stage starts on an atom boundary
    assert p.act_stage_bytes % (8 * p.row_bytes) == 0 and p.weight_stage_bytes % (8 * p.row_bytes) == 0
    assert p.sub_tiles == (4 if (ks == 3 and S == 2) else 1)
    assert 1 <= p.act_stages <= 4 and 1 <= p.weight_stages <= 8
    if p.weight_stages < 2:     # all weights of a tile stay in shared memory: its one stage, and more tiles than CTAs
        ncb_ = -(-Cin // (p.row_bytes // es))
        assert ncb_ * (ks * ks * (2 if dt == F32 else 1) // p.taps_per_weight_stage) == 1 and p.tiles > 148 - 148 % (1 if p.positions_on_m else -(-Cout // 128))
    assert p.taps_per_weight_stage in ((1, 3) if ks == 3 else (1,))
    assert p.act_stages * p.act_stage_bytes + p.weight_stages * p.weight_stage_bytes < p.shared_bytes
    # the tiles cover the output
    tiles_y = -(-Ho // p.rows_per_tile)
    tiles_x = -(-Wo // p.cols_per_tile)
    co_tiles = 1 if p.positions_on_m else -(-Cout // 128)
    assert p.tiles == N * tiles_y * tiles_x * co_tiles
    assert p.positions_on_m == (1 if (ks == 1 and Cout <= 64 and dt != F32) else 0)
    cb_ch = p.row_bytes // es
    ncb = -(-Cin // cb_ch)
    assert 1 <= p.split_k <= min(8, ncb)
    if p.split_k > 1:
        assert p.tiles * 2 <= 148 and not p.positions_on_m
    return p


def test_every_layer_of_both_model_families():
    for N, layers in ((16, synth.yolov5s_stack()), (1, synth.yolov5s_stack()), (4, synth.retinanet_r50fpn_stack())):
        for L in layers:
            if L["cin"] % 8:
                continue
            p = check(N, L["H"], L["W"], L["stride"], L["ksize"], L["cin"], L["cout"], BF16)
            assert p.eligible, L["name"]


def test_odd_shapes_and_types():
    for (H, W), S, ks, (Cin, Cout), dt in itertools.product(
            [(1, 1), (7, 9), (13, 255), (64, 64), (5, 700), (200, 272), (3, 2000)], (1, 2), (1, 3),
            [(8, 8), (24, 20), (32, 32), (40, 80), (64, 48), (72, 200), (256, 256), (2048, 512)], (BF16, F16, F32)):
        check(2, H, W, S, ks, Cin, Cout, dt)
        check(1, H, W, S, ks, Cin, Cout, dt, residual=True)


def test_ineligible_shapes_and_bad_arguments():
    assert not rt.rtoss_tensor_plan_of(1, 8, 8, 1, 3, 12, 16, BF16).eligible      # rows of 24 bytes: not a multiple of 16
    assert not rt.rtoss_tensor_plan_of(1, 8, 8, 1, 3, 6, 16, F32).eligible
    assert not rt.rtoss_tensor_plan_of(1, 8, 8, 1, 3, 64, 64, BF16, layout=rt.NCHW).eligible
    for bad in ((0, 8, 8, 1, 3, 64, 64), (1, 8, 8, 3, 3, 64, 64), (1, 8, 8, 1, 2, 64, 64), (1, 8, 8, 1, 3, 0, 64)):
        with pytest.raises(rt.RtossError):
            rt.rtoss_tensor_plan_of(*bad, BF16)


@pytest.mark.parametrize("N,H,W", [(1, 1, 1), (1, 20, 20), (4, 50, 68), (3, 7, 300), (16, 160, 160), (2, 5, 700)])
@pytest.mark.parametrize("Cin,Cout", [(64, 64), (256, 1024), (72, 200), (2048, 512)])
def test_rows_of_all_pixels(N, H, W, Cin, Cout):
    """1x1 layers of stride 1: the plan of the images is the plan of one row of their pixels, tiles of one row, as many positions
    as they have pixels (rounded up to 16)."""
    p = check(N, H, W, 1, 1, Cin, Cout, BF16)
    q = check(1, 1, N * H * W, 1, 1, Cin, Cout, BF16)
    assert p.eligible and all(getattr(p, f) == getattr(q, f) for f, _ in p._fields_)
    assert p.rows_per_tile == 1 and p.positions == -(-p.cols_per_tile // 16) * 16


def test_weights_that_stay():
    p = check(16, 160, 160, 1, 1, 64, 64, BF16)       # one stage of weights, thousands of tiles
    assert p.weight_stages == 1 and p.act_stages >= 3
    q = check(4, 100, 136, 1, 1, 512, 256, BF16)      # eight stages do not fit beside three activation stages
    assert q.act_stages * q.act_stage_bytes + q.weight_stages * q.weight_stage_bytes <= q.shared_bytes


def test_narrow_layers_stage_half_rows_and_keep_a_deeper_ring():
    p = check(16, 160, 160, 1, 3, 32, 32, BF16)
    assert p.row_bytes == 64 and p.act_stages > 2        # one channel block per tile: the next tile's block is the next stage
    q = check(16, 160, 160, 1, 3, 128, 128, BF16)
    assert q.row_bytes == 128 and q.act_stages == 2


def _random_call(rng, stride):
    d = rt.ConvDesc(rng.randint(1, 32), rng.randint(7, 160), rng.randint(7, 160), stride, rt.NHWC, BF16, 0, None, 0, 0, 0, None, 0)
    return ctypes.byref(d), 3, 8 * rng.randint(2, 64), 8 * rng.randint(2, 64), BF16, 0, ctypes.byref(rt.TensorPlan())


def _fastest(calls, passes):
    """Nanoseconds of each call, the fastest of its repeats; the calls take turns."""
    best = [1 << 60] * len(calls)
    for _ in range(passes):
        for i, args in enumerate(calls):
            t = time.perf_counter_ns()
            rt.lib.rtoss_tensor_plan_of(*args)
            best[i] = min(best[i], time.perf_counter_ns() - t)
    return best


def _again_if_slow(calls, passes, usual):
    """The slowest call, measured again up to six times while it takes three times the usual: the machine may have been busy
    elsewhere, while a call that is planned again is slow every time."""
    for _ in range(6):
        slowest = max(_fastest(calls, passes))
        if slowest <= 3 * usual:
            break
        time.sleep(0.02)
    return slowest


def test_a_repeated_call_is_not_planned_again():
    """Planning searches for tens of microseconds; a thread remembers its plans, and a call looks up one key, so asking twice in a
    row never searches twice.  A thousand random layers of stride 2 against their median."""
    rng = random.Random(6)
    calls = [_random_call(rng, 2) for _ in range(1000)]
    took = [_fastest([c], 40)[0] for c in calls]
    usual = sorted(took)[500]
    assert all(t <= 3 * usual or _again_if_slow([c], 40, usual) <= 3 * usual for c, t in zip(calls, took))


def test_fifty_calls_in_turn_are_not_planned_again():
    """As many plans as a grouped call looks up: asked for one after the other, over and over, none of them is searched twice.
    Twenty sets of fifty layers against their median."""
    rng = random.Random(7)
    for _ in range(20):
        calls = [_random_call(rng, 1) for _ in range(50)]
        usual = sorted(_fastest(calls, 20))[25]
        assert _again_if_slow(calls, 20, usual) <= 3 * usual


@pytest.mark.parametrize("dtype,ksize,cin,units", [("bf16", 3, 64, 1), ("f16", 1, 36, 1), ("f32", 3, 64, 4), ("f32", 3, 36, 6), ("f32", 1, 64, 6)])
def test_tensor_time_of_a_product(dtype, ksize, cin, units):
    """What the rooflines of bench.py and the sweep divide the tensor peak by, and that both have a name for it."""
    assert synth.tensor_units(dict(ksize=ksize, cin=cin), dtype) == units and units in synth.TENSOR_BOUND
