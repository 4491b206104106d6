"""What the tile planner's cost model must never do, over sizes from single pixels to large batches (host arithmetic):
launch more clusters than the device holds at once, change the order of a sum because of a residual operand, or give a
layer tiles it has no use for."""
import itertools

import pytest

from paper_2303_02191_b200 import binding as rt

BF16, F32 = rt.DTYPE_NAMES["bf16"], rt.DTYPE_NAMES["f32"]
MOST_CLUSTERS = {2: 74, 3: 40, 4: 32, 5: 20, 6: 20, 7: 15, 8: 15}


@pytest.mark.parametrize("dt", [BF16, F32])
@pytest.mark.parametrize("ks,S", [(1, 1), (1, 2), (3, 1), (3, 2)])
def test_splits(ks, S, dt):
    split = 0
    for N, (H, W), (Cin, Cout) in itertools.product((1, 4, 16), [(1, 1), (7, 11), (20, 20), (28, 44), (56, 88), (100, 136)],
                                                    [(64, 64), (128, 128), (256, 256), (512, 2048), (2048, 512)]):
        p = rt.rtoss_tensor_plan_of(N, H, W, S, ks, Cin, Cout, dt)
        q = rt.rtoss_tensor_plan_of(N, H, W, S, ks, Cin, Cout, dt, residual=True)
        assert p.eligible and q.eligible
        if not p.positions_on_m:
            assert p.split_k == q.split_k
        if p.split_k > 1:
            split += 1
            assert p.tiles <= MOST_CLUSTERS[p.split_k] and p.tiles * p.split_k <= 148
    assert split > 0


def test_small_layers_spread_over_the_chip_and_large_ones_fill_their_tiles():
    small = rt.rtoss_tensor_plan_of(1, 40, 40, 1, 1, 128, 128, BF16)
    assert small.tiles >= 28            # 1600 positions: not seven tiles of 240
    large = rt.rtoss_tensor_plan_of(16, 160, 160, 1, 1, 128, 128, BF16)
    assert large.positions > 192        # thousands of tiles: as many positions each as fit
