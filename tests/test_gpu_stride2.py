"""16-bit 3x3 layers of stride 2, whose channel blocks come in two activation stages (even and odd input rows): odd and even
sides, one row or column, 64-byte rows (32 channels and fewer), ragged channels and filters, one and several channel blocks,
few tiles (cut along K), many tiles a CTA, and a shared launch."""
import pytest
import torch

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from oracle import rtoss_oracle as orc
    from paper_2303_02191_b200 import binding as rt
    from paper_2303_02191_b200 import synth
    import gpu_util as gu

TOL = {"bf16": 2 ** -7, "f16": 2 ** -10}   # one unit in the last place of the result (7 and 10 bits behind the leading one)


@pytest.mark.parametrize("N,Cin,Cout,H,W,dt", [
    (1, 32, 64, 1, 1, "bf16"), (2, 32, 64, 40, 56, "bf16"), (1, 16, 24, 9, 200, "f16"), (1, 64, 128, 21, 33, "bf16"), (2, 72, 200, 14, 15, "f16"),
    (1, 128, 256, 2, 40, "bf16"), (1, 512, 512, 14, 22, "bf16"), (4, 128, 128, 80, 80, "bf16"), (16, 64, 128, 64, 64, "f16"), (3, 100, 75, 35, 51, "f16"),
])
def test_against_the_oracle(N, Cin, Cout, H, W, dt):
    masks = orc.pattern_preset(4, orc.PRESET_CENTRE8)
    x = synth.round_like(synth.activations(92, Cin + H, N, Cin, H, W), dt)
    w = synth.kaiming_weights(92, Cin + H, Cout, Cin, 3)
    _, packed = gu.select_pack(w, 3, masks, 4, dt)
    _, wd, _ = gu.oracle_weights(w, 3, masks, 4, dt)
    y = gu.run_conv(packed, 3, x, dt, 2, "none", None, "nhwc")
    assert orc.rel_err(y, gu.oracle_conv(3, x, wd, None, 2, "none", dt)) <= TOL[dt]
    assert gu.ctx().rtoss_device_status() == 0
    packed.close()


def test_shared_launch():
    c = gu.ctx()
    masks = orc.pattern_preset(4, orc.PRESET_CENTRE8)
    w = synth.kaiming_weights(92, 1, 128, 128, 3)
    _, packed = gu.select_pack(w, 3, masks, 4, "bf16")
    _, wd, _ = gu.oracle_weights(w, 3, masks, 4, "bf16")
    items, keep = [], []
    for i, (h, w_) in enumerate([(50, 68), (25, 34), (13, 17)]):
        x = synth.round_like(synth.activations(92, 50 + i, 2, 128, h, w_), "bf16")
        xd = gu.to_dev(x, "bf16", "nhwc")
        yd = torch.empty(2, (h + 1) // 2, (w_ + 1) // 2, 128, dtype=torch.bfloat16, device="cuda")
        items.append(c.conv_item(packed, xd, yd, 2, h, w_, 2, rt.NHWC, rt.ACT_RELU, None))
        keep.append((x, xd, yd))
    assert c.rtoss_conv_group(items) == 1
    torch.cuda.synchronize()
    for x, xd, yd in keep:
        assert orc.rel_err(gu.from_dev(yd, "nhwc"), gu.oracle_conv(3, x, wd, None, 2, "relu", "bf16")) <= TOL["bf16"]
    assert c.rtoss_device_status() == 0
    packed.close()
