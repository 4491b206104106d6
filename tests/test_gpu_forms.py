"""Kernel forms of the tensor path (conv_tc_forms.cuh): every kind x activation x split x residual x layout that has a form
of its own, at filter counts that end inside a quarter of 32 filters (whole 16-byte pieces, the last quarter partly
empty), against the oracle.  Tolerance: both sides round the result once (a residual behind the activation twice) to the
16-bit type, so they differ by at most one unit in the last place per rounding, plus the SiLU's 2^-11."""
import pytest
import torch

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from oracle import rtoss_oracle as orc
    from paper_2303_02191_b200 import binding as rt
    from paper_2303_02191_b200 import synth
    import gpu_util as gu

ULP = {"bf16": 2.0 ** -7, "f16": 2.0 ** -10}
SILU = 2.0 ** -10
# ks, Cin, Cout, H, W, stride: uncut 1x1 and 3x3, positions on M, cut along K (many channels, few tiles)
SHAPES = [(1, 64, 104, 20, 24, 1), (1, 512, 136, 9, 10, 1), (1, 48, 40, 17, 13, 2), (3, 64, 72, 12, 14, 1), (3, 256, 136, 8, 9, 1), (3, 32, 24, 15, 22, 2),
          (3, 32, 8, 9, 9, 1)]


@pytest.mark.parametrize("dt", ["bf16", "f16"])
@pytest.mark.parametrize("act", ["none", "relu", "silu"])
@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "-".join(str(v) for v in s))
def test_forms(shape, act, dt):
    ks, Cin, Cout, H, W, stride = shape
    N, k = 2, 4
    masks = orc.pattern_preset(k, orc.PRESET_CENTRE8)
    x = synth.round_like(synth.activations(91, Cin + Cout, N, Cin, H, W), dt)
    w = synth.kaiming_weights(91, Cin + Cout, Cout, Cin, ks)
    b = synth.bias(91, Cout, Cout)
    _, packed = gu.select_pack(w, ks, masks, k, dt)
    _, wd, _ = gu.oracle_weights(w, ks, masks, k, dt)
    c, tol = gu.ctx(), ULP[dt] + (SILU if act == "silu" else 0.0)
    for layout in ("nhwc", "nchw"):
        y = gu.run_conv(packed, ks, x, dt, stride, act, b, layout, 8, Cout + 16)
        assert orc.rel_err(y[:, 8:8 + Cout], gu.oracle_conv(ks, x, wd, b, stride, act, dt)) <= tol
        assert (y[:, :8] == 7.0).all() and (y[:, 8 + Cout:] == 7.0).all()
    if ks == 1 and Cout <= 64:
        packed.close()
        return   # (positions on M: no residual operand)
    # a residual in front of and behind the activation
    Ho, Wo = synth.out_hw(H, W, stride)
    r = synth.round_like(synth.activations(92, Cout, N, Cout, Ho, Wo), dt)
    rd, xd, bd = gu.to_dev(r, dt, "nhwc"), gu.to_dev(x, dt, "nhwc"), torch.from_numpy(b).cuda()
    fn = c.rtoss_conv3x3_pattern if ks == 3 else c.rtoss_conv1x1_pattern
    ACT = {"none": orc.ACT_NONE, "relu": orc.ACT_RELU, "silu": orc.ACT_SILU}
    for post in (False, True):
        yd = torch.empty((N, Ho, Wo, Cout), dtype=gu.TORCH_DT[dt], device="cuda")
        fn(packed, xd, yd, N, H, W, stride, rt.NHWC, rt.ACT_NAMES[act], bd, residual=rd, residual_after_act=post)
        torch.cuda.synchronize()
        conv = gu.oracle_conv(ks, x, wd, b, stride, act if post else "none", dt)
        ref = orc.add_act(conv, r, ACT["none" if post else act], gu.ORC_DT[dt])
        assert orc.rel_err(gu.from_dev(yd, "nhwc"), ref) <= 2 * tol, post
    assert c.rtoss_device_status() == 0
    packed.close()


@pytest.mark.parametrize("acts", [("relu", "relu"), ("none", "relu"), ("silu", "silu")])
@pytest.mark.parametrize("ks", [1, 3])
def test_shared_launch_forms(ks, acts):
    """Members that agree on the activation, members that do not."""
    c, masks = gu.ctx(), orc.pattern_preset(4, orc.PRESET_CENTRE8)
    items, keep = [], []
    for i, (act, Cout) in enumerate(zip(acts, (72, 136))):
        x = synth.round_like(synth.activations(93, i, 2, 64, 18, 20), "bf16")
        w = synth.kaiming_weights(93, i + 10 * ks, Cout, 64, ks)
        b = synth.bias(93, i, Cout)
        _, packed = gu.select_pack(w, ks, masks, 4, "bf16")
        _, wd, _ = gu.oracle_weights(w, ks, masks, 4, "bf16")
        xd, bd = gu.to_dev(x, "bf16", "nhwc"), torch.from_numpy(b).cuda()
        y = torch.full((2, 18, 20, Cout), 7.0, dtype=torch.bfloat16, device="cuda")
        items.append(c.conv_item(packed, xd, y, 2, 18, 20, 1, rt.NHWC, rt.ACT_NAMES[act], bd))
        keep.append((packed, xd, bd, y, gu.oracle_conv(ks, x, wd, b, 1, act, "bf16")))
    assert c.rtoss_conv_group(items) == 1
    torch.cuda.synchronize()
    for packed, _, _, y, ref in keep:
        assert orc.rel_err(gu.from_dev(y, "nhwc"), ref) <= ULP["bf16"] + SILU
        packed.close()
