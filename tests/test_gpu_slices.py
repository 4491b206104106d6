"""Input slices and pools inside one tensor: a convolution that reads a channel slice gives the bits it gives on a dense copy
of the slice (the same operands in the same order), in place along a residual chain too; up-sampling from a slice and the
chained pools give the bits of the calls they stand for; what takes no slice says so."""
import pytest
import torch

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from oracle import rtoss_oracle as orc
    from paper_2303_02191_b200 import binding as rt
    from paper_2303_02191_b200 import synth
    import gpu_util as gu


def _layer(ks, Cin, Cout, dt, seed):
    w = synth.kaiming_weights(seed, Cin + Cout, Cout, Cin, ks)
    return gu.select_pack(w, ks, orc.pattern_preset(4, orc.PRESET_CENTRE8), 4, dt)[1], torch.from_numpy(synth.bias(seed, Cout, Cout)).cuda()


@pytest.mark.parametrize("dt", ["bf16", "f16", "f32"])
@pytest.mark.parametrize("shape", [(1, 64, 40, 17, 13, 1), (1, 512, 136, 9, 10, 1), (1, 48, 72, 11, 14, 2), (3, 32, 64, 15, 22, 2), (3, 256, 136, 8, 9, 1), (3, 72, 24, 10, 12, 1)],
                         ids=lambda s: "-".join(str(v) for v in s))
def test_conv_reads_a_slice(shape, dt):
    ks, Cin, Cout, H, W, stride = shape
    N, c = 2, gu.ctx()
    packed, b = _layer(ks, Cin, Cout, dt, 61)
    fn = c.rtoss_conv3x3_pattern if ks == 3 else c.rtoss_conv1x1_pattern
    wide = torch.full((N, H, W, Cin + 24), float("nan"), dtype=gu.TORCH_DT[dt], device="cuda")   # (what lies beside the slice is not read)
    x = gu.to_dev(synth.round_like(synth.activations(61, Cin, N, Cin, H, W), dt), dt, "nhwc")
    wide[..., 8:8 + Cin] = x
    Ho, Wo = synth.out_hw(H, W, stride)
    ys = [torch.empty((N, Ho, Wo, Cout), dtype=gu.TORCH_DT[dt], device="cuda") for _ in range(2)]
    fn(packed, x, ys[0], N, H, W, stride, rt.NHWC, rt.ACT_SILU, b, path=rt.PATH_TENSOR)
    fn(packed, wide[..., 8:], ys[1], N, H, W, stride, rt.NHWC, rt.ACT_SILU, b, x_channel_stride=Cin + 24)
    torch.cuda.synchronize()
    assert torch.equal(ys[0], ys[1]) and c.rtoss_device_status() == 0
    with pytest.raises(rt.RtossError) as e:
        fn(packed, wide[..., 8:], ys[1], N, H, W, stride, rt.NHWC, rt.ACT_SILU, b, path=rt.PATH_FMA, x_channel_stride=Cin + 24)
    assert e.value.status == rt.ERR_UNSUPPORTED
    with pytest.raises(rt.RtossError):
        fn(packed, wide[..., 8:], ys[1], N, H, W, stride, rt.NHWC, rt.ACT_SILU, b, x_channel_stride=Cin - 8)
    packed.close()


def test_bottleneck_in_place():
    """A bottleneck whose input and result are the same slice of a concatenation."""
    N, C, H, W, c = 2, 64, 18, 20, gu.ctx()
    (p1, b1), (p2, b2) = _layer(1, C, C, "bf16", 62), _layer(3, C, C, "bf16", 63)
    x = gu.to_dev(synth.round_like(synth.activations(62, C, N, C, H, W), "bf16"), "bf16", "nhwc")
    cat = torch.full((N, H, W, 2 * C), 7.0, dtype=torch.bfloat16, device="cuda")
    cat[..., :C] = x
    t, y = torch.empty_like(x), torch.empty_like(x)
    c.rtoss_conv1x1_pattern(p1, x, t, N, H, W, 1, rt.NHWC, rt.ACT_SILU, b1)
    c.rtoss_conv3x3_pattern(p2, t, y, N, H, W, 1, rt.NHWC, rt.ACT_SILU, b2, residual=x, residual_after_act=True)
    c.rtoss_conv1x1_pattern(p1, cat, t, N, H, W, 1, rt.NHWC, rt.ACT_SILU, b1, x_channel_stride=2 * C)
    c.rtoss_conv3x3_pattern(p2, t, cat, N, H, W, 1, rt.NHWC, rt.ACT_SILU, b2, 0, 2 * C, residual=cat, residual_after_act=True)
    torch.cuda.synchronize()
    assert torch.equal(cat[..., :C], y) and (cat[..., C:] == 7.0).all()
    p1.close(), p2.close()


@pytest.mark.parametrize("dt", ["bf16", "f16"])
@pytest.mark.parametrize("shape", [(2, 16, 20, 20, 5), (1, 8, 3, 4, 5), (3, 24, 1, 1, 3), (1, 8, 80, 80, 5)], ids=lambda s: "-".join(str(v) for v in s))
def test_pools_and_upsampling_inside_a_tensor(shape, dt):
    N, C, H, W, k = shape
    x = gu.to_dev(synth.round_like(synth.activations(64, C, N, C, H, W), dt), dt, "nhwc")
    x.view(-1)[3] = float("nan")
    x.view(-1)[C * H * W // 2] = -0.0
    y = torch.full((N, H, W, 4 * C + 24), 7.0, dtype=gu.TORCH_DT[dt], device="cuda")
    y[..., 8:8 + C] = x
    rt.rtoss_pool_pyramid(y, N, C, H, W, k, rt.NHWC, 8, 4 * C + 24)
    ref = x
    for i in range(4):
        assert torch.equal(y[..., 8 + i * C:8 + (i + 1) * C].contiguous().view(torch.int16), ref.view(torch.int16)), i
        ref = rt.rtoss_maxpool2d(ref, torch.empty_like(x), N, C, H, W, k, 1, k // 2, rt.NHWC)
    assert (y[..., :8] == 7.0).all() and (y[..., 8 + 4 * C:] == 7.0).all()
    for layout in (rt.NHWC,):
        up = [torch.empty((N, 2 * H, 2 * W, C), dtype=x.dtype, device="cuda") for _ in range(2)]
        rt.rtoss_upsample2x(x, up[0], N, C, H, W, layout)
        rt.rtoss_upsample2x_slice(y[..., 8:], 4 * C + 24, up[1], N, C, H, W, layout)
        assert torch.equal(up[0].view(torch.int16), up[1].view(torch.int16))


def test_pools_decline():
    y = torch.zeros((1, 81, 80, 32), dtype=torch.bfloat16, device="cuda")
    for args in ((1, 8, 81, 80, 5, rt.NHWC, 0, 32), (1, 4, 8, 8, 5, rt.NHWC, 0, 32), (1, 8, 8, 8, 5, rt.NCHW, 0, 32)):
        with pytest.raises(rt.RtossError) as e:
            rt.rtoss_pool_pyramid(y, *args)
        assert e.value.status == rt.ERR_UNSUPPORTED
