"""Launches whose weights stay in shared memory from tile to tile: one and several filter tiles (a grid that is a multiple of
their number), positions on M, repeated filters, a residual operand, fp32, behind a layout pass -- a batch that gives a CTA
several tiles against the same images one by one, which gives it one.  Tolerance: one rounding to the data type (a layer of
one image may be cut along K, which sums in another order)."""
import pytest
import torch

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from oracle import rtoss_oracle as orc
    from paper_2303_02191_b200 import binding as rt
    from paper_2303_02191_b200 import synth
    import gpu_util as gu

TOL = {"bf16": 2.0 ** -7, "f16": 2.0 ** -10, "f32": 2.0 ** -18}
# ks, N, Cin, Cout, H, W, stride, dtype, residual
SHAPES = [(1, 8, 64, 64, 80, 80, 1, "bf16", False), (1, 6, 128, 384, 50, 68, 1, "bf16", False), (1, 6, 64, 256, 56, 100, 1, "f16", True), (1, 6, 128, 136, 160, 120, 2, "bf16", False),
          (3, 8, 24, 24, 60, 60, 1, "bf16", False), (3, 8, 32, 64, 100, 100, 2, "f16", False), (1, 8, 32, 128, 80, 60, 1, "f32", False), (1, 8, 70, 136, 60, 80, 1, "bf16", False)]


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "-".join(str(v) for v in s))
def test_batch_against_single_images(shape):
    ks, N, Cin, Cout, H, W, stride, dt, res = shape
    c = gu.ctx()
    w = synth.kaiming_weights(31, Cin + Cout, Cout, Cin, ks)
    _, packed = gu.select_pack(w, ks, orc.pattern_preset(4, orc.PRESET_CENTRE8), 4, dt)
    b = torch.from_numpy(synth.bias(31, Cout, Cout)).cuda()
    g = torch.Generator(device="cuda").manual_seed(5)
    Ho, Wo = synth.out_hw(H, W, stride)
    x = torch.empty((N, H, W, Cin), device="cuda").normal_(generator=g).to(gu.TORCH_DT[dt])
    r = torch.empty((N, Ho, Wo, Cout), device="cuda").normal_(generator=g).to(gu.TORCH_DT[dt]) if res else None
    fn = c.rtoss_conv3x3_pattern if ks == 3 else c.rtoss_conv1x1_pattern
    y, one = torch.empty((N, Ho, Wo, Cout), dtype=x.dtype, device="cuda"), torch.empty((N, Ho, Wo, Cout), dtype=x.dtype, device="cuda")
    fn(packed, x, y, N, H, W, stride, rt.NHWC, rt.ACT_RELU, b, residual=r)
    for n in range(N):
        fn(packed, x[n], one[n], 1, H, W, stride, rt.NHWC, rt.ACT_RELU, b, residual=r[n] if res else None)
    torch.cuda.synchronize()
    assert c.rtoss_device_status() == 0
    assert ((y - one).abs().max() / one.abs().max()).item() <= TOL[dt] * (2 if res else 1)
    assert y.abs().max() > 0
    packed.close()
