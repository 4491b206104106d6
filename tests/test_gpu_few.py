"""The kernel for calls of few outputs (conv_few.cu): fewer channels than warps, shares of unequal length, more channels than a
warp expands at a time, maps that end inside a lane's pixels or a tile's rows, rows of whole vectors and not, filters that end
inside a group of four, both layouts and strides, channel slices, against the oracle.  fp32: the sums differ in their order
only (9 * 70 products: 2e-6 of the largest result); 16-bit: one rounding, plus the SiLU's 2^-11."""
import pytest
import torch

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from oracle import rtoss_oracle as orc
    from paper_2303_02191_b200 import binding as rt
    from paper_2303_02191_b200 import synth
    import gpu_util as gu

TOL = {"f32": 1e-5, "bf16": 2.0 ** -7 + 2.0 ** -10, "f16": 2.0 ** -10 + 2.0 ** -10}
# ks, N, Cin, Cout, H, W, stride
SHAPES = [(3, 1, 5, 3, 1, 1, 1), (3, 2, 8, 4, 7, 5, 2), (3, 1, 17, 9, 33, 6, 1), (3, 3, 70, 21, 9, 13, 2), (3, 1, 32, 32, 32, 32, 1), (3, 1, 9, 5, 3, 132, 1),
          (3, 2, 33, 6, 5, 4, 2), (3, 1, 8, 8, 21, 140, 2), (1, 1, 1, 1, 1, 1, 1), (1, 2, 7, 10, 6, 9, 2), (1, 1, 70, 33, 17, 8, 1), (1, 3, 130, 6, 3, 132, 2)]


@pytest.mark.parametrize("dt", ["f32", "bf16", "f16"])
@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "-".join(str(v) for v in s))
def test_few(shape, dt):
    ks, N, Cin, Cout, H, W, stride = shape
    k, masks = 4, orc.pattern_preset(4, orc.PRESET_CENTRE8)
    x = synth.round_like(synth.activations(51, Cin + Cout, N, Cin, H, W), dt)
    w = synth.kaiming_weights(51, Cin + Cout, Cout, Cin, ks)
    b = synth.bias(51, Cout, Cout)
    _, packed = gu.select_pack(w, ks, masks, k, dt)
    _, wd, _ = gu.oracle_weights(w, ks, masks, k, dt)
    ref = gu.oracle_conv(ks, x, wd, b, stride, "silu", dt)
    for layout in ("nchw", "nhwc"):
        y = gu.run_conv(packed, ks, x, dt, stride, "silu", b, layout, 2, Cout + 3, path=rt.PATH_FMA)
        assert orc.rel_err(y[:, 2:2 + Cout], ref) <= TOL[dt]
        assert (y[:, :2] == 7.0).all() and (y[:, 2 + Cout:] == 7.0).all()
    packed.close()
