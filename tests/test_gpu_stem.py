"""The matrix-instruction kernel of three-channel stems (16-bit, channels last, stride 2, even rows): rows that end inside
a fragment, a warp's 32 pixels or at a fragment's edge, odd heights, filter counts that end inside a lane's eight, channel
slices that take 16-byte stores and slices that do not.  Tolerance: one rounding to the 16-bit type, plus the SiLU's 2^-11."""
import pytest
import torch

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from oracle import rtoss_oracle as orc
    from paper_2303_02191_b200 import synth
    import gpu_util as gu

ULP = {"bf16": 2.0 ** -7, "f16": 2.0 ** -10}


@pytest.mark.parametrize("dt,act", [("bf16", "silu"), ("f16", "relu"), ("bf16", "none")])
@pytest.mark.parametrize("shape", [(1, 32, 2, 2), (1, 8, 7, 2), (2, 40, 9, 34), (1, 35, 12, 64), (3, 32, 31, 66), (1, 64, 5, 130), (9, 32, 160, 322)],
                         ids=lambda s: "-".join(str(v) for v in s))
def test_stem(shape, dt, act):
    N, Cout, H, W = shape
    k, masks = 4, orc.pattern_preset(4, orc.PRESET_CENTRE8)
    x = synth.round_like(synth.activations(81, Cout, N, 3, H, W), dt)
    w = synth.kaiming_weights(81, Cout, Cout, 3, 3)
    b = synth.bias(81, Cout, Cout)
    _, packed = gu.select_pack(w, 3, masks, k, dt)
    _, wd, _ = gu.oracle_weights(w, 3, masks, k, dt)
    ref = gu.oracle_conv(3, x, wd, b, 2, act, dt)
    for off, stride in ((8, Cout + 16 + (-Cout) % 8), (3, Cout + 4)):
        y = gu.run_conv(packed, 3, x, dt, 2, act, b, "nhwc", off, stride)
        assert orc.rel_err(y[:, off:off + Cout], ref) <= ULP[dt] + (2.0 ** -10 if act == "silu" else 0.0)
        assert (y[:, :off] == 7.0).all() and (y[:, off + Cout:] == 7.0).all()
    packed.close()


@pytest.mark.parametrize("dt,handle", [("bf16", "f32"), ("f16", "bf16")])
@pytest.mark.parametrize("shape", [(1, 32, 2, 8), (2, 40, 9, 24), (1, 35, 7, 16), (1, 32, 5, 520), (1, 32, 4, 20)], ids=lambda s: "-".join(str(v) for v in s))
def test_handle_of_another_type(shape, dt, handle):
    """The general stem kernel: rows of whole 16-byte groups of eight pixels (the last case: not), the first and the last window
    of a row, odd heights.  fp32 weights are not rounded to the data's type: the oracle gets the handle's values."""
    N, Cout, H, W = shape
    k, masks = 4, orc.pattern_preset(4, orc.PRESET_CENTRE8)
    x = synth.round_like(synth.activations(82, Cout, N, 3, H, W), dt)
    w = synth.kaiming_weights(82, Cout, Cout, 3, 3)
    b = synth.bias(82, Cout, Cout)
    _, packed = gu.select_pack(w, 3, masks, k, handle)
    _, wd, _ = gu.oracle_weights(w, 3, masks, k, handle)
    ref = gu.oracle_conv(3, x, wd, b, 2, "silu", dt)
    for off, stride in ((8, Cout + 16 + (-Cout) % 8), (3, Cout + 4)):
        y = gu.run_conv(packed, 3, x, dt, 2, "silu", b, "nhwc", off, stride)
        assert orc.rel_err(y[:, off:off + Cout], ref) <= ULP[dt] + 2.0 ** -10
        assert (y[:, :off] == 7.0).all() and (y[:, off + Cout:] == 7.0).all()
    packed.close()
