"""Element-store forms of the tensor path: filter counts of no multiple of eight, unaligned channel slices, 1x1 and 3x3, cut
along K and not, native and behind a layout pass, against the oracle (one rounding to the 16-bit type, plus the SiLU's 2^-11)."""
import pytest
import torch

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from oracle import rtoss_oracle as orc
    from paper_2303_02191_b200 import synth
    import gpu_util as gu

ULP = {"bf16": 2.0 ** -7, "f16": 2.0 ** -10}
# ks, N, Cin, Cout, H, W, stride
SHAPES = [(1, 2, 128, 75, 23, 21, 1), (1, 2, 70, 131, 23, 21, 1), (1, 1, 512, 250, 6, 7, 1), (1, 2, 72, 129, 9, 12, 2), (3, 3, 64, 75, 20, 22, 1), (3, 2, 100, 33, 40, 31, 1),
          (3, 1, 256, 250, 7, 9, 1), (3, 1, 250, 129, 9, 8, 2), (3, 2, 64, 17, 30, 31, 1)]


@pytest.mark.parametrize("dt", ["bf16", "f16"])
@pytest.mark.parametrize("act", ["none", "relu", "silu"])
@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "-".join(str(v) for v in s))
def test_ragged(shape, act, dt):
    ks, N, Cin, Cout, H, W, stride = shape
    masks = orc.pattern_preset(4, orc.PRESET_CENTRE8)
    x = synth.round_like(synth.activations(41, Cin + Cout, N, Cin, H, W), dt)
    w = synth.kaiming_weights(41, Cin + Cout, Cout, Cin, ks)
    b = synth.bias(41, Cout, Cout)
    _, packed = gu.select_pack(w, ks, masks, 4, dt)
    _, wd, _ = gu.oracle_weights(w, ks, masks, 4, dt)
    ref, tol = gu.oracle_conv(ks, x, wd, b, stride, act, dt), ULP[dt] + (2.0 ** -10 if act == "silu" else 0.0)
    for off, cs in ((0, Cout), (3, Cout + 5)):
        y = gu.run_conv(packed, ks, x, dt, stride, act, b, "nhwc", off, cs)
        assert orc.rel_err(y[:, off:off + Cout], ref) <= tol
        assert (y[:, :off] == 7.0).all() and (y[:, off + Cout:] == 7.0).all()
    assert gu.ctx().rtoss_device_status() == 0
    packed.close()
