"""fp32 3x3 layers of whole blocks of 32 channels: tf32 heads with bf16 corrections.  Error against 64-bit sums no larger than
three tf32 products left on the same inputs (measured, the bound of each case: what decides is the accumulation, which cuts
off a part of the sum per instruction, two thirds as often now; the two corrections' factors are rounded to 2^-9 of a term
that is 2^-12 of the product, 7e-7 in all); values near fp32's largest stay finite; the single-layer and the whole-model
packing give the same outputs, bit for bit."""
import math

import pytest
import torch

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_2303_02191_b200 import binding as rt
    import gpu_util as gu


def _layer(cin, cout, k, scale=1.0):
    c = gu.ctx()
    masks = rt.rtoss_pattern_preset(k, rt.PRESET_CENTRE8 if k == 4 else rt.PRESET_CONN4)
    g = torch.Generator(device="cuda")
    g.manual_seed(cin + cout)
    w = torch.randn(cout, cin, 3, 3, device="cuda", generator=g) * math.sqrt(2.0 / (9 * cin)) * scale
    pid = c.rtoss_select_patterns(w, 3, masks, k)
    return c, masks, g, w, pid, c.rtoss_pack(w, 3, masks, k, pid, rt.F32)


def _conv(c, packed, x, cout, stride):
    N, H, W, _ = x.shape
    y = torch.empty(N, (H - 1) // stride + 1, (W - 1) // stride + 1, cout, device="cuda")
    c.rtoss_conv3x3_pattern(packed, x, y, N, H, W, stride, rt.NHWC, rt.ACT_NONE, None, path=rt.PATH_TENSOR)
    torch.cuda.synchronize()
    assert c.rtoss_device_status() == 0
    return y


@pytest.mark.parametrize("cin,cout,H,W,stride,k,bound", [
    (32, 16, 9, 11, 1, 2, 2.31e-6), (32, 128, 33, 40, 1, 4, 2.69e-6), (96, 64, 21, 26, 1, 4, 6.27e-6), (64, 130, 15, 15, 2, 3, 2.54e-6),
    (256, 256, 20, 20, 1, 4, 2.65e-6), (256, 32, 7, 9, 2, 2, 1.20e-5), (128, 128, 60, 60, 2, 4, 2.71e-6), (512, 512, 14, 14, 1, 4, 4.36e-6)])
def test_error_against_64_bits(cin, cout, H, W, stride, k, bound):
    c, masks, g, w, pid, packed = _layer(cin, cout, k)
    x = torch.randn(2, H, W, cin, device="cuda", generator=g)
    y = _conv(c, packed, x, cout, stride)
    ref = torch.nn.functional.conv2d(x.double().cpu().permute(0, 3, 1, 2), packed.to_dense().double().cpu().reshape(w.shape), stride=stride, padding=1)
    e = y.double().cpu().permute(0, 3, 1, 2) - ref
    assert (e.norm() / ref.norm()).item() <= bound
    packed.close()


def test_large_values_stay_finite():
    c, masks, g, w, pid, packed = _layer(32, 32, 4, 1e-3)
    x = torch.randn(1, 8, 8, 32, device="cuda", generator=g)
    x[0, 4, 4, 5] = torch.finfo(torch.float32).max
    y = _conv(c, packed, x, 32, 1)
    ref = torch.nn.functional.conv2d(x.double().cpu().permute(0, 3, 1, 2), packed.to_dense().double().cpu().reshape(w.shape), padding=1)
    d = (y.double().cpu().permute(0, 3, 1, 2) - ref).abs()
    assert torch.isfinite(y).all() and (d <= 1e-4 * ref.abs().clamp(min=ref.abs().median().item())).all()
    packed.close()


@pytest.mark.parametrize("cin,cout", [(32, 32), (64, 50), (96, 130), (36, 40)])   # (36: the layers that keep fp32 remainders)
def test_both_ways_of_packing(cin, cout):
    c, masks, g, w, pid, packed = _layer(cin, cout, 4)
    x = torch.randn(1, 13, 17, cin, device="cuda", generator=g)
    y0 = _conv(c, packed, x, cout, 1)
    batch = c.rtoss_batch_create([dict(w=w, ksize=3, masks=masks, k=4, packed=packed)])
    batch.rtoss_batch_select_pack()
    assert torch.equal(y0, _conv(c, packed, x, cout, 1))
    batch.close()
    packed.close()


def _error(N, cin, cout, H, W, stride, k, patterns, relu):
    c = gu.ctx()
    masks = rt.rtoss_pattern_preset(k, rt.PRESET_CENTRE8 if k == 4 else rt.PRESET_CONN4)
    g = torch.Generator(device="cuda")
    g.manual_seed(cin + cout + H + W)
    w = torch.randn(cout, cin, 3, 3, device="cuda", generator=g) * math.sqrt(2.0 / (9 * cin))
    pid = c.rtoss_select_patterns_shared(w, masks, k, 128, 16) if patterns == "block" else c.rtoss_select_patterns(w, 3, masks, k)
    packed = c.rtoss_pack(w, 3, masks, k, pid, rt.F32)
    x = torch.randn(N, H, W, cin, device="cuda", generator=g)
    if relu:
        x = torch.relu(x)
    y = _conv(c, packed, x, cout, stride)
    ref = torch.nn.functional.conv2d(x.double().permute(0, 3, 1, 2), packed.to_dense().double().reshape(w.shape), stride=stride, padding=1)
    packed.close()
    return ((y.double().permute(0, 3, 1, 2) - ref).norm() / ref.norm()).item()


ERRORS = [   # N, channels, filters, H, W, stride, k, patterns, input after a ReLU, the error of three tf32 products
    (3, 96, 360, 42, 33, 1, 4, "kernel", True, 3.31e-6),
    (27, 96, 73, 11, 24, 1, 4, "kernel", False, 3.89e-6),
    (2, 416, 78, 19, 37, 1, 3, "kernel", True, 3.42e-6),
    (2, 480, 328, 12, 13, 2, 2, "kernel", False, 3.72e-6),
    (1, 32, 16, 9, 11, 1, 2, "block", False, 1.02e-6),
    (4, 32, 28, 76, 20, 2, 2, "block", True, 1.00e-6),
    (2, 32, 70, 57, 10, 1, 2, "block", True, 0.95e-6),
    (1, 96, 162, 16, 30, 1, 2, "block", True, 1.00e-6),
    (2, 256, 64, 40, 40, 1, 2, "block", False, 4.30e-6),
    (2, 256, 64, 40, 40, 1, 3, "block", True, 6.06e-6),
    (1, 256, 256, 20, 20, 1, 3, "block", False, 1.35e-6),
    (5, 96, 160, 20, 86, 2, 4, "block", True, 2.19e-6),
]


@pytest.mark.parametrize("N,cin,cout,H,W,stride,k,patterns,relu,bound", ERRORS)
def test_error_no_larger_than_of_three_products(N, cin, cout, H, W, stride, k, patterns, relu, bound):
    """Layers cut along K in several ways (the longer a share, the larger the error), and block patterns of few kept taps and channels,
    where the fewest accumulations stand against the rounded factors."""
    assert _error(N, cin, cout, H, W, stride, k, patterns, relu) <= bound
