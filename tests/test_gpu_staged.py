"""Calls made large enough, with many filters or images and ragged edges, that they run on the kernels they name: the staged
kernels of the FMA path (small calls run on the few-outputs kernel instead), one case for every shape, stride, layout, kind of
staging and vector width of theirs that a call can reach; and 16-bit calls that take the layout pass.  Which kernel runs, and
the staging plan, are asked of the library and checked, the results compared with the oracle.  Tolerance: one rounding to the
16-bit type plus the SiLU's 2^-11; fp32 sums in another order."""
import pytest
import torch

from paper_2303_02191_b200 import binding as rt

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from oracle import rtoss_oracle as orc
    from paper_2303_02191_b200 import synth
    import gpu_util as gu

TOL = {"f32": 1e-5, "bf16": 2.0 ** -7 + 2.0 ** -10, "f16": 2.0 ** -10 + 2.0 ** -10}
NONE, NCHW, NHWC = 0, 1, 2     # rtoss_fma_plan's staging
# N, Cin, Cout, H, W, stride, type, layout -> pixels per lane, staging, vector bytes
STAGED_3x3 = [
    ((5, 5, 330, 9, 9, 1, "bf16", "nchw"), (4, NONE, 0)), ((5, 5, 130, 9, 34, 1, "f16", "nchw"), (4, NCHW, 4)),
    ((5, 5, 700, 7, 8, 1, "bf16", "nchw"), (4, NCHW, 8)), ((5, 5, 130, 9, 40, 1, "f16", "nchw"), (4, NCHW, 16)),
    ((5, 5, 1030, 7, 9, 1, "bf16", "nchw"), (8, NONE, 0)), ((5, 5, 258, 13, 34, 1, "f16", "nchw"), (8, NCHW, 4)),
    ((5, 5, 130, 13, 68, 1, "bf16", "nchw"), (8, NCHW, 8)), ((5, 5, 1030, 7, 8, 1, "f16", "nchw"), (8, NCHW, 16)),
    ((5, 5, 700, 7, 9, 2, "bf16", "nchw"), (4, NONE, 0)), ((5, 5, 330, 9, 34, 2, "f16", "nchw"), (4, NCHW, 4)),
    ((5, 5, 700, 7, 20, 2, "bf16", "nchw"), (4, NCHW, 8)), ((5, 5, 700, 7, 8, 2, "f16", "nchw"), (4, NCHW, 16)),
    ((5, 5, 1030, 7, 9, 2, "bf16", "nchw"), (8, NONE, 0)), ((5, 5, 1030, 7, 22, 2, "f16", "nchw"), (8, NCHW, 4)),
    ((5, 5, 1030, 7, 20, 2, "bf16", "nchw"), (8, NCHW, 8)), ((5, 5, 1030, 7, 8, 2, "f16", "nchw"), (8, NCHW, 16)),
    ((5, 5, 330, 9, 9, 1, "f32", "nchw"), (4, NCHW, 4)), ((5, 5, 130, 9, 34, 1, "f32", "nchw"), (4, NCHW, 8)),
    ((5, 5, 700, 7, 8, 1, "f32", "nchw"), (4, NCHW, 16)), ((5, 5, 1030, 7, 9, 1, "f32", "nchw"), (8, NCHW, 4)),
    ((5, 5, 258, 13, 34, 1, "f32", "nchw"), (8, NCHW, 8)), ((5, 5, 1030, 7, 8, 1, "f32", "nchw"), (8, NCHW, 16)),
    ((5, 5, 700, 7, 9, 2, "f32", "nchw"), (4, NONE, 0)), ((5, 5, 1030, 7, 9, 2, "f32", "nchw"), (8, NONE, 0)),
    ((5, 5, 330, 9, 9, 1, "bf16", "nhwc"), (4, NONE, 0)), ((1, 8, 330, 9, 9, 1, "f16", "nhwc"), (4, NHWC, 0)),
    ((5, 8, 1030, 7, 9, 1, "bf16", "nhwc"), (8, NHWC, 0)), ((5, 8, 130, 7, 9, 2, "f16", "nhwc"), (4, NHWC, 0)),
    ((5, 8, 1030, 7, 34, 2, "bf16", "nhwc"), (8, NHWC, 0)), ((1, 8, 330, 9, 9, 1, "f32", "nhwc"), (4, NHWC, 0)),
    ((5, 8, 1030, 7, 9, 1, "f32", "nhwc"), (8, NHWC, 0)), ((5, 8, 130, 7, 9, 2, "f32", "nhwc"), (4, NONE, 0)),
    ((4, 27, 1700, 5, 6, 1, "bf16", "nchw"), None), ((4, 21, 1700, 5, 7, 2, "f32", "nchw"), None), ((2, 72, 330, 9, 9, 1, "bf16", "nhwc"), None),
]
STAGED_1x1 = [(17, 13, 1003, 3, 5, 1, "f32", "nchw"), (17, 70, 1003, 5, 3, 2, "bf16", "nchw"), (17, 24, 1003, 4, 4, 1, "f16", "nhwc"), (18, 33, 1001, 3, 5, 1, "f32", "nhwc"),
              (21, 40, 1003, 4, 4, 1, "f32", "nchw")]


def _run(ks, call, path, act="silu"):
    N, Cin, Cout, H, W, S, dt, layout = call
    masks = orc.pattern_preset(4, orc.PRESET_CENTRE8)
    x = synth.round_like(synth.activations(53, Cin + Cout, N, Cin, H, W), dt)
    w = synth.kaiming_weights(53, Cin + Cout, Cout, Cin, ks)
    b = synth.bias(53, Cout, Cout)
    _, packed = gu.select_pack(w, ks, masks, 4, dt)
    _, wd, _ = gu.oracle_weights(w, ks, masks, 4, dt)
    y = gu.run_conv(packed, ks, x, dt, S, act, b, layout, 2, Cout + 3, path=path)
    assert orc.rel_err(y[:, 2:2 + Cout], gu.oracle_conv(ks, x, wd, b, S, act, dt)) <= TOL[dt]
    assert (y[:, :2] == 7.0).all() and (y[:, 2 + Cout:] == 7.0).all() and gu.ctx().rtoss_device_status() == 0
    packed.close()


def _route(ks, call, path):
    N, Cin, Cout, H, W, S, dt, layout = call
    return rt.rtoss_conv_route_of(N, H, W, S, ks, rt.NHWC if layout == "nhwc" else rt.NCHW, rt.DTYPE_NAMES[dt], Cin, Cout, path)


@pytest.mark.parametrize("call,plan", STAGED_3x3, ids=str)
def test_staged_3x3(call, plan):
    N, Cin, Cout, H, W, S, dt, layout = call
    assert _route(3, call, rt.PATH_FMA) == rt.ROUTE_STAGED
    p = rt.rtoss_fma_plan3x3(N, H, W, S, rt.NHWC if layout == "nhwc" else rt.NCHW, rt.DTYPE_NAMES[dt], Cin, Cout, 4)
    if plan:
        assert (p.pixels_per_lane, p.staging, p.vector_bytes if p.staging == NCHW else 0) == plan
    _run(3, call, rt.PATH_FMA)


@pytest.mark.parametrize("call", STAGED_1x1, ids=str)
def test_staged_1x1(call):
    assert _route(1, call, rt.PATH_FMA) == rt.ROUTE_STAGED
    _run(1, call, rt.PATH_FMA)


REPACKED = [
    (3, (19, 40, 20, 21, 30, 2, "f16", "nchw")),     # stride 2, four filter copies
    (3, (1, 57, 16, 1, 1, 1, "bf16", "nchw")),       # a single pixel
    (3, (17, 12, 24, 20, 31, 1, "f16", "nhwc")),     # four filter copies, 8-byte loads
    (1, (9, 64, 48, 25, 31, 1, "bf16", "nchw")),     # positions on M
    (1, (40, 61, 90, 14, 9, 2, "f16", "nhwc")),      # element loads, kept pixels only
    (1, (30, 7, 24, 30, 30, 1, "bf16", "nhwc")),
]


@pytest.mark.parametrize("act", ["none", "relu"])
@pytest.mark.parametrize("ks,call", REPACKED, ids=str)
def test_layout_pass(ks, call, act):
    assert _route(ks, call, rt.PATH_AUTO) == rt.ROUTE_TENSOR_REPACKED
    _run(ks, call, rt.PATH_AUTO, act)
