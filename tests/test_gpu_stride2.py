"""16-bit 3x3 layers of stride 2.  The first two tests: odd and even sides, one row or column, 64-byte rows (32 channels and
fewer), ragged channels and filters, one and several channel blocks, cut along K, a shared launch; the planner takes them
with a channel block in one activation stage.  The others: layers whose channel blocks come in two activation stages (odd and
even input rows), which the plan is asked to confirm; a call adds up in the order of a shared launch, which has one stage, so
uncut ones give its bits."""
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


def _two_stages(N, H, W, Cin, Cout, dt, residual=False):
    """(in two stages?, stages, shares) by the plan: the bytes of an activation stage against those of its sub-tiles."""
    p = rt.rtoss_tensor_plan_of(N, H, W, 2, 3, Cin, Cout, rt.DTYPE_NAMES[dt], residual=residual)
    sub = (max(p.positions + p.pitch + 1, p.staged_rows * p.pitch) + 7) // 8 * 8 * p.row_bytes
    return p.act_stage_bytes == 2 * sub, p.act_stages, p.split_k


def _layer(N, Cin, Cout, H, W, dt, patterns, k=4):
    c = gu.ctx()
    masks = rt.rtoss_pattern_preset(k, rt.PRESET_CENTRE8 if k == 4 else rt.PRESET_CONN4)
    g = torch.Generator(device="cuda")
    g.manual_seed(Cin + Cout + H)
    w = torch.randn(Cout, Cin, 3, 3, device="cuda", generator=g) * (2.0 / (9 * Cin)) ** 0.5
    pid = c.rtoss_select_patterns_shared(w, masks, k, 128, 16) if patterns == "block" else c.rtoss_select_patterns(w, 3, masks, k)
    packed = c.rtoss_pack(w, 3, masks, k, pid, rt.DTYPE_NAMES[dt])
    x = torch.randn(N, H, W, Cin, device="cuda", generator=g).to(gu.TORCH_DT[dt])
    bias = torch.randn(Cout, device="cuda", generator=g) * 0.1
    return c, packed, x, bias, g


def _exact(packed, x, bias, act):
    w = packed.to_dense().double().reshape(packed.info.Cout, packed.info.Cin, 3, 3)
    y = torch.nn.functional.conv2d(x.double().permute(0, 3, 1, 2), w, bias.double(), stride=2, padding=1).permute(0, 2, 3, 1)
    return {"none": lambda v: v, "relu": torch.relu, "silu": torch.nn.functional.silu}[act](y)


def _near(y, ref, dt, act="none"):
    """Within a unit, and SiLU's approximation: tanh to 2^-11 of itself, times half of an input of up to 5.5
    deviations, against the 0.6 that the result's root mean square is of a deviation."""
    bound = TOL[dt] + (2 ** -11 * 5.5 / 2 / 0.6 if act == "silu" else 0)
    return ((y.double() - ref).abs() / torch.maximum(ref.abs(), ref.pow(2).mean().sqrt())).max().item() <= bound


UNCUT = [   # N, Cin, Cout, H, W, dtype, activation, stages
    (10, 64, 16, 116, 55, "bf16", "none", 2), (11, 40, 16, 51, 130, "f16", "relu", 2), (8, 64, 16, 131, 26, "f16", "silu", 3),
    (31, 56, 16, 33, 36, "bf16", "silu", 3), (18, 16, 16, 125, 125, "bf16", "relu", 3),                # (64-byte rows, resident weights)
    (15, 160, 216, 79, 62, "bf16", "relu", 2), (8, 96, 128, 80, 80, "f16", "none", 3), (9, 416, 208, 71, 84, "bf16", "none", 3),
]


@pytest.mark.parametrize("patterns", ["kernel", "block"])
@pytest.mark.parametrize("N,Cin,Cout,H,W,dt,act,stages", UNCUT)
def test_two_stages_give_the_bits_of_one(N, Cin, Cout, H, W, dt, act, stages, patterns):
    assert _two_stages(N, H, W, Cin, Cout, dt) == (True, stages, 1)
    c, packed, x, bias, _ = _layer(N, Cin, Cout, H, W, dt, patterns)
    y = [torch.empty(N, (H + 1) // 2, (W + 1) // 2, Cout, dtype=x.dtype, device="cuda") for _ in range(3)]
    c.rtoss_conv3x3_pattern(packed, x, y[0], N, H, W, 2, rt.NHWC, rt.ACT_NAMES[act], bias)
    assert c.rtoss_conv_group([c.conv_item(packed, x, t, N, H, W, 2, rt.NHWC, rt.ACT_NAMES[act], bias) for t in y[1:]]) == 1
    assert torch.equal(y[0], y[1]) and torch.equal(y[1], y[2])
    assert _near(y[0], _exact(packed, x, bias, act), dt, act)
    assert c.rtoss_device_status() == 0
    packed.close()


@pytest.mark.parametrize("act,after_act", [("none", False), ("relu", False), ("relu", True)])
@pytest.mark.parametrize("N,Cin,Cout,H,W,dt", [(10, 64, 16, 116, 55, "bf16"), (11, 40, 16, 51, 130, "f16"), (9, 384, 440, 13, 34, "bf16")])
def test_with_a_residual_operand_in_one_stage(N, Cin, Cout, H, W, dt, act, after_act):
    """Such calls keep one stage; they give the bits of the call without the operand, in two, and an addition."""
    assert _two_stages(N, H, W, Cin, Cout, dt)[0] and not _two_stages(N, H, W, Cin, Cout, dt, residual=True)[0]
    c, packed, x, bias, g = _layer(N, Cin, Cout, H, W, dt, "kernel")
    res = torch.randn(N, (H + 1) // 2, (W + 1) // 2, Cout, device="cuda", generator=g).to(x.dtype)
    y, plain = torch.empty_like(res), torch.empty_like(res)
    c.rtoss_conv3x3_pattern(packed, x, y, N, H, W, 2, rt.NHWC, rt.ACT_NAMES[act], bias, residual=res, residual_after_act=after_act)
    c.rtoss_conv3x3_pattern(packed, x, plain, N, H, W, 2, rt.NHWC, rt.ACT_NAMES[act if after_act else "none"], bias)
    two = (plain.float() + res.float()).to(x.dtype)
    assert torch.equal(y, torch.relu(two) if act == "relu" and not after_act else two)
    assert c.rtoss_device_status() == 0
    packed.close()


@pytest.mark.parametrize("act", ["none", "relu", "silu"])
@pytest.mark.parametrize("N,Cin,Cout,H,W,dt", [(10, 64, 16, 116, 55, "bf16"), (31, 56, 18, 33, 36, "f16"), (8, 96, 128, 80, 80, "bf16")])
def test_behind_the_layout_pass(N, Cin, Cout, H, W, dt, act):
    assert _two_stages(N, H, W, Cin, (Cout + 7) // 8 * 8, dt)[0]   # (planned alike: the filters are one tile)
    c, packed, x, bias, _ = _layer(N, Cin, Cout, H, W, dt, "kernel")
    xc, shape = x.permute(0, 3, 1, 2).contiguous(), (N, Cout, (H + 1) // 2, (W + 1) // 2)
    y = torch.empty(shape, dtype=x.dtype, device="cuda")
    c.rtoss_conv3x3_pattern(packed, xc, y, N, H, W, 2, rt.NCHW, rt.ACT_NAMES[act], bias)
    assert _near(y.permute(0, 2, 3, 1), _exact(packed, x, bias, act), dt, act)
    assert c.rtoss_device_status() == 0
    packed.close()


@pytest.mark.parametrize("N,Cin,Cout,H,W,dt,act,stages,shares", [
    (8, 392, 264, 11, 39, "bf16", "relu", 2, 4), (9, 384, 440, 13, 34, "f16", "silu", 2, 3), (11, 272, 144, 14, 21, "bf16", "none", 3, 3),
    (15, 320, 72, 8, 88, "f16", "silu", 3, 3), (4, 488, 448, 12, 123, "bf16", "silu", 3, 2), (5, 456, 288, 61, 11, "f16", "none", 3, 4),
])
def test_cut_along_k(N, Cin, Cout, H, W, dt, act, stages, shares):
    assert _two_stages(N, H, W, Cin, Cout, dt) == (True, stages, shares)
    c, packed, x, bias, _ = _layer(N, Cin, Cout, H, W, dt, "kernel")
    y = torch.empty(N, (H + 1) // 2, (W + 1) // 2, Cout, dtype=x.dtype, device="cuda")
    c.rtoss_conv3x3_pattern(packed, x, y, N, H, W, 2, rt.NHWC, rt.ACT_NAMES[act], bias)
    assert _near(y, _exact(packed, x, bias, act), dt, act)
    assert c.rtoss_device_status() == 0
    packed.close()
