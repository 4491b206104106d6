"""16-bit calls whose activations the tensor path cannot read where they lie (NCHW; channels last with pixels of no
multiple of 16 bytes): one pass lays them out, the tensor path does the rest.  Against the oracle, and against the FMA
path, at the edges of the layout pass (64 channels x 64 pixels, loads of 16 / 4 / 2 bytes) and of the NCHW epilogue
(pairs of positions, quarters of 32 filters).  Tolerance: half a unit in the last place of the output type on each side
(bf16 2^-9, fp16 2^-12 of the value, of the RMS below it) plus the fp32 sums' rounding, far below the 2e-2 both paths
are held to."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from oracle import rtoss_oracle as orc
    from paper_2303_02191_b200 import binding as rt
    from paper_2303_02191_b200 import synth
    import gpu_util as gu

ULP = {"bf16": 2.0 ** -7, "f16": 2.0 ** -10}   # one unit in the last place, relative: both sides round once


def _table(k):
    return orc.pattern_preset(k, orc.PRESET_CENTRE8 if k == 4 else orc.PRESET_CONN4)


CASES = [
    # ks, N, Cin, Cout, H, W, stride, k, dt, act, layout, (channel offset, channels of y)
    (3, 2, 64, 64, 16, 24, 1, 4, "bf16", "silu", "nchw", (0, 0)),      # planes of a multiple of eight: 16-byte loads; two filter copies
    (3, 1, 72, 130, 9, 14, 1, 3, "f16", "relu", "nchw", (0, 0)),       # even planes: 4-byte loads; 130 filters: a quarter of two
    (3, 3, 67, 75, 13, 17, 1, 3, "bf16", "none", "nchw", (0, 0)),      # odd planes: element loads and stores
    (3, 1, 256, 128, 10, 10, 1, 4, "bf16", "silu", "nchw", (0, 0)),    # few tiles, many channels: cut along K
    (3, 1, 40, 20, 21, 30, 2, 4, "f16", "silu", "nchw", (0, 0)),       # stride 2, four filter copies
    (3, 1, 17, 16, 1, 1, 1, 4, "bf16", "none", "nchw", (0, 0)),        # a single pixel
    (3, 2, 16, 32, 50, 41, 1, 4, "bf16", "silu", "nchw", (0, 0)),      # few channels: just above the outputs from which the pass pays
    (3, 1, 24, 96, 7, 300, 1, 4, "bf16", "relu", "nchw", (3, 101)),    # wide rows cut into segments, a channel slice
    (1, 2, 64, 48, 12, 20, 1, 4, "bf16", "silu", "nchw", (0, 0)),      # positions on M
    (1, 1, 100, 33, 15, 15, 2, 3, "f16", "relu", "nchw", (5, 44)),     # positions on M, kept pixels only, a channel slice
    (1, 2, 130, 200, 11, 13, 2, 3, "bf16", "silu", "nchw", (0, 0)),
    (1, 1, 1024, 256, 8, 10, 1, 4, "bf16", "none", "nchw", (0, 0)),    # cut along K
    (3, 3, 100, 75, 13, 21, 1, 3, "f16", "relu", "nhwc", (0, 0)),      # channels last, 8-byte loads
    (3, 2, 70, 64, 9, 12, 2, 4, "bf16", "silu", "nhwc", (8, 80)),      # 4-byte loads, aligned output slice
    (3, 1, 33, 40, 20, 20, 1, 2, "bf16", "none", "nhwc", (0, 0)),      # element loads
    (1, 2, 61, 90, 14, 9, 2, 3, "f16", "silu", "nhwc", (0, 0)),
    (1, 1, 7, 24, 30, 30, 1, 4, "bf16", "relu", "nhwc", (0, 0)),
]


@pytest.mark.parametrize("case", CASES, ids=lambda c: "-".join(str(v) for v in c))
def test_repacked_calls(case):
    ks, N, Cin, Cout, H, W, stride, k, dt, act, layout, (off, cs) = case
    x = synth.round_like(synth.activations(61, Cin + W, N, Cin, H, W), dt)
    w = synth.kaiming_weights(61, Cin + W, Cout, Cin, ks)
    b = synth.bias(61, Cin + W, Cout)
    masks = _table(k)
    _, packed = gu.select_pack(w, ks, masks, k, dt)
    _, wd, _ = gu.oracle_weights(w, ks, masks, k, dt)
    ref = gu.oracle_conv(ks, x, wd, b, stride, act, dt)
    y = gu.run_conv(packed, ks, x, dt, stride, act, b, layout, off, cs)
    got = y[:, off:off + Cout]
    assert orc.rel_err(got, ref) <= ULP[dt]
    y_fma = gu.run_conv(packed, ks, x, dt, stride, act, b, layout, off, cs, path=rt.PATH_FMA)
    assert orc.rel_err(got, y_fma[:, off:off + Cout]) <= ULP[dt]
    if cs:   # the channels around the slice stay as they were
        rest = np.delete(y, np.s_[off:off + Cout], axis=1)
        assert (rest == 7.0).all()
    assert gu.ctx().rtoss_device_status() == 0
    packed.close()


def test_repacked_calls_on_two_streams_and_in_a_graph():
    """Every call has a copy of its own: calls of different shapes in flight on two streams, and a captured pair."""
    masks, k = _table(4), 4
    c = gu.ctx()
    jobs = []
    for i, (Cin, Cout, H, W) in enumerate([(64, 64, 40, 40), (96, 128, 33, 50)]):
        w = synth.kaiming_weights(62, i, Cout, Cin, 3)
        _, packed = gu.select_pack(w, 3, masks, k, "bf16")
        xd = gu.to_dev(synth.activations(62, i, 4, Cin, H, W), "bf16")
        want = torch.empty((4, Cout, H, W), dtype=torch.bfloat16, device="cuda")
        c.rtoss_conv3x3_pattern(packed, xd, want, 4, H, W, 1, rt.NCHW, rt.ACT_SILU, None)
        jobs.append((packed, xd, want, torch.zeros_like(want), H, W))
    torch.cuda.synchronize()

    def call(j):
        packed, xd, _, y, H, W = j
        c.rtoss_conv3x3_pattern(packed, xd, y, 4, H, W, 1, rt.NCHW, rt.ACT_SILU, None)

    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    for _ in range(20):
        for s, j in zip(streams, jobs):
            with torch.cuda.stream(s):
                call(j)
    torch.cuda.synchronize()
    for j in jobs:
        assert torch.equal(j[2], j[3])
        j[3].zero_()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        for j in jobs:
            call(j)
    for _ in range(3):
        g.replay()
    torch.cuda.synchronize()
    for j in jobs:
        assert torch.equal(j[2], j[3])
    assert c.rtoss_device_status() == 0
    for j in jobs:
        j[0].close()


def test_first_repacked_call_of_a_context_inside_a_capture():
    """The pool of the channels-last copies is made on first use, which a stream capture does not forbid."""
    masks, k = _table(4), 4
    w = synth.kaiming_weights(63, 0, 64, 96, 3)
    xd = gu.to_dev(synth.activations(63, 0, 2, 96, 24, 24), "bf16")
    y, want = (torch.zeros((2, 64, 24, 24), dtype=torch.bfloat16, device="cuda") for _ in range(2))
    c = rt.Context(0)
    wd = torch.from_numpy(w).cuda()
    packed = c.rtoss_pack(wd, 3, masks, k, c.rtoss_select_patterns(wd, 3, masks, k), rt.BF16)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        c.rtoss_conv3x3_pattern(packed, xd, y, 2, 24, 24, 1, rt.NCHW, rt.ACT_SILU, None)
    g.replay()
    c.rtoss_conv3x3_pattern(packed, xd, want, 2, 24, 24, 1, rt.NCHW, rt.ACT_SILU, None)
    torch.cuda.synchronize()
    assert want.abs().max() > 0 and torch.equal(y, want)
    packed.close()
    del g
    c.close()
