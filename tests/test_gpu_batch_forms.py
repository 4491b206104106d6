"""The whole-model pass in its other form: beside a layer that makes the model a large one (blocks of 256 threads, channels
ordered sixteen at a time), the layers of the edge cases, which alone take blocks of 64 threads and a warp per channel, give the
bits that rtoss_pack gives them.  Also: a layer that inherits another one's patterns, in a small and in a large model."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_2303_02191_b200 import binding as rt
    from paper_2303_02191_b200 import synth
    import gpu_util as gu

from test_gpu_batch_edges import CASES, PRESET


def _layer(c, co, ci, ks, k, preset, wdt, cdt, seed):
    masks = rt.rtoss_pattern_preset(k, PRESET[preset])
    w = synth.kaiming_weights(seed, co + ci, co, ci, ks)
    flat = w.reshape(-1)
    if flat.size > 100:
        flat[5], flat[40], flat[9:18] = 6e4, np.inf, np.nan
    wd = gu.to_dev(synth.round_like(w, wdt), wdt)
    pid = c.rtoss_select_patterns(wd, ks, masks, k)
    want = c.rtoss_pack(wd, ks, masks, k, pid, rt.DTYPE_NAMES[cdt])
    blank = torch.zeros_like(wd)
    got = c.rtoss_pack(blank, ks, masks, k, c.rtoss_select_patterns(blank, ks, masks, k), rt.DTYPE_NAMES[cdt])
    return dict(w=wd, ksize=ks, masks=masks, k=k, packed=got, pid=torch.zeros_like(pid)), want, pid


def _same(a, b):
    return all(np.array_equal(a[key].view(np.uint8), b[key].view(np.uint8)) for key in b)


@pytest.mark.parametrize("large", [False, True])
@pytest.mark.parametrize("case", CASES, ids=lambda c: "-".join(str(v) for v in c))
def test_forms_agree(case, large):
    c = gu.ctx()
    layers = [_layer(c, *case, 73)]
    if large:
        layers = [_layer(c, 400, 400, 3, 4, "centre8", "f32", "bf16", 74)] + layers + [_layer(c, 40, 20, 1, 4, "centre8", "f32", "bf16", 75)]
    b = c.rtoss_batch_create([L[0] for L in layers])
    for _ in range(2):
        b.rtoss_batch_select_pack()
    torch.cuda.synchronize()
    for item, want, pid in layers:
        assert torch.equal(item["pid"], pid) and _same(item["packed"].export(), want.export())
    # (the tensor path's weights and issue words, which no export shows: test_gpu_repack_then_read.py and the layer calls below)
    co, ci, ks = case[0], case[1], case[2]
    x = torch.randn((1, 12, 14, ci), device="cuda").to(gu.TORCH_DT[case[6]])
    ys = [torch.zeros((1, 12, 14, co), dtype=x.dtype, device="cuda") for _ in range(2)]
    fn = c.rtoss_conv3x3_pattern if ks == 3 else c.rtoss_conv1x1_pattern
    i = 1 if large else 0
    for packed, y in zip((layers[i][1], layers[i][0]["packed"]), ys):
        fn(packed, x, y, 1, 12, 14, 1, rt.NHWC)
    torch.cuda.synchronize()
    assert torch.equal(ys[0].view(torch.uint8), ys[1].view(torch.uint8)) and c.rtoss_device_status() == 0
    b.close()
    for item, want, _ in layers:
        item["packed"].close(), want.close()


@pytest.mark.parametrize("large", [False, True])
def test_inherited_patterns(large):
    c, masks = gu.ctx(), rt.rtoss_pattern_preset(4, rt.PRESET_CENTRE8)
    for ks, co, ci in ((3, 70, 18), (1, 48, 97)):
        w = [gu.to_dev(synth.kaiming_weights(76, i + ks, co, ci, ks), "f32") for i in range(2)]
        pid = c.rtoss_select_patterns(w[0], ks, masks, 4)
        want = c.rtoss_pack(w[1], ks, masks, 4, pid, rt.BF16)
        items = [dict(w=v, ksize=ks, masks=masks, k=4, packed=c.rtoss_pack(v, ks, masks, 4, c.rtoss_select_patterns(v, ks, masks, 4), rt.BF16)) for v in w]
        items[1]["pid_from"] = 0
        if large:
            big = _layer(c, 400, 400, 3, 4, "centre8", "f32", "bf16", 77)
            items.append(big[0])
        b = c.rtoss_batch_create(items)
        b.rtoss_batch_select_pack()
        torch.cuda.synchronize()
        assert _same(items[1]["packed"].export(), want.export())
        b.close(), want.close()
        for it in items:
            it["packed"].close()
