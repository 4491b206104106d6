"""The whole-model pass at the edges of its block steps (512 kernels, two to a thread; 32-filter segments, 16 channels to an
ordering block), for tables on both sides of the limits that choose a form, for weights that are infinite or not a number,
and for a to-dense target that is not aligned.  Everything is compared bit for bit with the oracle."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from oracle import rtoss_oracle as orc
    from paper_2303_02191_b200 import binding as rt
    from paper_2303_02191_b200 import synth
    import gpu_util as gu

CASES = [
    # Cout, Cin, ksize, k, preset, w type, compute type
    (512, 16, 3, 4, "centre8", "f32", "bf16"),     # the most filters a thread per (segment, channel) takes
    (513, 16, 3, 4, "centre8", "f32", "bf16"),     # one more: a warp per channel
    (33, 17, 3, 4, "conn4", "f32", "f16"),         # 36 patterns, odd channels (padded rows), one channel in the last block
    (64, 40, 3, 5, "conn4", "bf16", "bf16"),       # 49 patterns: a warp per channel, factors
    (70, 24, 3, 4, "all", "f16", "bf16"),          # 126 patterns: predicated sums
    (19, 27, 3, 1, "all", "f32", "bf16"),          # 513 kernels: a chunk and one kernel; k = 1
    (1, 1, 3, 4, "centre8", "f32", "bf16"),        # one kernel
    (48, 97, 1, 3, "conn4", "f32", "f16"),         # 1x1, padded rows: 517 runs and three weights left over
    (64, 73, 1, 2, "conn4", "bf16", "f32"),        # 1x1 to fp32 (no tensor-path weights)
    (40, 68, 1, 4, "centre8", "f32", "f32"),       # 1x1, heads and remainders
    (20, 44, 3, 2, "conn4", "f16", "f32"),
    (18, 77, 3, 4, "centre8", "f16", "bf16"),      # four copies of every filter, odd rows, segments of two filters
    (40, 30, 3, 3, "conn4", "f32", "f16"),         # two copies, whole words; ids byte by byte
    (257, 20, 3, 4, "centre8", "f32", "bf16"),     # words of four ids; segments of 32, the last of one filter
]
PRESET = {"centre8": 2, "conn4": 1, "all": 0}


@pytest.mark.parametrize("case", CASES, ids=lambda c: "-".join(str(v) for v in c))
def test_batch_edges(case):
    co, ci, ks, k, preset, wdt, cdt = case
    c = gu.ctx()
    masks = rt.rtoss_pattern_preset(k, PRESET[preset])
    w = synth.round_like(synth.kaiming_weights(71, co + ci, co, ci, ks), wdt)
    flat = w.reshape(-1)
    if flat.size > 100:          # squares that overflow, an infinity, a kernel of nothing but NaNs
        flat[5], flat[40] = 1e30 if wdt != "f16" else 6e4, np.inf
        flat[9:18] = np.nan
        flat[20] = np.nan
        w = synth.round_like(w, wdt)
    wd = gu.to_dev(w, wdt)
    n = co * ci if ks == 3 else co * ci // 9
    store = torch.zeros(n + 1, dtype=torch.uint8, device="cuda")
    L = dict(w=wd, w_np=w, ksize=ks, masks=masks, k=k, wdt=wdt, pid=store[1:])      # an id array that is not aligned
    pid = c.rtoss_select_patterns(wd, ks, masks, k)
    L["packed"] = c.rtoss_pack(wd, ks, masks, k, pid, rt.DTYPE_NAMES[cdt])
    pid_single = pid.cpu().numpy()
    batch = c.rtoss_batch_create([L])
    for _ in range(2):
        batch.rtoss_batch_select_pack()
    torch.cuda.synchronize()
    pid_o = (orc.select_3x3(w, masks) if ks == 3 else orc.select_1x1(w.reshape(co, ci), masks)).ravel()
    assert np.array_equal(pid_single, pid_o)
    got = L["packed"].export()
    assert np.array_equal(store[1:].cpu().numpy(), pid_o) and np.array_equal(got["pid"], pid_o)
    ref = (orc.pack_3x3(w, masks, k, pid_o.reshape(co, ci), gu.ORC_DT[cdt]) if ks == 3
           else (orc.pack_1x1(w.reshape(co, ci), masks, k, pid_o, gu.ORC_DT[cdt]),))
    assert np.array_equal(gu.val_as_f32(got["val"], cdt), np.asarray(ref[0]).ravel(), equal_nan=True)
    if ks == 3:
        assert np.array_equal(got["perm"], np.asarray(ref[1]).ravel()) and np.array_equal(got["bucket_off"], np.asarray(ref[2]).ravel())
    # to-dense into memory that is not 16-byte aligned: the same bits as into memory that is
    dense = L["packed"].to_dense().reshape(-1)
    off = torch.zeros(dense.numel() + 1, dtype=dense.dtype, device="cuda")
    c._check(rt.lib.rtoss_packed_to_dense(c.h, L["packed"].h, off[1:].data_ptr(), torch.cuda.current_stream().cuda_stream))
    torch.cuda.synchronize()
    want = orc.unpack_3x3(ref[0], co, ci, masks, k, pid_o.reshape(co, ci)) if ks == 3 else orc.unpack_1x1(ref[0], co, ci, masks, k, pid_o)
    assert np.array_equal(dense.float().cpu().numpy(), np.asarray(want, dtype=np.float32).ravel(), equal_nan=True)
    assert np.array_equal(off[1:].float().cpu().numpy(), np.asarray(want, dtype=np.float32).ravel(), equal_nan=True)
    batch.close()
    L["packed"].close()


def test_convolution_on_repacked_weights_of_odd_channels():
    """The padded rows and the copies of narrow layers are what the tensor path reads: outputs after a batch re-pack."""
    c = gu.ctx()
    for co, ci, ks in [(24, 20, 3), (75, 35, 3), (90, 27, 1)]:
        masks = rt.rtoss_pattern_preset(4, PRESET["centre8"])
        w0, w1 = (synth.kaiming_weights(72 + i, co, co, ci, ks) for i in range(2))
        wd = gu.to_dev(w0, "f32")
        pid = c.rtoss_select_patterns(wd, ks, masks, 4)
        packed = c.rtoss_pack(wd, ks, masks, 4, pid, rt.BF16)
        batch = c.rtoss_batch_create([dict(w=wd, ksize=ks, masks=masks, k=4, packed=packed)])
        wd.copy_(gu.to_dev(w1, "f32"))
        batch.rtoss_batch_select_pack()
        x = synth.round_like(synth.activations(72, co, 2, ci, 24, 30), "bf16")
        y = gu.run_conv(packed, ks, x, "bf16", 1, "none", None, "nchw")
        _, wdense, _ = gu.oracle_weights(w1, ks, masks, 4, "bf16")
        assert orc.rel_err(y, gu.oracle_conv(ks, x, wdense, None, 1, "none", "bf16")) <= 2 ** -7   # one unit in the last place
        batch.close()
        packed.close()
